"""Parity of the CTA-pair matmul whose last tiles are taken in halves with the CPU oracle (needs a B200)."""
import pytest

from paper_2203_15952_b200 import binding as aqt
from test_gpu_kernels import _run_qmatmul

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plan", ["pair256s4e8", "pair256s6e4"])
@pytest.mark.parametrize("M,N,K,act,with_res", [(256 * 74 + 1, 256, 640, aqt.ACT_NONE, True), (256 * 36 + 100, 516, 528, aqt.ACT_SWISH, False),
                                                (256 * 55, 512, 576, aqt.ACT_NONE, False), (256 * 60, 640, 1024, aqt.ACT_GLU, True),
                                                (256 * 25 + 3, 776, 544, aqt.ACT_GLU_SWISH, False)])
def test_last_pair_tiles_in_halves(plan, M, N, K, act, with_res):
    # 74 pairs: one to 37 tiles in the last round, taken as halves; halves that start beyond the last column
    _run_qmatmul(M, N, K, 8, 8, act, True, with_res, plan=plan)
