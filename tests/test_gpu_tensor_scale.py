"""The whole layer with one scale for the activation tensor on both sides of the lines between the quantizer's forms, against
the CPU oracle (needs a B200)."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


# 4096 elements a block: one block's share, one more, a ragged last block, 592 blocks (all beside pass 1), 593
@pytest.mark.parametrize("M,K,pad", [(65, 256, 0), (65, 352, 4), (129, 512, 0), (1000, 288, 0), (2368, 1024, 0), (2369, 1024, 0), (2372, 1024, 8)])
def test_linear_with_one_scale(M, K, pad):
    rng = np.random.default_rng(M + K)
    N = 128
    x = rng.standard_normal((M, K)).astype(np.float32)
    x[M - 1, K - 1] = -7.5  # the maximum in the last block's share
    wq = rng.integers(-127, 128, (N, K)).astype(np.int8)
    s_w = rng.uniform(1e-4, 5e-3, N).astype(np.float32)
    buf = torch.full((M, K + pad), float("nan"), device="cuda")
    buf[:, :K] = torch.from_numpy(x).cuda()
    for _ in range(3):  # the input is written right ahead of the call
        buf[:, :K] = torch.from_numpy(x).cuda()
        y = aqt.aqt_linear_fwd(buf[:, :K], torch.from_numpy(wq).cuda(), torch.from_numpy(s_w).cuda(), a_scale_kind=aqt.SCALE_TENSOR)
        q, s = orc.quantize(x, 8, orc.AXIS_TENSOR, aqt.ROUND_NEAREST_EVEN)
        ref = orc.epilogue_f32(orc.int_matmul(q, wq), s.reshape(-1), aqt.SCALE_TENSOR, s_w, None, None, 1.0, aqt.ACT_NONE)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    assert aqt.aqt_device_status() == 0
