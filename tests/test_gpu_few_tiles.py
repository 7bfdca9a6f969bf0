"""Parity of the matmul for outputs of a few tiles with the CPU oracle: tile widths, ragged edges, depths beyond its ring,
residual and gate forms, and the form that quantizes the last columns only (needs a B200)."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt
from test_gpu_kernels import _run_qmatmul
from test_gpu_requant import _codes, _dev, _run

pytestmark = pytest.mark.gpu

# (148 SMs) one CTA per tile: 32, 64 and 128 columns, the last size that each covers, rows and columns that end inside a tile,
# one k-block, a ragged one, as many as the ring has stages, one more, and several turns of the ring
SHAPES = [(1, 512, 512, "few32"), (113, 1056, 144, "few128"), (128, 4736, 64, "few128"), (129, 512, 9 * 128, "few32"),
          (1013, 512, 9 * 128 + 16, "few32"), (1153, 512, 512, "few64"), (2304, 512, 2048, "few64"), (2305, 512, 512, "few128"),
          (300, 1024, 7 * 128, "few64"), (700, 800, 8 * 128, "few64"), (1013, 2048, 512, "few128"), (37 * 128, 512, 512, "few128")]


@pytest.mark.parametrize("M,N,K,plan", SHAPES)
@pytest.mark.parametrize("with_res", [False, True])
def test_few_tiles_requant(M, N, K, plan, with_res):
    refused = 1024 < K < 2048  # without y
    _run(M, N, K, 8, 8, aqt.ACT_NONE, True, with_res, 8, aqt.ROUND_NEAREST_EVEN, False, special_rows=not with_res, may_refuse_without_y=refused,
         plan=plan, plan_without_y=None if refused else plan, may_wait=True)


@pytest.mark.parametrize("M,N,K,plan", [(200, 512, 512, "few32"), (1013, 2048, 256, "few128"), (1000, 1024, 96, "few64")])
@pytest.mark.parametrize("rounding", [aqt.ROUND_NEAREST_EVEN, aqt.ROUND_HALF_UP_FLOOR])
def test_few_tiles_packed_weights_swish(M, N, K, plan, rounding):
    _run(M, N, K, 4, 4, aqt.ACT_SWISH, False, False, 4, rounding, False, plan=plan, plan_without_y=plan)


@pytest.mark.parametrize("plan", ["few32", "few64", "few128"])
def test_few_tiles_plans_named(plan):
    # accumulators and output of every width, whether or not the library would choose it: one row, edges of tiles in both
    # directions, one k-block up to several turns of the ring, packed weights expanded in the kernel and ahead of it
    _run_qmatmul(1, 4, 32, 8, 8, aqt.ACT_NONE, True, True, plan=plan, extremes=True)
    _run_qmatmul(129, 36, 512, 8, 4, aqt.ACT_SWISH, True, True, plan=plan)
    _run_qmatmul(333, 1000, 400, 4, 4, aqt.ACT_NONE, False, False, plan=plan, s_x_kind=aqt.SCALE_TENSOR)
    _run_qmatmul(700, 260, 1296, 8, 8, aqt.ACT_NONE, True, True, plan=plan)
    if plan != "few32":
        _run_qmatmul(200, 520, 512, 8, 4, aqt.ACT_GLU, True, True, plan=plan)
        _run_qmatmul(129, 72, 1040, 8, 8, aqt.ACT_GLU_SWISH, False, False, plan=plan)
    with pytest.raises(aqt.AqtError) as e:  # a tile per SM, and no more
        _run_qmatmul(149 * 128, 32, 32, 8, 8, aqt.ACT_NONE, False, False, plan=plan)
    assert e.value.status == -3
    with pytest.raises(aqt.AqtError) as e:
        _run_qmatmul(130, 64, 64, 8, 8, aqt.ACT_GLU, False, False, plan="few32")
    assert e.value.status == -3


@pytest.mark.parametrize("M,N,K,first,plan", [(200, 768, 256, 512, "few32"), (1013, 1536, 512, 1024, "few128"), (1537, 1536, 512, 1024, "few64"),
                                              (140, 96, 64, 32, "few32"), (300, 480, 128, 16, "few32"), (4800, 640, 64, 128, "ws128")])
@pytest.mark.parametrize("bits_w", [4, 8])
def test_last_columns_quantized(M, N, K, first, plan, bits_w):
    # one launch or (1537 rows: 156 tiles of 128 columns) two by the size; first = 16 is no multiple of a tile's columns
    assert aqt.aqt_plan_qmatmul_requant(M, N, K, 8, bits_w, with_y=True, first=first) == plan
    rng = np.random.default_rng(M + N + first)
    xq, wq = _codes(rng, M, K, 8), _codes(rng, N, K, bits_w)
    s_x, s_w = rng.uniform(1e-3, 5e-2, M).astype(np.float32), rng.uniform(1e-4, 5e-3, N).astype(np.float32)
    bias = (rng.standard_normal(N) * 0.1).astype(np.float32)
    y = torch.full((M, N), float("nan"), device="cuda")
    q = torch.full((M, N - first), 0x55, dtype=torch.int8, device="cuda")
    s = torch.full((M,), float("nan"), device="cuda")
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_QMATMUL_REQUANT, M, N, K, 8, bits_w), dtype=torch.uint8, device="cuda")
    aqt.aqt_qmatmul_requant_from(first, _dev(xq), _dev(s_x), _dev(orc.pack_int4(wq) if bits_w == 4 else wq), _dev(s_w), _dev(bias), K=K,
                                 bits_w=bits_w, q_out=q, s_out=s, y=y, workspace=ws)
    assert aqt.aqt_device_status() == 0
    ref = orc.epilogue_f32(orc.int_matmul(xq, wq), s_x, aqt.SCALE_ROW, s_w, bias, None, 1.0, aqt.ACT_NONE)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    q_ref, s_ref = orc.quantize(np.ascontiguousarray(ref[:, first:]), 8, orc.AXIS_ROW, aqt.ROUND_NEAREST_EVEN)
    assert np.array_equal(q.cpu().numpy(), q_ref) and np.array_equal(s.cpu().numpy().view(np.uint32), s_ref.reshape(-1).view(np.uint32))


def test_few_tiles_replayed():
    # the exchange words of one execution must not pass for the next one's
    M, N, K = 1013, 512, 512
    rng = np.random.default_rng(3)
    xq, wq = _dev(_codes(rng, M, K, 8)), _dev(_codes(rng, N, K, 8))
    s_x, s_w = _dev(rng.uniform(1e-3, 5e-2, M).astype(np.float32)), _dev(rng.uniform(1e-4, 5e-3, N).astype(np.float32))
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_QMATMUL_REQUANT, M, N, K, 8, 8), dtype=torch.uint8, device="cuda")
    q, s = torch.empty(M, N, dtype=torch.int8, device="cuda"), torch.empty(M, device="cuda")

    def call():
        aqt.aqt_qmatmul_requant(xq, s_x, wq, s_w, K=K, q_out=q, s_out=s, workspace=ws)
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    for scale in (1.0, 0.25, 3.0, 0.5) * 5:
        s_x.mul_(scale)
        g.replay()
        want = aqt.aqt_qmatmul(xq, s_x, wq, s_w, K=K)
        q_ref, s_ref = aqt.aqt_quantize(want, 8)
        assert torch.equal(q, q_ref) and torch.equal(s, s_ref)
        s_x.div_(scale)
    assert aqt.aqt_device_status() == 0


def test_few_tiles_do_without_room_for_their_exchange():
    # the area that the wider tiles need, one row short of it, and the bits of either form
    M, N, K = 300, 512, 512
    rng = np.random.default_rng(5)
    args = (_dev(_codes(rng, M, K, 8)), _dev(rng.uniform(1e-3, 5e-2, M).astype(np.float32)), _dev(_codes(rng, N, K, 8)),
            _dev(rng.uniform(1e-4, 5e-3, N).astype(np.float32)))
    need = -(-M // 256) * 256 * (N // 64) * 8 + 256 * 4
    assert aqt.aqt_workspace_bytes(aqt.OP_QMATMUL_REQUANT, M, N, K, 8, 8) > need
    assert aqt.aqt_plan_qmatmul_requant(M, N, K) == "few32" and aqt.aqt_plan_qmatmul_requant(M, N, K, workspace_bytes=need) == "ws128"
    q0, s0, _ = aqt.aqt_qmatmul_requant(*args, K=K)
    q1, s1, _ = aqt.aqt_qmatmul_requant(*args, K=K, workspace=torch.empty(need, dtype=torch.uint8, device="cuda"))
    assert torch.equal(q0, q1) and torch.equal(s0, s1) and aqt.aqt_device_status() == 0
    with pytest.raises(aqt.AqtError):
        aqt.aqt_qmatmul_requant(*args, K=K, workspace=torch.empty(need - 256, dtype=torch.uint8, device="cuda"))
