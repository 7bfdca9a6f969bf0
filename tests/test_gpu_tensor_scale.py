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
    N, turns = 128, 6
    wq = rng.integers(-127, 128, (N, K)).astype(np.int8)
    s_w = rng.uniform(1e-4, 5e-3, N).astype(np.float32)
    wq_d, s_w_d = torch.from_numpy(wq).cuda(), torch.from_numpy(s_w).cuda()
    xs = [rng.standard_normal((M, K)).astype(np.float32) for _ in range(turns)]
    for i, x in enumerate(xs):
        x[M - 1, K - 1] = -7.5 - i  # the maximum in the last block's share
    xs_d = [torch.from_numpy(x).cuda() for x in xs]
    # what a layer ahead writes: another scale on every turn
    pq, p_w = (torch.from_numpy(rng.integers(-127, 128, n).astype(np.int8)).cuda() for n in ((M, 64), (K, 64)))
    p_sx = [torch.full((1,), 1e-3 * (i + 1), device="cuda") for i in range(turns)]
    p_sw = torch.full((K,), 0.01, device="cuda")
    buf = torch.full((M, K + pad), float("nan"), device="cuda")
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_FWD, M, N, K, 8, 8), dtype=torch.uint8, device="cuda")
    copied, ys = [], []
    torch.cuda.synchronize()
    for i in range(turns):  # the input is written right ahead of the call, other values on every turn: by a copy, by a layer
        if i % 2 == 0:
            buf[:, :K] = xs_d[i]
        else:
            aqt.aqt_qmatmul(pq, p_sx[i], p_w, p_sw, K=64, s_x_kind=aqt.SCALE_TENSOR, y=buf[:, :K])
        ys.append(aqt.aqt_linear_fwd(buf[:, :K], wq_d, s_w_d, a_scale_kind=aqt.SCALE_TENSOR, workspace=ws))
        copied.append(buf[:, :K].clone())
    for i in range(turns):
        x = copied[i].cpu().numpy()
        assert i % 2 == 1 or np.array_equal(x, xs[i])
        q, s = orc.quantize(x, 8, orc.AXIS_TENSOR, aqt.ROUND_NEAREST_EVEN)
        ref = orc.epilogue_f32(orc.int_matmul(q, wq), s.reshape(-1), aqt.SCALE_TENSOR, s_w, None, None, 1.0, aqt.ACT_NONE)
        assert np.array_equal(ys[i].cpu().numpy().view(np.uint32), ref.view(np.uint32)), i
    assert aqt.aqt_device_status() == 0


@pytest.mark.parametrize("M,K,N,bits_w", [(130, 256, 256, 8), (1013, 512, 512, 4), (300, 96, 1024, 4), (700, 512, 2048, 8)])
@pytest.mark.parametrize("kind", [aqt.SCALE_ROW, aqt.SCALE_TENSOR])
def test_weights_written_right_ahead_of_the_layer(M, K, N, bits_w, kind):
    """The layer's matmul may fetch its weights while the quantizer of its activations drains; they may have been written by
    the call ahead of the layer.  Other weights and biases on every turn."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 8, bits_w).startswith("few")
    rng = np.random.default_rng(M + N)
    turns = 6
    w = [rng.standard_normal((N, K)).astype(np.float32) * (i + 1) for i in range(turns)]
    w_d = [torch.from_numpy(a).cuda() for a in w]
    x = rng.standard_normal((M, K)).astype(np.float32)
    x_d = torch.from_numpy(x).cuda()
    bias_d = [torch.full((N,), float(i), device="cuda") for i in range(turns)]
    wq = torch.zeros((N, K // 2 if bits_w == 4 else K), dtype=torch.uint8 if bits_w == 4 else torch.int8, device="cuda")
    s_w, bias = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda")
    ys = [torch.empty((M, N), device="cuda") for _ in range(turns)]
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_FWD, M, N, K, 8, bits_w), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for i in range(turns):
        bias.copy_(bias_d[i])
        aqt.aqt_quantize(w_d[i], bits_w, pack=bits_w == 4, q_out=wq, scale_out=s_w)
        aqt.aqt_linear_fwd(x_d, wq, s_w, bias, bits_w=bits_w, a_scale_kind=kind, y=ys[i], workspace=ws)
    q, s = orc.quantize(x, 8, orc.AXIS_ROW if kind == aqt.SCALE_ROW else orc.AXIS_TENSOR, aqt.ROUND_NEAREST_EVEN)
    for i in range(turns):
        wr, sr = orc.quantize(w[i], bits_w, orc.AXIS_ROW, aqt.ROUND_NEAREST_EVEN)
        ref = orc.epilogue_f32(orc.int_matmul(q, wr), s.reshape(-1), kind, sr.reshape(-1), np.full(N, i, np.float32), None, 1.0, aqt.ACT_NONE)
        assert np.array_equal(ys[i].cpu().numpy().view(np.uint32), ref.view(np.uint32)), i
    assert aqt.aqt_device_status() == 0
