"""The one-launch layer for a few rows against the quantizer and the matmul called one after the other.  Both compute exact
integer sums and then the same operations in the same order, so the bits are the same."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


def _case(M, N, K, bits_w, bits_a, act, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lo, hi = (-8, 8) if bits_w == 4 else (-127, 128)
    w = torch.randint(lo, hi, (N, K), generator=g, device="cuda", dtype=torch.int8)
    wq = aqt.aqt_pack_int4(w) if bits_w == 4 else w
    glu = act in (aqt.ACT_GLU, aqt.ACT_GLU_SWISH)
    x = torch.randn(M, K, generator=g, device="cuda")
    x[M // 2] *= 37.0
    x[M - 1, : K // 2] = 0.0
    if M > 2:
        x[1] = 0.0  # a row of zeros
    n_out = N // 2 if glu else N
    return (x, wq, torch.rand(N, generator=g, device="cuda") * 1e-2 + 1e-4, torch.randn(N, generator=g, device="cuda"),
            torch.randn(M, n_out, generator=g, device="cuda"))


def _two_calls(x, wq, s_w, bias, res, rs, bits_a, bits_w, kind, rounding, act):
    K = x.shape[1]
    q, s = aqt.aqt_quantize(x, bits_a, aqt.AXIS_ROW if kind == aqt.SCALE_ROW else aqt.AXIS_TENSOR, rounding=rounding)
    return aqt.aqt_qmatmul(q, s, wq, s_w, bias, res, rs, K=K, bits_a=8 if bits_a == 8 else aqt.BITS_4_UNPACKED, bits_w=bits_w, act=act, s_x_kind=kind)


# rows: the edges of 1, 2, 4 and 8 tiles of eight; K: half a piece of weights, not a multiple of one, the most registers hold,
# more than that, the largest for each row count; N: four columns, one tile less four, the edges of 16, 32 and 64
# channels per CTA over 148 SMs and the first beyond
@pytest.mark.parametrize("bits_w,bits_a,kind,rounding", [(4, 8, aqt.SCALE_ROW, aqt.ROUND_NEAREST_EVEN), (8, 4, aqt.SCALE_TENSOR, aqt.ROUND_HALF_UP_FLOOR),
                                                         (8, 8, aqt.SCALE_ROW, aqt.ROUND_HALF_UP_FLOOR), (4, 4, aqt.SCALE_TENSOR, aqt.ROUND_NEAREST_EVEN)])
@pytest.mark.parametrize("M,N,K,act", [
    (1, 4, 32, aqt.ACT_NONE), (8, 28, 160, aqt.ACT_SWISH), (9, 2368, 1024, aqt.ACT_NONE), (16, 2372, 1056, aqt.ACT_SWISH), (17, 4736, 256, aqt.ACT_NONE),
    (32, 4740, 1024, aqt.ACT_NONE), (33, 9472, 128, aqt.ACT_SWISH), (64, 9476, 128, aqt.ACT_NONE), (64, 512, 512, aqt.ACT_SWISH), (64, 512, 544, aqt.ACT_NONE),
    (65, 512, 64, aqt.ACT_NONE), (8, 512, 8192, aqt.ACT_NONE), (16, 48, 4096, aqt.ACT_NONE), (16, 48, 4128, aqt.ACT_NONE),
    (48, 8192, 512, aqt.ACT_SWISH), (49, 4092, 512, aqt.ACT_NONE), (49, 4096, 512, aqt.ACT_NONE),  # either side of 48 rows and of 2 M weights
    (5, 8, 64, aqt.ACT_GLU), (16, 2376, 512, aqt.ACT_GLU_SWISH), (40, 4728, 288, aqt.ACT_GLU_SWISH), (3, 4096, 1024, aqt.ACT_GLU)])
def test_one_launch_gives_the_bits_of_two(M, N, K, act, bits_w, bits_a, kind, rounding):
    x, wq, s_w, bias, res = _case(M, N, K, bits_w, bits_a, act)
    for b, r in ((bias, None), (None, res)):
        y = aqt.aqt_linear_fwd(x, wq, s_w, b, r, 0.5, bits_a=bits_a, bits_w=bits_w, a_scale_kind=kind, rounding=rounding, act=act)
        ref = _two_calls(x, wq, s_w, b, r, 0.5, bits_a, bits_w, kind, rounding, act)
        assert torch.equal(y.view(torch.int32), ref.view(torch.int32))
    assert aqt.aqt_device_status() == 0


def test_pitched_unaligned_and_in_place():
    M, K = 24, 256
    x, wq, s_w, bias, _ = _case(M, K, K, 8, 8, aqt.ACT_NONE)
    ref = _two_calls(x, wq, s_w, bias, None, 1.0, 8, 8, aqt.SCALE_ROW, aqt.ROUND_NEAREST_EVEN, aqt.ACT_NONE)
    for pitch, first in ((K + 4, 0), (K + 4, 4), (K + 3, 0), (K + 4, 1)):  # the last two: rows that are no float4s
        buf = torch.zeros(M * pitch + 8, device="cuda")
        xv = torch.as_strided(buf, (M, K), (pitch, 1), first)
        xv.copy_(x)
        assert torch.equal(aqt.aqt_linear_fwd(xv, wq, s_w, bias), ref)
    y = x.clone()
    assert torch.equal(aqt.aqt_linear_fwd(y, wq, s_w, bias, y=y), ref)  # x and y the same buffer


@pytest.mark.parametrize("rows,cols", [(64, 256), (65, 256), (16, 1028), (127, 129)])
def test_whole_tensor_quantizer_around_the_size_that_one_block_takes(rows, cols):
    x = torch.randn(rows, cols, device="cuda")
    q, s = aqt.aqt_quantize(x, 8, aqt.AXIS_TENSOR)
    q_ref, s_ref = orc.quantize(x.cpu().numpy(), 8, orc.AXIS_TENSOR)
    assert s.item() == float(s_ref.reshape(-1)[0]) and np.array_equal(q.cpu().numpy(), q_ref)
