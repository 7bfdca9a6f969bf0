"""The one-launch layer on rows whose scales take the general sequence, beside rows that do not: the bits of the two kernels (needs a B200)."""
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


# rows per warp of the kernel 1, 1, 2 and 4; one step of the conversion and several
@pytest.mark.parametrize("M,K", [(7, 512), (7, 4096), (16, 1024), (13, 1536), (30, 512), (30, 1056), (64, 512), (57, 256)])
@pytest.mark.parametrize("bits_w,bits_a,rounding", [(4, 8, aqt.ROUND_NEAREST_EVEN), (8, 4, aqt.ROUND_HALF_UP_FLOOR), (8, 8, aqt.ROUND_NEAREST_EVEN)])
@pytest.mark.parametrize("which", ["all", "one", "none"])
def test_scales_of_the_general_sequence(M, K, bits_w, bits_a, rounding, which):
    g = torch.Generator(device="cuda").manual_seed(M * K)
    N = 272
    x = torch.randn(M, K, generator=g, device="cuda")
    odd = {"all": range(M), "one": [M - 1], "none": []}[which]
    for r in odd:
        x[r] *= (2.0 ** -70, 2.0 ** 70, 2.0 ** -130, 1.0, 1.0)[r % 5]
        if r % 5 == 3:
            x[r, 5] = float("nan")
        if r % 5 == 4:
            x[r, 7] = float("inf")
    x[0, :] = 0.0
    wq, s_w = aqt.aqt_quantize(torch.randn(N, K, generator=g, device="cuda") * K ** -0.5, bits_w, pack=bits_w == 4)
    bias = torch.randn(N, generator=g, device="cuda")
    y = aqt.aqt_linear_fwd(x, wq, s_w, bias, None, 1.0, bits_a=bits_a, bits_w=bits_w, rounding=rounding, act=aqt.ACT_SWISH)
    xq, s_x = aqt.aqt_quantize(x, bits_a, rounding=rounding)
    want = aqt.aqt_qmatmul(xq, s_x, wq, s_w, bias, K=K, bits_a=8 if bits_a == 8 else aqt.BITS_4_UNPACKED, bits_w=bits_w, act=aqt.ACT_SWISH)
    assert torch.equal(torch.isnan(y), torch.isnan(want))
    assert torch.equal(torch.nan_to_num(y).view(torch.int32), torch.nan_to_num(want).view(torch.int32)) and aqt.aqt_device_status() == 0
