"""Which tiles a shallow matmul with a residual runs on (host-only), and that they give the same bits (needs a B200)."""
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

NONE, SWISH = aqt.ACT_NONE, aqt.ACT_SWISH


@pytest.mark.parametrize("M,N,K,bits_w,act,plan", [
    (7411, 512, 512, 8, NONE, "stream128s4e16"), (7411, 512, 512, aqt.BITS_4_UNPACKED, NONE, "stream128s4e16"),
    (28671, 1024, 256, 8, NONE, "stream128s4e16"), (28672, 1024, 256, 8, NONE, "pair128s6e8"), (28672, 1024, 240, 8, NONE, "stream128s4e16"),
    (45055, 2048, 240, 8, NONE, "stream128s4e16"), (45056, 2048, 240, 8, NONE, "pair128s6e8"),
    # packed weights, which only the weight-stationary kernel expands, unless their rows have no 16-byte pitch
    (28672, 1024, 256, 4, NONE, "ws128e16"), (28672, 1024, 272, 4, NONE, "pair128s6e8"),
    (28672, 1024, 256, 8, SWISH, "ws128e16"), (300, 256, 256, 8, NONE, "few32")])
def test_line_of_shallow_matmuls_with_a_residual(M, N, K, bits_w, act, plan):
    assert aqt.aqt_plan_qmatmul(M, N, K, 8, bits_w | aqt.PLAN_RESIDUAL, act, sm_count=148) == plan
    if not plan.startswith("few"):
        assert aqt.aqt_plan_qmatmul(M, N, K, 8, bits_w, act, sm_count=148) == "ws128e16"  # without one


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,plan", [(28672, 1024, 256, "pair128s6e8"), (28673, 1028, 240, "stream128s4e16"), (45057, 2052, 48, "pair128s6e8"),
                                        (45055, 2048, 16, "stream128s4e16")])
def test_both_sides_of_the_line_give_the_same_bits(M, N, K, plan):
    assert aqt.aqt_plan_qmatmul(M, N, K, 8, 8 | aqt.PLAN_RESIDUAL) == plan
    g = torch.Generator(device="cuda").manual_seed(M + K)
    xq, wq = (torch.randint(-127, 128, (n, K), generator=g, device="cuda", dtype=torch.int8) for n in (M, N))
    s_x, s_w, bias = (torch.rand(n, generator=g, device="cuda") for n in (M, N, N))
    r = torch.randn(M, N, generator=g, device="cuda")
    out = [torch.full((M, N), float("nan"), device="cuda") for _ in range(2)]
    for y, name in zip(out, (None, "ws128e16")):
        aqt.aqt_qmatmul(xq, s_x, wq, s_w, bias, r, 0.5, K=K, y=y, plan=name)
    assert torch.equal(*out) and not torch.isnan(out[0]).any() and aqt.aqt_device_status() == 0
