"""Shallow matmuls with a residual run on other tiles than without one: the same bits as on the weight-stationary ones."""
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


# more tiles of 128 columns than SMs, ragged edges, both sides of the 28 M outputs from which CTA pairs take the call
@pytest.mark.parametrize("M,N,K,pad", [(4737, 512, 512, 0), (7411, 516, 48, 4), (5000, 1000, 496, 0), (28671, 1024, 64, 0), (28672, 1024, 64, 12)])
def test_residual_plans_give_the_same_bits(M, N, K, pad):
    g = torch.Generator(device="cuda").manual_seed(M + K)
    xq, wq = (torch.randint(-127, 128, (n, K), generator=g, device="cuda", dtype=torch.int8) for n in (M, N))
    s_x, s_w, bias = (torch.rand(n, generator=g, device="cuda") for n in (M, N, N))
    r = torch.randn(M, N + pad, generator=g, device="cuda")[:, :N]
    out = [torch.full((M, N + pad), float("nan"), device="cuda")[:, :N] for _ in range(2)]
    for y, plan in zip(out, (None, "ws128e16")):
        aqt.aqt_qmatmul(xq, s_x, wq, s_w, bias, r, 0.5, K=K, y=y, plan=plan)
    assert torch.equal(*out) and not torch.isnan(out[0]).any()
    inplace = r.clone()
    aqt.aqt_qmatmul(xq, s_x, wq, s_w, bias, inplace, 0.5, K=K, y=inplace)
    assert torch.equal(inplace, out[0]) and aqt.aqt_device_status() == 0
