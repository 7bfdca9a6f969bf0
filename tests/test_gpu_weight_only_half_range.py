"""The weight-only layer on binary16 operands at the ends of what a scaled row can hold (needs a B200).

Rows with a value that is not zero and below 2^-28 of the row's largest take tf32 operands:  |z - z_ref| <= (2^-10 + K * 2^-24) * s_w * sum_k |x * wq|
+ 2^-23 * |z_ref|, also where nothing but such values meets a code that is not zero."""
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large,small", [(100, -70), (100, -60), (70, -100), (14, -120), (0, -120), (-90, -120), (100, -140), (40, -149)])
@pytest.mark.parametrize("M,N,K", [(1281, 4096, 256), (2605, 1024, 520)])
def test_small_values_beside_a_large_one(M, N, K, large, small):
    """One large value a row, in channels whose code for it is zero: what is left are the small ones."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 0, 8 | aqt.PLAN_WEIGHT_ONLY, float_kind=True) == "pair256s4e8f16"
    g = torch.Generator(device="cuda").manual_seed(K)
    x = torch.randint(1, 4, (M, K), generator=g, device="cuda").double() * 2.0 ** small
    x[:, 0] = 2.0 ** large
    x = x.float()
    wq = torch.randint(-7, 8, (N, K), generator=g, device="cuda", dtype=torch.int8)
    wq[::3, 0] = 0
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, M, N, K, 0, 8), dtype=torch.uint8, device="cuda")
    y = aqt.aqt_linear_fwd_weight_only(x, wq, torch.ones(N, device="cuda"), None, bits_w=8, y=torch.empty(M, N, device="cuda"), workspace=ws)
    tf32 = aqt.aqt_linear_fwd_weight_only(x, wq, torch.ones(N, device="cuda"), None, bits_w=8, y=torch.empty(M, N, device="cuda"), workspace=ws[:4 * N * K])
    assert torch.equal(y.view(torch.int32), tf32.view(torch.int32))  # every row is such a row
    if small >= -126:  # (the tensor core takes subnormal operands as it pleases)
        z, mag = x.double() @ wq.double().t(), x.double().abs() @ wq.double().abs().t()
        assert ((y.double() - z).abs() <= (2.0 ** -10 + K * 2.0 ** -24) * mag + 2.0 ** -23 * z.abs()).all()
    assert aqt.aqt_device_status() == 0
