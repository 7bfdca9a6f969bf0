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


def _pair(x, wq, N, K):
    """The call with the workspace asked for, and with room for tf32 operands alone."""
    s_w = torch.ones(N, device="cuda")
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, x.shape[0], N, K, 0, 8), dtype=torch.uint8, device="cuda")
    out = [aqt.aqt_linear_fwd_weight_only(x, wq, s_w, None, bits_w=8, y=torch.empty(x.shape[0], N, device="cuda"), workspace=w)
           for w in (ws, ws[:4 * N * K])]
    assert aqt.aqt_device_status() == 0
    return out


# Either form sums the same products into binary32, tf32 operands in K / 8 steps and binary16 ones in K / 16; a step drops at most 2^-23 of the
# running sum.  (Operands rounded instead of cut off are 6e-4 from these.)
def _same_products(y, tf32, K):
    return (y.double() - tf32.double()).norm() <= (K / 8 + K / 16) * 2.0 ** -23 * tf32.double().norm()


@pytest.mark.parametrize("M,N,K", [(2605, 1024, 520), (1281, 4096, 256), (5000, 3072, 768), (1100, 1280, 1024)])
def test_a_wide_row_changes_its_block_of_rows_alone(M, N, K):
    assert aqt.aqt_plan_qmatmul(M, N, K, 0, 8 | aqt.PLAN_WEIGHT_ONLY, float_kind=True) == "pair256s4e8f16"
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn(M, K, generator=g, device="cuda")
    x[x.abs() < 1e-6] = 0.0
    wq = torch.randint(-127, 128, (N, K), generator=g, device="cuda", dtype=torch.int8)
    plain, tf32 = _pair(x, wq, N, K)
    assert _same_products(plain, tf32, K) and not torch.equal(plain, tf32)  # (they are not the tf32 form's bits)
    x[700, 5] = 1e-12
    x[M - 1, 1] = -1e-30
    marked, tf32 = _pair(x, wq, N, K)
    for b in range(0, M, 256):
        want = tf32 if b in (512, (M - 1) // 256 * 256) else plain
        assert torch.equal(marked[b:b + 256].view(torch.int32), want[b:b + 256].view(torch.int32))


def test_rows_at_the_ends_of_the_scales():
    """Blocks of rows whose values are all of one size: from 2^-100 up to 2^101 they run on binary16, beyond on tf32 operands."""
    g = torch.Generator(device="cuda").manual_seed(3)
    exps, N, K = [-100, -101, 100, 101, 0, -126, 127 - 20], 4096, 256
    x = torch.cat([(1 + torch.rand(256, K, generator=g, device="cuda")) * torch.randn(256, K, generator=g, device="cuda").sign() * 2.0 ** e for e in exps])
    assert (x.abs() < 2 * 2.0 ** torch.tensor(exps, device="cuda").repeat_interleave(256)[:, None]).all()
    wq = torch.randint(-127, 128, (N, K), generator=g, device="cuda", dtype=torch.int8)
    y, tf32 = _pair(x, wq, N, K)
    z, mag = x.double() @ wq.double().t(), x.double().abs() @ wq.double().abs().t()
    for i, e in enumerate(exps):
        r = slice(256 * i, 256 * i + 256)
        assert _same_products(y[r], tf32[r], K) if -100 <= e <= 100 else torch.equal(y[r], tf32[r])
        assert ((y[r].double() - z[r]).abs() <= (2.0 ** -10 + K * 2.0 ** -24) * mag[r] + 2.0 ** -23 * z[r].abs()).all()


@pytest.mark.parametrize("M,N,K,act,tails", [(12800, 2048, 512, aqt.ACT_SWISH, False), (2600, 1024, 512, aqt.ACT_NONE, True), (4100, 2048, 1024, aqt.ACT_GLU, False)])
def test_the_binary16_form_has_the_results_of_the_tf32_form(M, N, K, act, tails):
    """Within 2e-5 of the norm, and no output further than 40 times that beside the root mean square."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 0, 4 | aqt.PLAN_WEIGHT_ONLY, act, float_kind=True) == "pair256s4e8f16"
    g = torch.Generator(device="cuda").manual_seed(K)
    x = torch.randn(M, K, generator=g, device="cuda")
    if tails:
        x /= sum(torch.randn(M, K, generator=g, device="cuda") ** 2 for _ in range(3)).sqrt()
    wq, s_w = aqt.aqt_quantize(torch.randn(N, K, generator=g, device="cuda") * K ** -0.5, 4, pack=True)
    bias = torch.randn(N, generator=g, device="cuda") * 0.01
    out = [aqt.aqt_linear_fwd_weight_only(x, wq, s_w, bias, bits_w=4, act=act, workspace=torch.empty(
        aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, rows, N, K, 0, 4), dtype=torch.uint8, device="cuda")).double() for rows in (M, 0)]
    d, rms = out[0] - out[1], out[1].square().mean().sqrt()
    assert d.norm() <= 2e-5 * out[1].norm() and d.abs().max() <= 8e-4 * rms
