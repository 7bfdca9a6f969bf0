"""The weight-only layer on binary16 operands (larger calls) against double precision (needs a B200).

Each activation enters with eleven significant bits, rounded to nearest (2^-11), as binary16 after an exact scaling of its row, or, in
blocks of 256 rows with a value that binary16 cannot hold beside its row's largest, as a tf32 operand (cut off, 2^-10).  Products are
exact, sums binary32:  |z - z_ref| <= (2^-11 or 2^-10 + K * 2^-24) * s_w * sum_k |x * wq| + 2^-23 * |z_ref|."""
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


def _call(x, wq, s_w, bias, residual, bits_w, act=aqt.ACT_NONE, small_workspace=False):
    (M, K), N = x.shape, s_w.numel()
    need = 4 * N * K if small_workspace else aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, M, N, K, 0, bits_w)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    y = torch.full((M, N // 2 if act >= aqt.ACT_GLU else N), float("nan"), device="cuda")
    return aqt.aqt_linear_fwd_weight_only(x, wq, s_w, bias, residual, 0.5, bits_w=bits_w, act=act, y=y, workspace=ws)


# both sides of K = 512 (rows per block of the pass), ragged rows, columns and k-blocks, a short last round of tiles
@pytest.mark.parametrize("M,N,K,bits_w,pad,res", [(1024, 2048, 640, 4, 0, False), (1025, 1284, 992, 8, 4, True), (1281, 4096, 256, 4, 8, False),
                                                  (2600, 1024, 512, 8, 0, True), (2605, 1024, 520, 4, 0, False), (12800, 2048, 512, 4, 0, False),
                                                  (1024, 1240, 1024, 8, 12, False)])
def test_against_double_precision(M, N, K, bits_w, pad, res):
    assert aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, M, N, K, 0, bits_w) > 4 * N * K  # such a call
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn(M, K + pad, generator=g, device="cuda")[:, :K]
    x[3] = 0.0
    x[5] *= 2.0 ** 90
    x[6] *= 2.0 ** -95
    x[M - 1, 2] = 1e-11  # the last block of rows is wide
    x[700, 1] = 1e30     # and this one
    wq, s_w = aqt.aqt_quantize(torch.randn(N, K, generator=g, device="cuda") * K ** -0.5, bits_w, pack=bits_w == 4)
    w = (aqt.aqt_unpack_int4(wq, K) if bits_w == 4 else wq).double()
    bias = torch.randn(N, generator=g, device="cuda") * 0.1
    r = torch.randn(M, N, generator=g, device="cuda") if res else None
    y = _call(x, wq, s_w, bias, r, bits_w)
    z = (x.double() @ w.t()) * s_w.double() + bias.double()
    mag = (x.double().abs() @ w.abs().t()) * s_w.double()
    # (a row is wide by its own values: 2^-28 of the largest; rows 3, 5 and 6 are scaled as a whole)
    t = x.abs() / x.abs().amax(dim=1, keepdim=True).clamp_min(1e-38)
    exps = torch.frexp(x.abs().amax(dim=1))[1]
    wide = ((t < 2.0 ** -28) & (x != 0)).any(dim=1) | ((exps < -98) | (exps > 99)) & (x != 0).any(dim=1)
    block = torch.arange(M, device="cuda") // 256
    wide_block = torch.zeros(int(block.max()) + 1, device="cuda").index_add_(0, block, wide.float())[block] > 0
    assert wide_block[700] and wide_block[M - 1]
    operand = torch.where(wide_block, 2.0 ** -10, 2.0 ** -11)[:, None].double()
    bound = (operand + K * 2.0 ** -24) * mag + 2.0 ** -23 * z.abs()
    want = z
    if res:
        want = 0.5 * z + r.double()
        bound = 0.5 * bound + 2.0 ** -23 * (want.abs() + z.abs())
    assert ((y.double() - want).abs() <= bound).all()
    # the tf32 operands of the same call, where the workspace has room for no others: wide blocks are the same bits
    same = _call(x, wq, s_w, bias, r, bits_w, small_workspace=True)
    assert torch.equal(y[wide_block], same[wide_block]) and aqt.aqt_device_status() == 0


def test_values_that_are_no_numbers():
    g = torch.Generator(device="cuda").manual_seed(1)
    M, N, K = 1536, 2048, 512
    x = torch.randn(M, K, generator=g, device="cuda")
    x[2, 7], x[300, 1], x[1000, 5] = float("nan"), float("inf"), -float("inf")
    wq, s_w = aqt.aqt_quantize(torch.randn(N, K, generator=g, device="cuda"), 8)
    for act in (aqt.ACT_NONE, aqt.ACT_SWISH, aqt.ACT_GLU):
        a, b = (_call(x, wq, s_w, None, None, 8, act, small) for small in (False, True))
        assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.isinf(a), torch.isinf(b))
        rows = torch.tensor([0, 2, 300, 1000], device="cuda")
        assert torch.equal(a[rows].view(torch.int32), b[rows].view(torch.int32))  # in blocks with such a row


def test_exact_where_nothing_is_rounded():
    """Activations of eleven bits and sums of fewer than 24: the integers themselves."""
    g = torch.Generator(device="cuda").manual_seed(2)
    M, N, K = 1100, 1280, 1024
    x = torch.randint(-63, 64, (M, K), generator=g, device="cuda").float() * 2.0 ** torch.randint(-20, 20, (M, 1), generator=g, device="cuda")
    wq = torch.randint(-127, 128, (N, K), generator=g, device="cuda", dtype=torch.int8)
    y = _call(x, wq, torch.ones(N, device="cuda"), None, None, 8)
    assert torch.equal(y.double(), x.double() @ wq.double().t())
