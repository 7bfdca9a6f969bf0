"""The weight-only layer's one-launch form for few rows against the binary64 oracle.

Operand error: the codes are exact in bf16; x is the sum of two bf16 terms up to 2^-16 of it (its upper sixteen bits, then eight
to nine of the rest), or exactly of three.  Every product and sum is then binary32 with truncation at worst: terms * K summands
at 2^-23 each of the sum of magnitudes."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200 import inputs as gen
from test_gpu_weight_only import _bound_out, _dev, _weights

pytestmark = pytest.mark.gpu


# rows: the edges of 8, 16 and 32 rows per CTA and several CTAs of rows; K: one group of four, a part of a piece, odd numbers of
# fours, the edges of a chunk of 512 and of 1024, several chunks; N: four columns, a partial tile, one wave of CTAs and
# more, both sides of two waves
@pytest.mark.parametrize("bits_w", [8, 4])
@pytest.mark.parametrize("precision", [aqt.FLOAT_TF32, aqt.FLOAT_TF32X2])
@pytest.mark.parametrize("M,N,K,act", [
    (1, 4, 4, orc.ACT_NONE), (8, 20, 36, orc.ACT_SWISH), (9, 64, 512, orc.ACT_NONE), (16, 2368, 516, orc.ACT_NONE), (16, 2372, 100, orc.ACT_SWISH),
    (17, 36, 1024, orc.ACT_NONE), (33, 132, 764, orc.ACT_NONE), (100, 40, 768, orc.ACT_SWISH), (5, 48, 1028, orc.ACT_NONE), (23, 144, 2684, orc.ACT_NONE),
    (256, 1184, 64, orc.ACT_NONE), (257, 1184, 64, orc.ACT_NONE), (7, 8, 48, orc.ACT_GLU), (12, 136, 516, orc.ACT_GLU_SWISH), (40, 200, 160, orc.ACT_GLU),
    (2, 4736, 128, orc.ACT_GLU_SWISH)])
def test_few_rows(M, N, K, act, precision, bits_w):
    x = gen.normal(3, 17, M, K)
    x[M // 2] *= 1e-30  # far from the others' range
    wq, s_w, w_dev = _weights(4, N, K, bits_w)
    bias = gen.normal(3, 19, 1, N, std=0.05)[0]
    n_out = N // 2 if act >= 2 else N
    res = gen.normal(3, 23, M, n_out)
    y_ref, z, mag = orc.linear_weight_only_f64(x, wq, s_w, bias=bias, residual=res, residual_scale=0.5, act=act, return_parts=True)
    buf = torch.full((M, K + 4), 7.0, device="cuda")  # pitched; the padding must not be read into the sum
    buf[:, :K] = _dev(x)
    y = torch.full((M, n_out), float("nan"), device="cuda")
    aqt.aqt_linear_fwd_weight_only(buf[:, :K], _dev(w_dev), _dev(s_w), _dev(bias), _dev(res), 0.5, bits_w=bits_w, precision=precision, act=act, y=y)
    got = y.cpu().numpy().astype(np.float64)
    # the first form beyond two waves, and the two-term form beyond K = 768, are the many-row form's, with its own operand error
    one_term, many = precision == aqt.FLOAT_TF32, (M, N) == (257, 1184) or (precision == aqt.FLOAT_TF32X2 and K > 768)
    operand = (2.0 ** -10 if one_term else 2.0 ** -20) if many else (2.0 ** -16 if one_term else 0.0)
    dz = (operand + (2 if one_term else 3) * K * 2.0 ** -23) * mag + 2.0 ** -22 * np.abs(z)
    tol = _bound_out(act, z, dz, 0.5, True, y_ref)
    err = np.abs(got - y_ref)
    assert np.all(err <= tol), (err / tol).max()


def test_not_finite_and_in_place():
    M, K = 8, 128
    wq, s_w, w_dev = _weights(4, K, K, 8)
    x = gen.normal(3, 17, M, K)
    ref = aqt.aqt_linear_fwd_weight_only(_dev(x), _dev(w_dev), _dev(s_w), bits_w=8)
    y = _dev(x)
    aqt.aqt_linear_fwd_weight_only(y, _dev(w_dev), _dev(s_w), bits_w=8, y=y)  # x and y the same buffer: the many-row form
    assert float((y - ref).abs().max()) <= 2.0 ** -9 * float(np.abs(x).sum(1).max()) * float(np.abs(wq * s_w[:, None]).max())
    x[3, 5] = np.float32(np.inf)
    x[4, 6] = np.float32(np.nan)
    x[5, 7] = np.float32(3.4028235e38)
    z = aqt.aqt_linear_fwd_weight_only(_dev(x), _dev(w_dev), _dev(s_w), bits_w=8)
    used = _dev(wq[:, 5] != 0)
    assert bool(z[3][used].isinf().all()) and bool(z[4].isnan().all())
    assert torch.equal(z[:3], ref[:3]) and torch.equal(z[6:], ref[6:])
