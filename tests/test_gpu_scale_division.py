"""The quantizer's scale and quotients are IEEE divisions in binary32, for every significand of a row's maximum."""
import numpy as np
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,exponent,rounding", [(8, 0, aqt.ROUND_NEAREST_EVEN), (4, 0, aqt.ROUND_HALF_UP_FLOOR), (8, -60, aqt.ROUND_HALF_UP_FLOOR),
                                                    (8, 59, aqt.ROUND_NEAREST_EVEN), (4, -61, aqt.ROUND_NEAREST_EVEN)])
def test_every_significand(bits, exponent, rounding):
    """Rows of four: the maximum and three values whose quotients lie at or beside ties."""
    qmax = np.float32(127 if bits == 8 else 7)
    amax = ((np.arange(1 << 23, dtype=np.uint32) | np.uint32(127 << 23)).view(np.float32) * np.float32(2.0) ** exponent).astype(np.float32)
    s = amax / qmax
    rng = np.random.default_rng(bits)
    ties = (rng.integers(-int(qmax), int(qmax), (3, amax.size)) + 0.5).astype(np.float32) * s
    x = np.stack([amax, *np.clip(ties, -amax, amax)], axis=1)
    q, scale = aqt.aqt_quantize(torch.from_numpy(x).cuda(), bits, rounding=rounding)
    v = x / s[:, None]
    want = np.rint(v) if rounding == aqt.ROUND_NEAREST_EVEN else np.floor((v + np.float32(0.5)).astype(np.float32))
    assert np.array_equal(scale.cpu().numpy().reshape(-1).view(np.uint32), s.view(np.uint32))
    assert np.array_equal(q.cpu().numpy(), np.clip(want, -qmax, qmax).astype(np.int8))
