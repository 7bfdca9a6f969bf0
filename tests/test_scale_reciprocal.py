"""The reciprocal of a row's scale by one Newton step: RN(1 / s) from either neighbour of 1 / s, but for one start value (CPU); at that
scale the quantizer's codes on the GPU (needs a B200)."""
import numpy as np
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt


def test_newton_step_from_either_neighbour():
    """s = S / 2^23 in [1, 2), y = Y / 2^24: both fused multiply-adds in integers, for every significand."""
    S = np.arange((1 << 23) + 1, 1 << 24, dtype=np.int64)  # (the power of two is its own case, without a rounding)
    down, rem = (1 << 47) // S, (1 << 47) % S
    nearest = down + (2 * rem > S)
    for Y in (down, down + 1):
        E = np.float32((1 << 47) - S * Y).astype(np.int64)  # fma(-s, y, 1) in units of 2^-47, rounded to 24 bits
        whole, part = np.divmod(E * Y, 1 << 47)             # fma(e, y, y) in units of 2^-24
        got = Y + whole + ((part > 1 << 46) | ((part == 1 << 46) & ((Y + whole) & 1 == 1)))
        wrong = np.flatnonzero(got != nearest)
        # all ones: from the power of two below, the exact result is a tie and goes back to it
        assert [(int(S[i]), int(Y[i])) for i in wrong] in ([], [((1 << 24) - 1, 1 << 23)])


@pytest.mark.gpu
@pytest.mark.parametrize("bits,amax,x", [(4, 7 / 4 - 2.0 ** -23, 1 / 8), (8, 127 / 64 - 2.0 ** -23, 1 / 128)])
@pytest.mark.parametrize("rounding", [aqt.ROUND_NEAREST_EVEN, aqt.ROUND_HALF_UP_FLOOR])
def test_scale_of_a_significand_of_ones(bits, amax, x, rounding):
    """x / s is the number after 0.5: code 1; with a reciprocal one unit low the quotient is 0.5 and the even code 0."""
    scale = 2.0 ** torch.arange(-60, 60, device="cuda", dtype=torch.float64)[:, None]
    rows = torch.cat([(torch.tensor([[amax, x, -x, 0.0]], device="cuda", dtype=torch.float64) * scale).float()] * 2)
    q, s = aqt.aqt_quantize(rows, bits, rounding=rounding)
    assert (s.view(torch.int32) & 0x7FFFFF == 0x7FFFFF).all()
    t = (rows[:, 1] / s).double()
    assert ((t > 0.5) & (t < 0.5000001)).all()
    assert torch.equal(q, torch.tensor([7 if bits == 4 else 127, 1, -1, 0], device="cuda", dtype=torch.int8).expand_as(q))
