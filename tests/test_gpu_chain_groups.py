"""Layers of a chain that read the same input run as one where they look alike: the bits of the single layers (needs a B200)."""
import ctypes

import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu


class Layer(ctypes.Structure):
    _fields_ = [(n, ctypes.c_void_p) for n in ("wq", "s_w", "bias", "y")] + [("ldy", ctypes.c_int64)] + [
        (n, ctypes.c_int32) for n in ("N", "K", "bits_w", "bits_a", "act", "flags")] + [("residual_scale", ctypes.c_float), ("reserved", ctypes.c_int32)]


# (N, side, bits_w, act, bias, y) per layer: groups of two, three and four, at the start, inside and at the end; layers that are beside one another
# but differ (width, activation), too wide for one epilogue (4 x 640 / 16 columns), a group without all outputs and biases, a side step at the end
CHAINS = {
    "two_first": [(256, 1, 8, 0, 1, 1), (256, 0, 8, 0, 0, 1), (128, 0, 8, 0, 1, 1)],
    "four": [(128, 0, 4, 0, 1, 1), (384, 1, 4, 0, 1, 1), (384, 1, 4, 0, 0, 0), (384, 1, 4, 0, 1, 1), (384, 0, 4, 0, 1, 1), (256, 0, 8, 1, 1, 1)],
    "three_last": [(256, 0, 8, 1, 1, 1), (640, 1, 4, 0, 1, 1), (640, 1, 4, 0, 1, 1), (640, 0, 4, 0, 1, 1)],
    "too_wide": [(640, 1, 8, 0, 1, 1), (640, 1, 8, 0, 1, 1), (640, 1, 8, 0, 1, 1), (640, 0, 8, 0, 1, 1), (128, 0, 4, 0, 1, 1)],
    "unlike": [(256, 1, 8, 0, 1, 1), (512, 1, 8, 0, 1, 1), (256, 1, 8, 1, 1, 1), (256, 0, 8, 0, 1, 1), (256, 0, 8, 0, 1, 1)],
    "side_last": [(256, 0, 4, 0, 1, 1), (128, 1, 8, 0, 1, 1), (128, 1, 8, 0, 1, 1)],
}


@pytest.mark.parametrize("name", list(CHAINS))
@pytest.mark.parametrize("M,K,bits_a", [(3, 256, 8), (16, 512, 4), (61, 128, 8)])
def test_groups_give_the_bits_of_the_layers(name, M, K, bits_a):
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn(M, K, generator=g, device="cuda")
    x[1] = 0.0
    layers, keep, want, got = [], [], [], []
    cur, width = x, K
    for N, side, bits_w, act, has_bias, has_y in CHAINS[name]:
        wq, s_w = aqt.aqt_quantize(torch.randn(N, width, generator=g, device="cuda") * width ** -0.5, bits_w, pack=bits_w == 4)
        bias = torch.randn(N, generator=g, device="cuda") if has_bias else None
        out = aqt.aqt_linear_fwd(cur, wq, s_w, bias, None, 1.0, bits_a=bits_a, bits_w=bits_w, act=act)
        y = torch.full((M, N), float("nan"), device="cuda")
        layers.append(Layer(wq.data_ptr(), s_w.data_ptr(), bias.data_ptr() if has_bias else None, y.data_ptr() if has_y else None, N, N, width, bits_w, bits_a,
                            act, side, 1.0, 0))
        keep += [wq, s_w, bias, y, out]
        if has_y:
            want.append(out)
            got.append(y)
        if not side:
            cur, width = out, N
    arr = (Layer * len(layers))(*layers)
    fwd = aqt.lib().aqt_chain_fwd
    fwd.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    assert fwd(x.data_ptr(), K, M, ctypes.cast(arr, ctypes.c_void_p), len(layers), aqt.ROUND_NEAREST_EVEN, torch.cuda.current_stream().cuda_stream) == 0
    for a, b in zip(want, got):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    assert aqt.aqt_device_status() == 0
