"""The one-launch chain of layers for a few rows (aqt_chain_fwd) gives the bits of the per-layer calls.

The per-layer calls are checked against the CPU oracle in the other files; here every chain result is
compared with them bit for bit, and a chain without a transcendental with the oracle itself."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200 import inputs as gen
from paper_2203_15952_b200.encoder import EncoderStack, FfnPair, QuantLinear

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _stack(M, d, ff, n_blocks, bits, seed, bias=False, **kw):
    g = torch.Generator(device=DEV).manual_seed(seed)
    specs = gen.block_linears(d, ff, *bits)
    blocks = [[QuantLinear.from_float(s, torch.randn((s.N, s.K), generator=g, device=DEV) * (0.5 * s.K ** -0.5),
                                      torch.randn(s.N, generator=g, device=DEV) * 0.1 if bias else None) for s in specs]
              for _ in range(n_blocks)]
    return EncoderStack(M, d, ff, blocks, DEV, **kw), torch.randn((M, d), generator=g, device=DEV)


def _layer_by_layer(stack, x):
    src = x
    for b, layers in enumerate(stack.blocks):
        dst = torch.empty_like(x)
        stack.block.forward(layers, src, dst)
        src = dst
    return src, stack.block.qkv.clone()


@pytest.mark.parametrize("M,d,ff,blocks,bits", [
    (1, 512, 2048, 2, (4, 8, 8)), (8, 512, 2048, 3, (4, 8, 8)), (9, 256, 1024, 2, (8, 4, 4)), (16, 384, 1536, 2, (4, 4, 8)),
    (17, 512, 2048, 1, (8, 8, 8)), (56, 512, 2048, 1, (4, 8, 4)), (57, 256, 1024, 1, (4, 4, 4)), (112, 512, 2048, 1, (4, 8, 8)),
    (5, 1024, 4096, 1, (4, 4, 8)), (90, 1024, 4096, 1, (4, 8, 8)), (3, 256, 1024, 27, (4, 8, 8))])
def test_encoder_chain_gives_the_per_layer_bits(M, d, ff, blocks, bits):
    """Row counts around an 8-row tile, one and two tiles per cluster, several clusters, every mix of packed and int8 weights, a stack longer than one launch takes; some rows zero or tiny."""
    stack, x = _stack(M, d, ff, blocks, bits, M + d, bias=True, rounding=aqt.ROUND_HALF_UP_FLOOR if M % 2 else aqt.ROUND_NEAREST_EVEN)
    if M > 2:
        x[1] = 0.0
        x[2] *= 1e-30
    want, want_qkv = _layer_by_layer(stack, x)
    stack.block.qkv.fill_(float("nan"))
    assert aqt.chain_encoder(x, stack.blocks, stack.block.qkv, stack.h0, stack.block.run.rounding)
    assert torch.equal(stack.h0.view(torch.int32), want.view(torch.int32))
    assert torch.equal(stack.block.qkv.view(torch.int32), want_qkv.view(torch.int32))
    out = stack.forward(x)
    assert torch.equal(out.view(torch.int32), want.view(torch.int32))
    assert aqt.aqt_device_status() == 0


@pytest.mark.parametrize("M,d,ff,bits_w,bits_a", [(1, 256, 1024, 4, 8), (8, 512, 2048, 4, 8), (30, 640, 2560, 8, 4), (100, 768, 3072, 4, 8),
                                                  (16, 1024, 4096, 8, 8)])
def test_ffn_chain_gives_the_per_layer_bits(M, d, ff, bits_w, bits_a):
    g = torch.Generator(device=DEV).manual_seed(M + d)
    specs = [gen.LinearSpec("ffn_1", d, ff, gen.ACT_SWISH, bits_w, bits_a), gen.LinearSpec("ffn_2", ff, d, gen.ACT_NONE, bits_w, bits_a)]
    layers = [QuantLinear.from_float(s, torch.randn((s.N, s.K), generator=g, device=DEV) * (s.K ** -0.5)) for s in specs]
    x = torch.randn((M, d), generator=g, device=DEV)
    y, y_ref = torch.full((M, d + 4), 7.0, device=DEV)[:, :d], torch.empty((M, d), device=DEV)
    assert aqt.chain_ffn(x, *layers, y, aqt.ROUND_NEAREST_EVEN)
    FfnPair(M, layers, DEV, fused=False).forward(x, y_ref)
    assert torch.equal(y, y_ref)
    # the entry point for host buffers takes the same path
    yh = torch.empty((M, d), pin_memory=True)
    aqt.aqt_ffn_fwd(x.cpu().pin_memory(), layers[0].mm_weight, layers[0].s_w, layers[0].mm_bits, layers[1].mm_weight, layers[1].s_w,
                    layers[1].mm_bits, yh, bits_a=bits_a)
    torch.cuda.synchronize()
    assert torch.equal(yh, y_ref.cpu())


def test_chain_without_activation_matches_the_oracle():
    """Two layers without a transcendental: codes, sums and outputs are IEEE operations only."""
    M, K, N = 13, 256, 512
    x = gen.normal(70, 1, M, K)
    w1, w2 = gen.weight(70, 2, K, N), gen.weight(70, 3, N, K)
    (q1, s1), (q2, s2) = orc.quantize(w1, 8, orc.AXIS_ROW), orc.quantize(w2, 4, orc.AXIS_ROW)
    u = orc.linear_fwd(x, q1, s1)
    want = orc.linear_fwd(u, q2, s2)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    l1 = QuantLinear(gen.LinearSpec("a", K, N, gen.ACT_NONE, 8, 8), dev(q1), dev(s1.reshape(-1)), None)
    l2 = QuantLinear(gen.LinearSpec("b", N, K, gen.ACT_NONE, 4, 8), dev(orc.pack_int4(q2)), dev(s2.reshape(-1)), None)
    y = torch.empty((M, K), device=DEV)
    assert aqt.chain_ffn(dev(x), l1, l2, y, aqt.ROUND_NEAREST_EVEN)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))


def test_chain_declines_what_it_cannot_take():
    """Widths that are no multiple of 128 and too many rows go layer by layer, with the same entry points."""
    stack, x = _stack(8, 144, 576, 1, (4, 8, 8), 1)
    assert not aqt.chain_encoder(x, stack.blocks, stack.block.qkv, stack.h0, stack.block.run.rounding)
    want, _ = _layer_by_layer(stack, x)
    assert torch.equal(stack.forward(x), want)
    stack, x = _stack(aqt.CHAIN_MAX_ROWS + 1, 256, 1024, 1, (4, 8, 8), 2)
    assert not aqt.chain_encoder(x, stack.blocks, stack.block.qkv, stack.h0, stack.block.run.rounding)
