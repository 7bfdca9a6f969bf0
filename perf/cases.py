"""What a user of this framework has it do: the measured cases and the ranges they stand for.

Every case runs one pass through the public entry points (``paper_2203_15952_b200.binding`` and
``.encoder``) on inputs made from a seed on the GPU.  The kinds:

  linear       one quantized layer on float activations: dynamic quantization, integer matmul,
               epilogue (a serving or evaluation forward of a single layer)
  ffn_pair     the feed-forward module of a Conformer block: two layers, the hidden tensor between
               them only as codes
  encoder      a stack of Conformer blocks' linears, from a streaming step of a few frames to a
               large offline batch
  ffn_host     the feed-forward module for activations in pinned host memory: copy in, two layers,
               copy out (a serving process that owns host buffers)
  weights      re-quantization of every encoder weight, as each training step does when the model is
               trained quantized from scratch
  weight_only  the layer of the weight-only configurations (int8 / int4 weights, float activations)
  train_layer  one layer's share of a training step: quantize the float weights, quantize the
               activations, forward matmul, straight-through backward (dx, dw, dbias)

Activations are normal, or Student-t with three degrees of freedom where heavy tails matter for the
abs-max scales; weights are normal with variance 1 / fan-in, biases small.
"""
import math

import torch

from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200.encoder import EncoderStack, FfnPair, QuantLinear, WeightArena
from paper_2203_15952_b200.inputs import LinearSpec, block_linears

ACTS = {"none": aqt.ACT_NONE, "swish": aqt.ACT_SWISH, "glu": aqt.ACT_GLU, "glu_swish": aqt.ACT_GLU_SWISH}
MAX_FLOPS = 2.0 * 65536 * 17 * (5 * 1024 * 1024 + 4 * 1024 * 4096 + 2 * 1024 * 1024)  # the d = 1024 encoder below
MAX_ELEMENTS = 1 << 28  # of the largest float tensor a drawn case makes


def _linear(name, M, K, N, bits_w=8, bits_a=8, act="none", scale="row", residual=False):
    return {"name": name, "kind": "linear", "M": M, "K": K, "N": N, "bits_w": bits_w, "bits_a": bits_a, "act": act, "scale": scale,
            "residual": residual}


def _encoder(name, M, d, blocks, bits_ffn=4, bits_attn=8, bits_a=8, tails=False):
    return {"name": name, "kind": "encoder", "M": M, "d": d, "ff": 4 * d, "blocks": blocks, "bits_ffn": bits_ffn, "bits_attn": bits_attn,
            "bits_a": bits_a, "tails": tails}


def listed():
    return [
        # the smallest call: one 8-bit layer on a short segment with one scale for the whole activation tensor
        _linear("linear_64x256x256", 64, 256, 256, scale="tensor"),
        # a streaming step's widest layer: eight frames, 4-bit weights kept packed
        _linear("linear_8x1024x4096_w4", 8, 1024, 4096, bits_w=4, act="swish"),
        # one layer of a mid-sized batch of ragged utterances: per-tensor activation scale (the usual
        # on-device form), residual add in the epilogue, a row count that is no multiple of any tile
        _linear("linear_7411x512x512_tensor", 7411, 512, 512, scale="tensor", residual=True),
        # a streaming step of eight frames through the whole 17-block encoder of width 512
        _encoder("encoder_stream_8_d512", 8, 512, 17),
        # one utterance of 1013 frames through one block, 4-bit weights and 4-bit activations
        _encoder("block_1013_d512_w4a4", 1013, 512, 1, bits_attn=4, bits_a=4),
        # the feed-forward module on a batch of 32 x 400 frames, 4-bit weights (the benchmark's own workload)
        {"name": "ffn_pair_12800_d512", "kind": "ffn_pair", "M": 12800, "d": 512, "ff": 2048, "bits_w": 4, "bits_a": 8},
        # the 17-block encoder on a batch of 64 x 400 frames: 4-bit feed-forward, 8-bit attention weights
        _encoder("encoder_25600_d512", 25600, 512, 17),
        # the large encoder on a batch of 128 x 512 frames with heavy-tailed activations
        _encoder("encoder_65536_d1024", 65536, 1024, 17, bits_attn=4, tails=True),
        # the feed-forward module called on pinned host buffers
        {"name": "ffn_host_12800_d512", "kind": "ffn_host", "M": 12800, "d": 512, "ff": 2048, "bits_w": 4, "bits_a": 8},
        # every weight of the d = 512 encoder from float to packed 4-bit codes and scales
        {"name": "weights_d512", "kind": "weights", "d": 512, "ff": 2048, "blocks": 17, "bits_ffn": 4, "bits_attn": 4},
        # first feed-forward layer with 4-bit weights and float activations
        {"name": "weight_only_12800x512x2048", "kind": "weight_only", "M": 12800, "K": 512, "N": 2048, "bits_w": 4, "act": "swish", "two_term": False},
        # first feed-forward layer in training
        {"name": "train_12800x512x2048", "kind": "train_layer", "M": 12800, "K": 512, "N": 2048, "bits_w": 4, "bits_a": 8},
    ]


def _log(rng, lo, hi, step=1):
    """A multiple of step, spread over the logarithm of [lo, hi]."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // step * step, max(-(-lo // step) * step, int(round(v / step)) * step))


def draw(rng):
    while True:
        c = _draw(rng)
        if work(c)["flops"] <= 0.5 * MAX_FLOPS and _largest_tensor(c) <= MAX_ELEMENTS:
            return c


def _draw(rng):
    kind = rng.choice(["linear", "linear", "ffn_pair", "encoder", "encoder", "ffn_host", "weights", "weight_only", "train_layer", "train_layer"])
    bits_w = rng.choice([4, 4, 8])
    if kind == "linear":
        act = rng.choice(["none", "none", "swish", "glu_swish"])
        return {"kind": kind, "M": _log(rng, 1, 65536), "K": _log(rng, 128, 4096, 32), "N": _log(rng, 128, 4096, 32), "bits_w": bits_w,
                "bits_a": rng.choice([8, 8, 4]), "act": act, "scale": rng.choice(["row", "row", "tensor"]),
                "residual": act == "none" and rng.random() < 0.5}
    if kind == "ffn_pair":
        d = rng.choice([256, 384, 512, 640, 768, 1024])
        return {"kind": kind, "M": _log(rng, 1, 65536), "d": d, "ff": 4 * d, "bits_w": bits_w, "bits_a": rng.choice([8, 8, 4])}
    if kind == "encoder":
        d = rng.choice([256, 384, 512, 512, 1024])
        return {"kind": kind, "M": _log(rng, 1, 65536), "d": d, "ff": 4 * d, "blocks": rng.randint(1, 17), "bits_ffn": bits_w,
                "bits_attn": rng.choice([4, 8]), "bits_a": rng.choice([8, 8, 4]), "tails": rng.random() < 0.3}
    if kind == "ffn_host":
        d = rng.choice([256, 512, 1024])
        return {"kind": kind, "M": _log(rng, 16, 32768), "d": d, "ff": 4 * d, "bits_w": bits_w, "bits_a": 8}
    if kind == "weights":
        d = rng.choice([256, 384, 512, 1024])
        return {"kind": kind, "d": d, "ff": 4 * d, "blocks": rng.randint(1, 17), "bits_ffn": 4, "bits_attn": rng.choice([4, 8])}
    K, N = _log(rng, 128, 4096, 4), _log(rng, 128, 4096, 8)
    if kind == "weight_only":
        return {"kind": kind, "M": _log(rng, 1, 65536), "K": K, "N": N, "bits_w": bits_w, "act": rng.choice(["none", "swish", "glu"]),
                "two_term": rng.random() < 0.3}
    K, N = _log(rng, 128, 4096, 32), _log(rng, 128, 4096, 32)
    return {"kind": kind, "M": _log(rng, 64, 65536), "K": K, "N": N, "bits_w": bits_w, "bits_a": rng.choice([8, 8, 4])}


def _largest_tensor(c):
    if c["kind"] in ("linear", "weight_only", "train_layer"):
        return c["M"] * max(c["K"], c["N"])
    if c["kind"] == "weights":
        return c["blocks"] * (8 * c["d"] * c["d"] + 4 * c["d"] * c["ff"])
    return c["M"] * c["ff"]


# ---------------------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape, std=1.0):
    return torch.randn(*shape, generator=g, device="cuda").mul_(std)


def _activations(g, M, K, tails=False):
    x = _normal(g, M, K)
    if tails:  # Student-t, three degrees of freedom, unit variance
        chi = torch.zeros_like(x)
        for _ in range(3):
            chi.addcmul_(*([_normal(g, M, K)] * 2))
        x.div_(chi.sqrt_())
    return x


def _quantized(g, spec, gain=1.0):
    return QuantLinear.from_float(spec, _normal(g, spec.N, spec.K, std=gain * spec.K ** -0.5))


def _block(g, specs, blocks):
    """One block's layers.  Those that add to the residual stream start 1 / sqrt(4 x blocks) smaller,
    so that the stream keeps its size through the stack, as it does in a trained model."""
    return [_quantized(g, s, (4 * blocks) ** -0.5 if s.name.endswith("2") or s.name == "attn_o" else 1.0) for s in specs]


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    g, kind, c = _gen(seed), case["kind"], case
    if kind == "linear":
        M, K, N, act = c["M"], c["K"], c["N"], ACTS[c["act"]]
        n_out = N // 2 if c["act"].startswith("glu") else N
        wq, s_w = aqt.aqt_quantize(_normal(g, N, K, std=K ** -0.5), c["bits_w"], pack=c["bits_w"] == 4)
        return {"kind": kind, "x": _activations(g, M, K), "wq": wq, "s_w": s_w, "bias": _normal(g, N, std=0.01),
                "residual": _normal(g, M, n_out) if c["residual"] else None, "bits_w": c["bits_w"], "bits_a": c["bits_a"], "act": act,
                "scale": aqt.SCALE_ROW if c["scale"] == "row" else aqt.SCALE_TENSOR, "y": torch.empty(M, n_out, device="cuda"),
                "ws": _bytes(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_FWD, M, N, K, c["bits_a"], c["bits_w"]))}
    if kind == "ffn_pair":
        specs = [LinearSpec("ffn_1", c["d"], c["ff"], aqt.ACT_SWISH, c["bits_w"], c["bits_a"]),
                 LinearSpec("ffn_2", c["ff"], c["d"], aqt.ACT_NONE, c["bits_w"], c["bits_a"])]
        return {"kind": kind, "pair": FfnPair(c["M"], [_quantized(g, s) for s in specs], "cuda"), "x": _activations(g, c["M"], c["d"]),
                "y": torch.empty(c["M"], c["d"], device="cuda")}
    if kind == "encoder":
        specs = block_linears(c["d"], c["ff"], c["bits_ffn"], c["bits_attn"], c["bits_a"])
        blocks = [_block(g, specs, c["blocks"]) for _ in range(c["blocks"])]
        return {"kind": kind, "stack": EncoderStack(c["M"], c["d"], c["ff"], blocks, "cuda"), "x": _activations(g, c["M"], c["d"], c["tails"])}
    if kind == "ffn_host":
        M, d, ff, bits = c["M"], c["d"], c["ff"], c["bits_w"]
        l1 = _quantized(g, LinearSpec("ffn_1", d, ff, aqt.ACT_SWISH, bits, 8))
        l2 = _quantized(g, LinearSpec("ffn_2", ff, d, aqt.ACT_NONE, bits, 8))
        x = torch.empty(M, d, pin_memory=True)
        x.copy_(_activations(g, M, d))
        return {"kind": kind, "x": x, "y": torch.empty(M, d, pin_memory=True), "l1": l1, "l2": l2,
                "ws": _bytes(aqt.aqt_workspace_bytes(aqt.OP_FFN_FWD, M, ff, d, 8, 4))}
    if kind == "weights":
        arena = WeightArena(block_linears(c["d"], c["ff"], c["bits_ffn"], c["bits_attn"], 8) * c["blocks"], "cuda")
        for w in arena.float_arena.values():
            w.normal_(std=w.shape[1] ** -0.5, generator=g)
        return {"kind": kind, "arena": arena}
    M, K, N = c["M"], c["K"], c["N"]
    if kind == "weight_only":
        n_out = N // 2 if c["act"].startswith("glu") else N
        wq, s_w = aqt.aqt_quantize(_normal(g, N, K, std=K ** -0.5), c["bits_w"], pack=c["bits_w"] == 4)
        op = aqt.OP_LINEAR_WEIGHT_ONLY_X2 if c["two_term"] else aqt.OP_LINEAR_WEIGHT_ONLY
        return {"kind": kind, "x": _activations(g, M, K), "wq": wq, "s_w": s_w, "bias": _normal(g, N, std=0.01), "bits_w": c["bits_w"],
                "act": ACTS[c["act"]], "precision": aqt.FLOAT_TF32X2 if c["two_term"] else aqt.FLOAT_TF32,
                "y": torch.empty(M, n_out, device="cuda"), "ws": _bytes(aqt.aqt_workspace_bytes(op, M, N, K, 0, c["bits_w"]))}
    ws = max(aqt.aqt_workspace_bytes(aqt.OP_QMATMUL, M, N, K, 8, c["bits_w"]), aqt.aqt_workspace_bytes(aqt.OP_LINEAR_BWD, M, N, K, 0, 0))
    return {"kind": kind, "w": _normal(g, N, K, std=K ** -0.5), "x": _activations(g, M, K), "dy": _normal(g, M, N, std=1e-3),
            "bias": _normal(g, N, std=0.01), "bits_w": c["bits_w"], "bits_a": c["bits_a"], "K": K, "y": torch.empty(M, N, device="cuda"),
            "ws": _bytes(ws)}


# ------------------------------------------------------------------------------------------ passes

def run(state):
    s, kind = state, state["kind"]
    if kind == "linear":
        return aqt.aqt_linear_fwd(s["x"], s["wq"], s["s_w"], s["bias"], s["residual"], bits_a=s["bits_a"], bits_w=s["bits_w"],
                                  a_scale_kind=s["scale"], act=s["act"], y=s["y"], workspace=s["ws"])
    if kind == "ffn_pair":
        return s["pair"].forward(s["x"], s["y"])
    if kind == "encoder":
        return s["stack"].forward(s["x"])
    if kind == "ffn_host":
        l1, l2 = s["l1"], s["l2"]
        return aqt.aqt_ffn_fwd(s["x"], l1.mm_weight, l1.s_w, l1.mm_bits, l2.mm_weight, l2.s_w, l2.mm_bits, s["y"], s["ws"])
    if kind == "weights":
        a = s["arena"]
        a.quantize()
        return [list(a.code_arena.values()), list(a.scale_arena.values())]
    if kind == "weight_only":
        return aqt.aqt_linear_fwd_weight_only(s["x"], s["wq"], s["s_w"], s["bias"], bits_w=s["bits_w"], precision=s["precision"], act=s["act"],
                                              y=s["y"], workspace=s["ws"])
    bits_a = 8 if s["bits_a"] == 8 else aqt.BITS_4_UNPACKED
    wq, s_w = aqt.aqt_quantize(s["w"], s["bits_w"], pack=s["bits_w"] == 4)
    xq, s_x = aqt.aqt_quantize(s["x"], s["bits_a"])
    y = aqt.aqt_qmatmul(xq, s_x, wq, s_w, s["bias"], K=s["K"], bits_a=bits_a, bits_w=s["bits_w"], y=s["y"], workspace=s["ws"])
    dx, dw, db = aqt.aqt_linear_bwd(s["dy"], xq, s_x, wq, s_w, K=s["K"], bits_a=bits_a, bits_w=s["bits_w"], workspace=s["ws"])
    return {"y": y, "dx": dx, "dw": dw, "dbias": db}


# ------------------------------------------------------------------------------- work and tolerance

def work(case):
    c, kind = case, case["kind"]
    if kind in ("linear", "weight_only"):
        M, K, N = c["M"], c["K"], c["N"]
        n_out = N // 2 if c["act"].startswith("glu") else N
        out = M * n_out * (2 if c.get("residual") else 1)
        return {"bytes": 4 * M * K + N * K * c["bits_w"] / 8 + 8 * N + 4 * out, "flops": 2.0 * M * N * K}
    if kind in ("ffn_pair", "ffn_host"):
        M, d, ff = c["M"], c["d"], c["ff"]
        return {"bytes": 8 * M * d + 2 * d * ff * c["bits_w"] / 8 + 4 * (d + ff), "flops": 4.0 * M * d * ff}
    if kind == "train_layer":
        M, K, N = c["M"], c["K"], c["N"]
        return {"bytes": 4 * (2 * M * K + 2 * M * N + 2 * N * K + 2 * N), "flops": 6.0 * M * N * K}
    d, ff = c["d"], c["ff"]
    ffn, attn = c["blocks"] * 4 * d * ff, c["blocks"] * 7 * d * d
    if kind == "weights":
        return {"bytes": 4 * (ffn + attn) + ffn * c["bits_ffn"] / 8 + attn * c["bits_attn"] / 8, "flops": 0}
    return {"bytes": 8 * c["M"] * d + ffn * c["bits_ffn"] / 8 + attn * c["bits_attn"] / 8, "flops": 2.0 * c["M"] * (ffn + attn)}


def tolerance(case):
    """About four times what one path shows against double precision (single layers), or against itself
    with every channel scale moved by one unit in the last place (chains, where such a change flips a
    few codes: 5e-5 in a feed-forward pair; 5e-3 and, with 4-bit activations, 2.6e-2 after 16 or 17 blocks)."""
    kind = case["kind"]
    if kind == "weights":
        return "exact"  # codes and scales are whole numbers and one IEEE division
    if kind == "linear":
        return {"rel": 4e-7}  # exact integer sums, a handful of binary32 operations: 9e-8 seen
    if kind in ("ffn_pair", "ffn_host"):
        return {"rel": 3e-4}
    if kind == "encoder":
        return {"rel": 2e-2 if case["bits_a"] == 8 else 1e-1}
    if kind == "weight_only":
        return {"rel": 5e-6 if case["two_term"] else 2e-3}  # tf32 activations: 5e-4 seen; two terms: 1.1e-6
    return {"rel": 3e-3}  # tf32 gradients: 8e-4 seen
