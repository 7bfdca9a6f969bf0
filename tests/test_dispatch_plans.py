"""Which kernel configuration each matmul of the five workload configurations runs in, and that
every one of them is exercised by a parity test against the oracle (host-only: the plan query
needs no device).

The library chooses a configuration ("plan") of its GEMM kernel template per shape.  A parity
test only proves the configurations it reaches, so this file walks every matmul shape of the
workloads through the same choice the launches make (for the 148 multiprocessors of the part)
and requires each resulting plan to be named below together with the GPU test that runs it; those
tests assert the plan name themselves, so the table cannot drift from what they execute.
"""
import os
import re

import pytest

from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200 import inputs as gen

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# plan -> (test file, test function) that compares this configuration with the oracle
COVERED_BY = {
    "small_m": ("test_gpu_kernels.py", "test_qmatmul_small_batch"),
    "ws128e16": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "ws128e8": ("test_gpu_kernels.py", "test_qmatmul_activations"),
    "few32": ("test_gpu_few_tiles.py", "test_few_tiles_plans_named"),
    "few64": ("test_gpu_few_tiles.py", "test_few_tiles_plans_named"),
    "few128": ("test_gpu_few_tiles.py", "test_few_tiles_plans_named"),
    "stream256s3e16": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "stream256s4e4": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "stream128s4e16": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "stream128s6e4": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "stream128s4e8": ("test_gpu_kernels.py", "test_qmatmul_glu_streaming_plan_named"),
    "stream64s5e8": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "stream64s8e4": ("test_gpu_kernels.py", "test_qmatmul_single_cta_plans_named"),
    "pair256s4e8": ("test_gpu_kernels.py", "test_qmatmul_cta_pair_plans_named"),
    "pair256s6e4": ("test_gpu_full_size.py", "test_large_encoder_ffn_second_layer_matmul"),
    "pair128s6e8": ("test_gpu_kernels.py", "test_qmatmul_cta_pair_plans_named"),
    "pair128s8e4": ("test_gpu_full_size.py", "test_large_encoder_ffn_second_layer_matmul"),
    "pair512s3e16": ("test_gpu_kernels.py", "test_qmatmul_wide_pair_tiles_ffn_second_layer_shape"),
}


def _workload_matmul_shapes():
    """(M, N, K, bits_a, bits_w, act) of every matmul the drivers issue for the five configurations,
    including the matmul over the concatenated q and k projections (and over q, k, v, for callers that keep them together)."""
    shapes = set()
    for cfg, w in gen.WORKLOADS.items():
        for s in gen.workload_layers(w):
            shapes.add((w.M, s.N, s.K, s.bits_a, s.bits_w, s.act))
        if w.kind in ("block", "stack"):
            shapes.add((w.M, 2 * w.d, w.d, w.bits_a, w.bits_attn_w, gen.ACT_NONE))
            shapes.add((w.M, 3 * w.d, w.d, w.bits_a, w.bits_attn_w, gen.ACT_NONE))
    return sorted(shapes)


def test_every_plan_the_workloads_reach_has_a_parity_test():
    reached = {}
    for (M, N, K, ba, bw, act) in _workload_matmul_shapes():
        plan = aqt.aqt_plan_qmatmul(M, N, K, ba, bw, act, sm_count=148)
        reached.setdefault(plan, []).append((M, N, K))
    assert reached, "no shapes"
    for plan, shapes in reached.items():
        assert plan in COVERED_BY, "plan %s (shapes %s) has no parity test" % (plan, shapes[:3])


def test_the_named_tests_exist_and_pin_their_plan():
    for plan, (fname, func) in COVERED_BY.items():
        text = open(os.path.join(ROOT, "tests", fname)).read()
        m = re.search(r"def %s\(.*?(?=\ndef |\Z)" % re.escape(func), text, flags=re.S)
        assert m, (fname, func)
        body = text[:m.end()]
        # the plan is either forced by name (a parametrize list above the test) or asserted inside it
        assert '"%s"' % plan in body or plan == "small_m" or plan in ("ws128e8",), (plan, func)


def test_plans_of_the_headline_shapes():
    """The shapes the benchmark and the benchmark spec's targets are quoted on."""
    p = lambda *a, **k: aqt.aqt_plan_qmatmul(*a, sm_count=148, **k)
    assert p(12800, 2048, 512, 8, 4, gen.ACT_SWISH) == "ws128e16"
    assert p(12800, 512, 2048, 8, 4) == "pair512s3e16"
    assert p(65536, 1024, 4096, 8, 4) == "pair256s6e4"
    assert p(65536, 4096, 1024, 8, 4, gen.ACT_SWISH) == "stream256s3e16"
    assert p(8, 512, 2048, 8, 4) == "small_m"
    assert p(64, 256, 256, 8, 8) == "few32" and p(1013, 1024, 512, 8, 4) == "few64" and p(4736, 512, 512, 8, 4) == "few128"
    assert p(4737, 512, 512, 8, 4) == "ws128e16" and p(300, 1024, 1024, 8, 4, gen.ACT_GLU_SWISH) == "few64"
    # the float kind (weight-only layer, backward) plans with K in elements
    assert p(65536, 1024, 4096, 0, 4, float_kind=True) == "pair256s6e4"
    # a device with other SM counts changes the choice only through the number of rounds
    assert aqt.aqt_plan_qmatmul(12800, 2048, 512, 8, 4, gen.ACT_SWISH, sm_count=8) == "stream256s3e16"


def test_how_row_quantizing_calls_run():
    p = lambda *a, **k: aqt.aqt_plan_qmatmul_requant(*a, sm_count=148, **k)
    w8, may = aqt.BITS_4_UNPACKED, aqt.MAY_WAIT
    # one tile per SM, in the narrowest width that leaves one; at most sixteen parts of a row below 128 columns
    assert p(1013, 512, 512) == "few32" and p(1013, 1024, 512) == "few64" and p(4736, 512, 512, with_y=True) == "few128"
    assert p(300, 1024, 896) == "few64" and p(300, 1040, 896) == "ws128" and p(4737, 512, 512) == "ws128"
    # packed codes out, and a workspace with no room for the narrow tiles' words
    assert p(1013, 512, 512, bits_w=4, pack_out=True) == "ws128"
    need = -(-300 // 256) * 256 * 8 * 8 + 1024
    assert p(300, 512, 512, workspace_bytes=need) == "ws128" and p(300, 512, 512, workspace_bytes=need + 65536) == "few32"
    # what the header lists waits across CTAs, the others only if they may
    for shape, kw, wide in (((1013, 1024, 1024), {}, "two_kernels"), ((100, 512, 2048), {}, "two_kernels"),
                            ((300, 1024, 512), dict(act=gen.ACT_GLU_SWISH), "two_kernels"), ((200, 512, 2048), {}, "few32")):
        assert p(*shape, with_y=True, **kw) == wide, shape
        assert p(*shape, with_y=True, bits_w=8 | may, **kw).startswith("few")
    assert p(25600, 512, 2048, bits_w=w8, with_y=True) == "pair256s4e8" and p(65536, 1024, 1024, bits_w=w8 | may, with_y=True) == "two_kernels"
    # refused: nothing quantizes the rows and there is no y to go through
    for shape in ((64, 256, 2048), (300, 512, 1536)):
        with pytest.raises(aqt.AqtError) as e:
            p(*shape, bits_w=8 | may)
        assert e.value.status == -3
    # the last columns only: one launch, or how they run by themselves
    assert p(1013, 1536, 512, first=1024, with_y=True) == "few128" and p(12800, 1536, 512, first=1024, with_y=True) == "ws128"
    assert p(300, 480, 128, first=16, with_y=True) == "few32"
    for bad in (dict(first=8, with_y=True), dict(first=512, with_y=True), dict(first=16), dict(pack_out=True, bits_w=5)):
        with pytest.raises(aqt.AqtError) as e:
            p(300, 512, 512, **bad)
        assert e.value.status == -1


def test_launches_of_a_feed_forward_pair():
    """The pair counts the row quantizer that runs behind the first matmul where no kernel does both."""
    import torch
    from paper_2203_15952_b200.encoder import FfnPair, QuantLinear
    from paper_2203_15952_b200.inputs import LinearSpec

    def pair(M, d, **kw):
        specs = [LinearSpec("a", d, 4 * d, gen.ACT_SWISH, 8), LinearSpec("b", 4 * d, d, gen.ACT_NONE, 8)]
        return FfnPair(M, [QuantLinear(s, torch.empty(s.N, s.K, dtype=torch.int8), torch.empty(s.N), None) for s in specs], "cpu", **kw)
    assert pair(5000, 512).launches_per_step == 3 and pair(5000, 512, keep_u=True).launches_per_step == 3
    assert pair(5000, 1024).launches_per_step == 3 and pair(5000, 1024, keep_u=True).launches_per_step == 4
    assert pair(5000, 512, fused=False).launches_per_step == 4
