"""The tf32 form of the weight-only layer on CTA pairs with an activation, against the CPU oracle (needs a B200): sizes that have no
binary16 form, and those of calls whose workspace has no room for it.

Tolerance per pre-activation z:  |z - z_ref| <= (2^-10 + K * 2^-24) * s_w * sum_k |x * wq| + 2^-23 * |z_ref|, through the activation by its
Lipschitz constant (Swish 1.1; gates: 1 for the values, |value| / 4 for the gates), and 4e-7 |z| for the kernel's sigmoid."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,act", [(12800, 2048, 512, orc.ACT_SWISH), (5000, 3072, 768, orc.ACT_SWISH), (4100, 2048, 1024, orc.ACT_GLU_SWISH),
                                       (12805, 1000, 260, orc.ACT_SWISH), (9700, 2056, 516, orc.ACT_GLU)])
def test_tf32_pairs_with_an_activation(M, N, K, act):
    assert aqt.aqt_plan_qmatmul(M, N, K, 0, 4, act, float_kind=True) == "pair256s4e8"
    x = gen.normal(11, 17, M, K)
    wq, s_w = orc.quantize(gen.normal(11, 904, N, K, std=1.0 / np.sqrt(K)), 4, orc.AXIS_ROW)
    bias = gen.normal(11, 19, 1, N, std=0.05)[0]
    n_out = N // 2 if act >= orc.ACT_GLU else N
    y = torch.full((M, n_out), float("nan"), device="cuda")
    tf32_bytes = aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, 0, N, K, 0, 4)  # of no rows: room for tf32 operands alone
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, orc.pack_int4(wq), s_w, bias)]
    aqt.aqt_linear_fwd_weight_only(*dev, bits_w=4, act=act, y=y, workspace=torch.empty(tf32_bytes, dtype=torch.uint8, device="cuda"))
    assert aqt.aqt_device_status() == 0
    rows = np.unique(np.concatenate([np.arange(0, 260), np.arange(M - 260, M), np.random.default_rng(4).integers(0, M, 200)]))
    y_ref, z, mag = orc.linear_weight_only_f64(x[rows], wq, s_w, bias=bias, act=act, return_parts=True)
    dz = (2.0 ** -10 + K * 2.0 ** -24) * mag + 2.0 ** -23 * np.abs(z)
    d = dz[:, :n_out]
    if act >= orc.ACT_GLU:
        d = d + (np.abs(z[:, :n_out]) + d) * 0.25 * dz[:, n_out:]
    if act in (orc.ACT_SWISH, orc.ACT_GLU_SWISH):
        d = 1.1 * d
    tol = d + 4e-7 * np.abs(z[:, :n_out]) + 1e-30 + 2.0 ** -23 * np.abs(y_ref)
    assert np.all(np.abs(y.cpu().numpy()[rows].astype(np.float64) - y_ref) <= tol)
