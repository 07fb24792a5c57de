"""fp32 layers of more tokens than one fused decode launch takes: token counts
around the token groups (4 and 8), the four-token router and the scratch slice,
widths that are no multiple of a warp's 128 columns or 8 rows, one to 256
experts, and all three activations.  Tolerances are those of the other parity
tests."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2605_28283_gb300 import workloads as wl
from parity import Y_TOL, check_route_selection, check_y, f32, logit_tolerance, to_host
from test_gpu_parity import dev, layer_parity, run_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [9, 10, 12, 63, 255, 256, 257, 261, 608, 609, 1024, 1027])
def test_ffn32_token_counts(pp, T):
    layer_parity(pp, "tiny_relu_f32", T, 0.9, d=128, E=6)


@pytest.mark.parametrize("d,E,T,p", [(64, 1, 9, 0.5), (68, 3, 20, 0.7), (1004, 33, 40, 0.9), (128, 256, 300, 0.95),
                                     (8192, 4, 11, 0.6), (256, 16, 64, 1.0)])
@pytest.mark.parametrize("act", ["relu", "gelu_tanh", "swiglu"])
def test_ffn32_shapes(pp, d, E, T, p, act):
    w = replace(wl.scaled(wl.WORKLOADS["tiny_relu_f32"], d, E), act=act)
    L = wl.host_layer(w, T, seed=3)
    pf = f32(p)
    counts, ids, logits, y, status = run_layer(pp, w, L, pf)
    assert status == pp.PP_OK
    g = oracle.logits(L.x, L.Wr)
    assert np.all(np.abs(logits - g) <= logit_tolerance(L.x, L.Wr))
    eps = np.abs(logits - g).max(axis=1)
    unique, _ = check_route_selection(counts, ids, g, eps, pf, "min_prefix")
    rc, ri, _, _ = oracle.select(g, pf, "min_prefix")
    check_y(L, y, rc, ri, g, E, act, "sigmoid", Y_TOL["f32"], unique, counts, ids)


@pytest.mark.parametrize("rule,p", [("paper", 0.8), ("topk", 3.0), ("lte", 0.9), ("lte", 1.0)])
def test_ffn32_rules(pp, rule, p):
    layer_parity(pp, "tiny_relu_f32", 50, p, rule, "none" if rule == "lte" else "sigmoid")


def test_ffn32_given_selection_with_a_zero_gate(pp):
    """pp_sparse_ffn: a selected expert with gate 0 adds nothing, a repeated id
    adds its gates, and nothing is read that an earlier call left behind."""
    import torch
    T, w = 13, wl.scaled(wl.WORKLOADS["tiny_relu_f32"], 128, 8)
    L = wl.host_layer(w, T, seed=5)
    ids = np.full((T, 8), -1, np.int32)
    gates = np.zeros((T, 8), np.float32)
    ids[:, 0], ids[:, 1], ids[:, 2] = 3, 5, 3
    gates[:, 0], gates[:, 1], gates[:, 2] = 0.25, 0.0, 0.5
    counts = np.full(T, 3, np.int32)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    x, Wr, Wu, Wd = dev(L.x), dev(L.Wr), dev(L.Wu), dev(L.Wd)
    y = torch.empty_like(x)
    pp.pp_layer(desc, x, T, Wr, None, Wu, Wd, 1.0, None, y, ws)  # every expert: fills the scratch
    pp.pp_sparse_ffn(desc, x, T, None, Wu, Wd, pp.Selection(dev(ids), dev(counts), dev(gates)), y, ws)
    torch.cuda.synchronize()
    h = np.maximum(L.x.astype(np.float64) @ L.Wu[192:256].astype(np.float64).T, 0.0) * 0.75
    ref = h @ L.Wd[:, 192:256].astype(np.float64).T
    err = np.abs(to_host(y) - ref).max(axis=1) / np.abs(ref).max(axis=1)
    assert err.max() <= Y_TOL["f32"]
