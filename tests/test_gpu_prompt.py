"""The prompt path (bf16, more than 256 tokens) at the sizes where it can go
wrong: lists around the 128-row work item, one expert to 256, whole and halved
work items, widths of one K chunk or no multiple of 64 or 128, selections from
empty to every expert (past the row buffer's capacity), and a selection given
by the caller with repeated ids.  Tolerances are those of the other parity
tests."""
import numpy as np
import pytest

from paper_2605_28283_gb300 import workloads as wl
from parity import Y_TOL, check_select_exact, f32, layer_inputs, to_host
from test_gpu_parity import dev, layer_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [257, 300, 383, 384, 385, 513])
@pytest.mark.parametrize("E", [1, 2, 40])
def test_prompt_token_counts(pp, T, E):
    layer_parity(pp, "llama3_8b_batched", T, 0.7, d=192, E=E)


@pytest.mark.parametrize("d,E,T", [(64, 30, 260), (72, 90, 300), (200, 256, 300), (1000, 33, 270), (2056, 20, 290)])
@pytest.mark.parametrize("name", ["llama3_8b_batched", "gpt2m_gelu_bf16"])
def test_prompt_widths(pp, name, d, E, T):
    layer_parity(pp, name, T, 0.8, d=d, E=E)


@pytest.mark.parametrize("rule,p,gate", [("topk", 1.0, "none"), ("topk", 9.0, "sigmoid"), ("paper", 0.9, "sigmoid"),
                                         ("min_prefix", 0.0, "sigmoid"), ("min_prefix", 1.0, "none"),
                                         ("lte", 0.97, "none"), ("lte", 1.0, "none"), ("lte", 0.0, "none")])
def test_prompt_rules(pp, rule, p, gate):
    layer_parity(pp, "llama3_8b_batched", 270, p, rule, gate, d=256, E=100)


def test_prompt_large_lists(pp):
    """600 tokens on 12 experts: several items per expert, more items than SMs are needed."""
    layer_parity(pp, "llama3_8b_batched", 600, 0.95, d=320, E=12)


@pytest.mark.parametrize("d,E,T,p", [(64, 1, 1025, 0.5), (64, 40, 1100, 0.8), (200, 12, 1300, 0.95), (1000, 70, 1030, 0.7),
                                     (2312, 9, 1041, 0.9), (264, 100, 1027, 1.0)])
@pytest.mark.parametrize("name", ["llama3_8b_batched", "gpt2m_gelu_bf16"])
def test_prompt_down_projection_by_token_rows(pp, name, d, E, T, p):
    """Above 1024 tokens the down projection has tokens as the M operand: full
    and partial groups of 32 rows, partial column slices, and with p = 1 pairs
    past the row buffer's capacity."""
    layer_parity(pp, name, T, p, d=d, E=E)


def test_prompt_repeated_calls(pp):
    """Back to back on one workspace, alternating lengths (and so kernels): every
    call gives the same bits."""
    import torch
    Ts, p = (1500, 300, 1100), f32(0.8)
    w, L = layer_inputs("llama3_8b_batched", max(Ts), d=1304, E=30)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, max(Ts))
    x, Wr, Wg, Wu, Wd = (dev(a) for a in (L.x, L.Wr, L.Wg, L.Wu, L.Wd))
    ref = {}
    for rep in range(8):
        for T in Ts:
            y = torch.empty_like(x[:T])
            pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, None, y, ws)
            ref.setdefault(T, []).append(y)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    for T in Ts:
        assert all(torch.equal(y, ref[T][0]) for y in ref[T]), T


@pytest.mark.parametrize("E", [20, 50, 120, 250])
@pytest.mark.parametrize("rule,p", [("min_prefix", 0.7), ("min_prefix", 1.0), ("paper", 0.9), ("topk", 6.0), ("lte", 0.9)])
def test_prompt_route_matches_select(pp, E, rule, p):
    """The warp-per-token selection of pp_route on its own logits, which hold
    many exact ties: the oracle's rule on the same logits, bit for bit."""
    import torch
    T, d = 700, 64
    rng = np.random.default_rng(E)
    x = np.zeros((T, d), np.float32)
    x[np.arange(T), rng.integers(0, d, T)] = 1.0  # a logit is one entry of W_r
    Wr = (np.round(rng.standard_normal((E, d)) * 4) / 2).astype(np.float32)
    desc = pp.make_desc(d, E, "bf16", "swiglu", "sigmoid", rule)
    ws = pp.alloc_workspace(desc, T)
    sel = pp.Selection.empty(T, E, "cuda")
    pp.pp_route(desc, dev(wl.f32_to_bf16_bits(x)), T, dev(wl.f32_to_bf16_bits(Wr)), f32(p), sel, ws)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    lg = to_host(sel.logits)
    assert np.array_equal(lg, x @ Wr.T)
    check_select_exact(to_host(sel.counts), to_host(sel.ids), lg.astype(np.float64), f32(p), rule)


def test_prompt_given_selection_with_repeated_ids(pp):
    """pp_sparse_ffn: gates of a repeated id add up; the call equals the one
    with the ids merged."""
    import torch
    T, E = 300, 24
    w, L = layer_inputs("llama3_8b_batched", T, d=256, E=E)
    rng = np.random.default_rng(2)
    first = rng.integers(0, E, (T, 2)).astype(np.int32)
    first[:, 1] = (first[:, 0] + 1 + first[:, 1] % (E - 1)) % E
    ids, gates = np.full((T, E), -1, np.int32), np.zeros((T, E), np.float32)
    ids[:, :2], gates[:, :2] = first, (0.75, 0.5)
    rep, rgates = ids.copy(), gates.copy()
    rep[:, 2], rgates[:, 0], rgates[:, 2] = first[:, 0], 0.25, 0.5
    desc = pp.make_desc(w.d_model, E, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    x, Wg, Wu, Wd = dev(L.x), dev(L.Wg), dev(L.Wu), dev(L.Wd)
    ys = []
    for i, g, k in ((ids, gates, 2), (rep, rgates, 3)):
        y = torch.empty_like(x)
        pp.pp_sparse_ffn(desc, x, T, Wg, Wu, Wd, pp.Selection(dev(i), dev(np.full(T, k, np.int32)), dev(g)), y, ws)
        ys.append(y)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    assert torch.equal(ys[0], ys[1])
