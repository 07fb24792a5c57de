"""The union kernel (bf16, 5 to 256 tokens) at the sizes where it can go wrong:
token counts around the MMA's column granularity, the 128-token tile of the
router and both ends of the range; unions from empty to every expert, so that
a CTA has no unit, one, one full tile, or two; rings of one and of two chunks a
stage; widths that are no multiple of 64 or 128; and repeated calls on one
workspace (the grid barrier's counter and every ring start where the previous
call left them).  Tolerances are those of the other parity tests."""
import numpy as np
import pytest

import oracle
from paper_2605_28283_gb300 import workloads as wl
from parity import Y_TOL, f32, layer_inputs, rel_err_per_token, to_host
from test_gpu_parity import dev, layer_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [5, 15, 16, 17, 31, 33, 63, 65, 127, 128, 129, 255, 256])
def test_union_token_counts(pp, T):
    layer_parity(pp, "llama3_8b_batched", T, 0.7, d=704, E=90)


@pytest.mark.parametrize("E,T,rule,p", [(256, 20, "min_prefix", 1.0), (256, 256, "min_prefix", 0.9), (256, 5, "topk", 1.0),
                                        (3, 9, "topk", 2.0), (1, 256, "min_prefix", 0.5), (200, 12, "topk", 7.0),
                                        (130, 40, "paper", 0.95), (130, 40, "lte", 0.97), (130, 40, "lte", 1.0)])
def test_union_sizes(pp, E, T, rule, p):
    """Down from one expert (fewer pairs than CTAs) up to all 256."""
    layer_parity(pp, "llama3_8b_batched", T, p, rule, d=1024, E=E)


@pytest.mark.parametrize("d,E,T", [(64, 40, 6), (72, 5, 130), (200, 33, 17), (1000, 40, 100), (4104, 20, 48), (8192, 12, 33)])
@pytest.mark.parametrize("name", ["llama3_8b_batched", "gpt2m_gelu_bf16"])
def test_union_widths(pp, name, d, E, T):
    layer_parity(pp, name, T, 0.8, d=d, E=E)


def _device_layer(name, T, d, E):
    w, L = layer_inputs(name, T, d=d, E=E)
    return w, L, [None if a is None else dev(a) for a in (L.x, L.Wr, L.Wg, L.Wu, L.Wd)]


def test_union_repeated_calls_one_workspace(pp):
    """Alternating token counts (so alternating ring shapes) on one workspace,
    back to back: every call gives the bits of the first one."""
    import torch
    Ts, p = (160, 32, 5, 64), f32(0.75)
    w, L, (x, Wr, Wg, Wu, Wd) = _device_layer("llama3_8b_batched", max(Ts), 1536, 140)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, max(Ts))
    ref, got = {}, []
    for rep in range(25):
        for T in Ts:
            y = torch.empty_like(x[:T])
            pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, None, y, ws)
            if rep == 0:
                ref[T] = y
            got.append((T, y))
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    for T, y in got:
        assert torch.equal(y.view(torch.int16), ref[T].view(torch.int16)), T


def test_union_selection_output_does_not_change_y(pp):
    """pp_layer with and without sel_out, and pp_sparse_ffn on its selection."""
    import torch
    T, p = 21, f32(0.6)
    w, L, (x, Wr, Wg, Wu, Wd) = _device_layer("llama3_8b_batched", T, 512, 70)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    ys = [torch.empty_like(x) for _ in range(3)]
    sel = pp.Selection.empty(T, w.n_experts, "cuda")
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, None, ys[0], ws)
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, sel, ys[1], ws)
    pp.pp_sparse_ffn(desc, x, T, Wg, Wu, Wd, sel, ys[2], ws)
    torch.cuda.synchronize()
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])


def test_union_non_finite_weight_stays_with_its_expert(pp):
    """W_down of one expert holds an infinity: tokens that did not select the
    expert are not affected by it."""
    import torch
    T, p = 24, f32(0.5)
    w, L, (x, Wr, Wg, Wu, Wd) = _device_layer("llama3_8b_batched", T, 384, 48)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    sel = pp.Selection.empty(T, w.n_experts, "cuda")
    y0, y1 = torch.empty_like(x), torch.empty_like(x)
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, sel, y0, ws)
    counts, ids = to_host(sel.counts), to_host(sel.ids)
    uses = np.array([[e in ids[t, :counts[t]] for e in range(w.n_experts)] for t in range(T)])
    e = int(np.argmax(uses.any(0) & ~uses.all(0)))
    Wd = Wd.clone()
    Wd[:, 64 * e + 5] = float("inf")
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, p, None, y1, ws)
    torch.cuda.synchronize()
    a, b = to_host(y0), to_host(y1)
    assert not np.isfinite(b[uses[:, e]]).any()
    assert np.isfinite(b[~uses[:, e]]).all()
    assert rel_err_per_token(b[~uses[:, e]], a[~uses[:, e]]).max() <= Y_TOL["bf16"]


@pytest.mark.parametrize("T,rule,p", [(2, "min_prefix", 1.0), (3, "min_prefix", 0.9), (4, "paper", 0.9), (4, "topk", 9.0),
                                      (3, "lte", 0.95)])
def test_union_small_batches_of_wide_layers(pp, T, rule, p):
    """2 to 4 tokens that the union kernel runs instead of the fused decode
    kernel: parity, and no less exact than the fused kernel (pp_layer_noalloc
    always takes it).  Both sides' error is the rounding of y to bf16; 3 % is
    four standard deviations of the ratio of two such errors over the 8192 or
    more elements."""
    import torch
    layer_parity(pp, "llama3_8b_batched", T, p, rule)
    w, L, (x, Wr, Wg, Wu, Wd) = _device_layer("llama3_8b_batched", T, 4096, 224)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act, "sigmoid", rule)
    ws = pp.alloc_workspace(desc, T)
    sels = [pp.Selection.empty(T, w.n_experts, "cuda") for _ in range(2)]
    ys = [torch.empty_like(x) for _ in range(2)]
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(p), sels[0], ys[0], ws)
    pp.pp_layer_noalloc(desc, x, T, Wr, Wg, Wu, Wd, f32(p), sels[1], ys[1])
    torch.cuda.synchronize()
    counts, ids = to_host(sels[0].counts), to_host(sels[0].ids)
    assert np.array_equal(counts, to_host(sels[1].counts)) and np.array_equal(ids, to_host(sels[1].ids))
    ref = oracle.sparse_ffn(L.x, L.Wg, L.Wu, L.Wd, counts, ids, oracle.logits(L.x, L.Wr), w.n_experts, w.act, "sigmoid")
    e = [np.linalg.norm(to_host(y).astype(np.float64) - ref) / np.linalg.norm(ref) for y in ys]
    assert e[0] <= 1.03 * e[1], e
