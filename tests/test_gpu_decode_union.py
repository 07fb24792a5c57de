"""Calls of 2 to 4 bf16 tokens of wide layers: the fused decode kernel makes the
selection and, where the tokens selected many experts together, goes on with the
union kernel's phases.  The selection is that of pp_route and pp_layer_noalloc
to the last bit, however many experts it holds (as in longer calls); a call with
few experts is the fused kernel's.  Tolerances are those of the other parity
tests."""
import pytest

from parity import f32, layer_inputs, to_host
from test_gpu_chained import chained
from test_gpu_parity import dev, layer_parity

pytestmark = pytest.mark.gpu


def _setup(pp, T, rule, seed=0, d=4096, E=224, spread=1.0):
    import torch
    w, L = layer_inputs("llama3_8b_batched", T, seed, 0, d, E)
    x, Wr, Wg, Wu, Wd = (dev(a) for a in (L.x, L.Wr, L.Wg, L.Wu, L.Wd))
    if spread != 1.0:
        Wr = (Wr.float() * spread).to(torch.bfloat16)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act, "sigmoid", rule)
    return desc, pp.alloc_workspace(desc, T), x, Wr, Wg, Wu, Wd, w.n_experts


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("T,rule,p", [(2, "min_prefix", 1.0), (2, "min_prefix", 0.97), (3, "paper", 0.9), (4, "min_prefix", 0.7),
                                      (4, "topk", 9.0), (4, "lte", 0.95), (3, "topk", 1.0)])
def test_selection_is_that_of_pp_route(pp, T, rule, p, seed):
    import torch
    desc, ws, x, Wr, Wg, Wu, Wd, E = _setup(pp, T, rule, seed)
    sels = [pp.Selection.empty(T, E, "cuda") for _ in range(3)]
    y = torch.empty_like(x)
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(p), sels[0], y, ws)
    pp.pp_route(desc, x, T, Wr, f32(p), sels[1], ws)
    pp.pp_layer_noalloc(desc, x, T, Wr, Wg, Wu, Wd, f32(p), sels[2], y)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    for s in sels[1:]:
        assert torch.equal(s.counts, sels[0].counts) and torch.equal(s.ids, sels[0].ids)
        assert torch.equal(s.logits.view(torch.int32), sels[0].logits.view(torch.int32))
        assert torch.equal(s.gates.view(torch.int32), sels[0].gates.view(torch.int32))


@pytest.mark.parametrize("T", [5, 40, 200, 300])
@pytest.mark.parametrize("d,E", [(4096, 224), (1000, 33)])
def test_batched_selection_is_that_of_pp_route(pp, T, d, E):
    import torch
    desc, ws, x, Wr, Wg, Wu, Wd, E = _setup(pp, T, "min_prefix", d=d, E=E)
    a, b = (pp.Selection.empty(T, E, "cuda") for _ in range(2))
    y = torch.empty_like(x)
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(0.8), a, y, ws)
    pp.pp_route(desc, x, T, Wr, f32(0.8), b, ws)
    torch.cuda.synchronize()
    assert torch.equal(a.counts, b.counts) and torch.equal(a.ids, b.ids)
    assert torch.equal(a.logits.view(torch.int32), b.logits.view(torch.int32))


@pytest.mark.parametrize("T,rule,p,spread", [(4, "min_prefix", 0.7, 20.0), (3, "min_prefix", 0.97, 20.0), (2, "min_prefix", 0.99, 20.0),
                                             (4, "lte", 0.9999, 1.0), (4, "lte", 1.0, 1.0), (4, "topk", 2.0, 1.0)])
def test_few_experts_stay_with_the_fused_kernel(pp, T, rule, p, spread):
    """One or two experts a token, whatever the rule's parameter promises: the
    result is the fused kernel's (pp_layer_noalloc), bit for bit."""
    import torch
    desc, ws, x, Wr, Wg, Wu, Wd, E = _setup(pp, T, rule, spread=spread)
    ys = [torch.empty_like(x) for _ in range(2)]
    sel = pp.Selection.empty(T, E, "cuda")
    pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(p), sel, ys[0], ws)
    pp.pp_layer_noalloc(desc, x, T, Wr, Wg, Wu, Wd, f32(p), None, ys[1])
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    assert to_host(sel.counts).max() <= 3
    assert torch.equal(ys[0].view(torch.int16), ys[1].view(torch.int16))


@pytest.mark.parametrize("name,T,d,E,p", [("llama3_8b_batched", 2, 5120, 216, 1.0), ("llama3_8b_batched", 3, 8192, 256, 0.95),
                                          ("llama3_8b_batched", 4, 4104, 200, 0.9), ("gpt2m_gelu_bf16", 4, 4096, 256, 0.95),
                                          ("gpt2m_gelu_bf16", 2, 6000, 129, 1.0), ("llama3_8b_batched", 4, 2056, 256, 1.0)])
def test_many_experts(pp, name, T, d, E, p):
    layer_parity(pp, name, T, p, d=d, E=E)


@pytest.mark.parametrize("T,p,d,E", [(2, 1.0, 4096, 224), (4, 0.9, 4096, 224), (3, 0.95, 5120, 216), (4, 0.9, 8192, 256)])
def test_chained(pp, T, p, d, E):
    chained(pp, "llama3_8b_batched", T, p, d=d, E=E)


def test_few_and_many_experts_in_turn_on_one_workspace(pp):
    """1 to 6 tokens, few and many experts: tagged words, launch counts and the
    barrier's counter in one workspace; every call repeats its first bits."""
    import torch
    desc, ws, x, Wr, Wg, Wu, Wd, E = _setup(pp, 6, "min_prefix")
    eps, first = 1e-6, {}
    for _ in range(6):
        for T, p, chain in ((1, 0.7, False), (4, 1.0, False), (4, 0.1, False), (6, 0.8, False), (3, 0.95, True), (2, 0.3, True),
                            (1, 1.0, True), (2, 1.0, False), (4, 0.9, True)):
            y, xo = torch.empty_like(x[:T]), torch.empty_like(x[:T])
            if chain:
                pp.pp_layer_chained(desc, x[:T], None, None, eps, T, Wr, Wg, Wu, Wd, f32(p), None, xo, y, ws)
            else:
                pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(p), None, y, ws)
            first.setdefault((T, p, chain), []).append(y)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    for key, ys in first.items():
        assert all(torch.equal(y.view(torch.int16), ys[0].view(torch.int16)) for y in ys), key
