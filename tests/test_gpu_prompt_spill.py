"""Prompts whose pairs exceed the row buffer (more than 64 experts a token on
average): the fp32 accumulator that takes the rest."""
import numpy as np
import pytest

from parity import Y_TOL, f32, layer_inputs, rel_err_per_token, to_host
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu


def _layer(name, T, d, E):
    w, L = layer_inputs(name, T, d=d, E=E)
    return w, [None if a is None else dev(a) for a in (L.x, L.Wr, L.Wg, L.Wu, L.Wd)]


@pytest.mark.parametrize("lengths", [(1500, 300, 256, 300), (256, 1100, 700, 300, 1100)])
def test_spilling_prompts_of_several_lengths_share_a_workspace(pp, lengths):
    """Every expert for every token, lengths in turn on one workspace: each call
    equals the one on a workspace of its own.  (The fp32 additions into the
    accumulator come in any order, so y may differ in its last bit: half of the
    parity bound is far above that and far below what a leftover adds.)"""
    import torch
    w, (x, Wr, Wg, Wu, Wd) = _layer("llama3_8b_batched", max(lengths), 264, 100)
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    shared = pp.alloc_workspace(desc, max(lengths))
    ys, alone = [], []
    for T in lengths:
        for ws, out in ((shared, ys), (pp.alloc_workspace(desc, T), alone)):
            out.append(torch.empty_like(x[:T]))
            pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(1.0), None, out[-1], ws)
            torch.cuda.synchronize()
            assert pp.pp_get_device_status(ws) == pp.PP_OK
    for T, y, ref in zip(lengths, ys, alone):
        assert rel_err_per_token(to_host(y), to_host(ref)).max() <= Y_TOL["bf16"] / 2, T


@pytest.mark.parametrize("T", [300, 1100])
def test_spilling_does_not_depend_on_the_order_of_the_lists(pp, T):
    """One expert's rows straddle the end of the row buffer (64 rows a token).
    Its tokens stand in its list in any order, but all of its pairs are summed
    in fp32, and as each token has one such pair at most nothing else is free:
    repeated calls give the same bits."""
    import torch
    E, skip = 66, 100
    w, (x, Wr, Wg, Wu, Wd) = _layer("llama3_8b_batched", T, 264, E)
    ids = np.tile(np.arange(E, dtype=np.int32), (T, 1))
    ids[:skip, 0] = 64  # `skip` tokens leave out expert 0: 64 T - skip pairs come before expert 64's T
    ids[:skip, 64] = -1
    ids[:, 65] = -1
    counts = np.where(np.arange(T) < skip, 64, 65).astype(np.int32)
    gates = np.where(ids >= 0, np.float32(0.7), np.float32(0))
    desc = pp.make_desc(w.d_model, E, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    sel = pp.Selection(dev(ids), dev(counts), dev(gates))
    ys = [torch.empty_like(x) for _ in range(20)]
    for y in ys:
        pp.pp_sparse_ffn(desc, x, T, Wg, Wu, Wd, sel, y, ws)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    assert all(torch.equal(y, ys[0]) for y in ys)
