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
