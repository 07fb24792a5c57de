"""A workspace for up to T tokens serves every shorter call: its size never
falls as T grows (the router's K splits, and with them the rows of its partial
sums, fall as T crosses a multiple of 128)."""
import numpy as np
import pytest

from paper_2605_28283_gb300 import binding as pp
from paper_2605_28283_gb300 import workloads as wl

SHAPES = [(w.d_model, w.n_experts, w.dtype, w.act) for w in wl.WORKLOADS.values()]
SHAPES += [(8192, 256, "bf16", "swiglu"), (200, 3, "bf16", "gelu_tanh"), (64, 1, "bf16", "swiglu"), (8192, 1, "bf16", "swiglu"),
           (4096, 64, "f32", "relu")]


@pytest.mark.parametrize("d,E,dtype,act", SHAPES)
def test_workspace_size_never_falls(d, E, dtype, act):
    desc = pp.make_desc(d, E, dtype, act)
    T = np.concatenate([np.arange(3000), np.arange(3000, 40000, 127)])
    size = np.array([pp.pp_workspace_size(desc, int(t)) for t in T])
    assert size[0] > 0 and np.all(np.diff(size) >= 0), T[1:][np.diff(size) < 0]


@pytest.mark.parametrize("T", [5, 64, 256])
def test_batched_calls_hold_no_prompt_buffers(T):
    """Up to 256 tokens: the decode kernel's words, the router's partial sums, the
    selection tables, the activations and the partial down-projection tiles;
    nothing of the size of a row or a list entry per (token, expert)."""
    for w in wl.WORKLOADS.values():
        if w.dtype != "bf16":
            continue
        d, E = w.d_model, w.n_experts
        base = 1280 + T * (12 * E + 4) + 64 * E + E * 8 * 64 * 8 + (T + 63) // 64 * (E + 2) * 8
        part = max(T, min(T * min((d + 63) // 64 // 4, 64), 152 * 128)) * E * 4
        tables = T * (32 + 4 * E) + max(T * E + 128, 15 * E) * 128
        tiles = (3 * 152 + (d + 127) // 128) * 128 * max(T, 16) * 4
        desc = pp.make_desc(d, E, w.dtype, w.act)
        assert pp.pp_workspace_size(desc, T) <= base + part + tables + tiles + 16 * 256
