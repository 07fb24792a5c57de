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
