"""pp_sparsity_stats and pp_router_stats at the edges of their blocks: token
counts around 2 (a warp), 64 (a block of the router statistics) and 256 (a block
of the histogram), one expert to 256, counts outside [0, E]."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import dev
from parity import to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 2, 3, 63, 64, 65, 255, 257, 2049])
@pytest.mark.parametrize("E", [1, 33, 256])
def test_router_stats_edges(pp, T, E):
    """Against fp64: fp32 softmax and sums of at most 2 + 32 + T / 64 additions
    in a row, so 2e-5 of the largest term is over 100 times their rounding."""
    import torch
    g = (np.random.default_rng(T * 1000 + E).standard_normal((T, E)) * 3).astype(np.float32)
    desc = pp.make_desc(64, E, "bf16", "swiglu")
    ws = pp.alloc_workspace(desc, T)
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    pp.pp_router_stats(desc, dev(g), T, 1e-9, out, ws)
    torch.cuda.synchronize()
    x = g.astype(np.float64)
    p = np.exp(x - x.max(1, keepdims=True))
    p /= p.sum(1, keepdims=True)
    ref = [-(p * np.log(p + 1e-9)).sum(1).mean(), E * (p.mean(0) ** 2).sum(), (1 / (1 + np.exp(-x))).mean()]
    np.testing.assert_allclose(to_host(out), ref, rtol=2e-5, atol=2e-5)


@pytest.mark.parametrize("T", [1, 31, 256, 257, 40000])
@pytest.mark.parametrize("E", [1, 200, 256])
def test_sparsity_stats_edges(pp, T, E):
    """Exact, accumulated over two calls; counts outside [0, E] are clamped."""
    import torch
    c = np.random.default_rng(T + E).integers(-1, E + 2, T).astype(np.int32)
    acc = torch.zeros(E + 2, dtype=torch.int64, device="cuda")
    for _ in range(2):
        pp.pp_sparsity_stats(dev(c), T, E, acc)
    torch.cuda.synchronize()
    k = np.clip(c, 0, E)
    ref = 2 * np.concatenate([[k.sum()], np.bincount(k, minlength=E + 1)])
    assert np.array_equal(to_host(acc), ref)
