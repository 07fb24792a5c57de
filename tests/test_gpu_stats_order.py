"""pp_router_stats, bit for bit: the order of its fp32 sums is part of the
result.  Eight consecutive tokens one after the other (per lane for the entropy
and gate terms, whose 32 lanes are then added by a butterfly), the eight groups
of a 64-token block one after the other, then the fixed trees over the blocks.
The terms themselves are made known: a token's logits are either equal or too
small to count, so that every probability is 1 / k, and the values of the
device's logarithm and sigmoid come from calls with one token."""
import numpy as np
import pytest

from parity import to_host
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu
F = np.float32
TOKENS = [1, 7, 8, 9, 63, 64, 65, 700, 2048, 2051]
LOW = F(-200.0)  # exp(LOW - 0) is 0 in fp32
EPS = 1e-9


def _stats(pp, g, E):
    import torch
    desc = pp.make_desc(64, E, "bf16", "swiglu")
    ws = pp.alloc_workspace(desc, len(g))
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    pp.pp_router_stats(desc, dev(np.ascontiguousarray(g, F)), len(g), EPS, out, ws)
    torch.cuda.synchronize()
    return to_host(out)


def _butterfly(v):
    for o in (16, 8, 4, 2, 1):
        v = (v + v[np.arange(32) ^ o]).astype(F)
    return v[0]


def _in_turn(terms):
    """fp32 sum over axis 0, one after the other, starting from zero."""
    a = np.zeros(terms.shape[1:], F)
    for t in terms:
        a = (a + t).astype(F)
    return a


def _blocks(terms):
    """[T, ...] -> [blocks, groups, ...]: groups of eight tokens added in turn."""
    T, n = len(terms), (len(terms) + 63) // 64
    return np.stack([np.stack([_in_turn(terms[min(T, b * 64 + w * 8):min(T, b * 64 + w * 8 + 8)]) for w in range(8)])
                     for b in range(n)])


def _tree1024(v):
    v = np.concatenate([v, np.zeros(1024 - len(v), F)]).reshape(32, 32)
    return _butterfly(np.array([_butterfly(w) for w in v], F))


def _scalar_total(terms):
    """[T, 32] per-lane terms -> the total over all blocks."""
    parts = [_in_turn(np.array([_butterfly(lanes) for lanes in groups], F)) for groups in _blocks(terms)]
    return _tree1024(np.array(parts, F))


@pytest.mark.parametrize("T", TOKENS)
def test_gate_term_order(pp, T):
    vals = np.array([-3.1, -0.7, 0.0, 0.3, 1.9, 2.7, 11.0], F)
    sig = np.array([_stats(pp, np.array([[v]]), 1)[2] for v in vals]).astype(F)
    pick = np.random.default_rng(T).integers(0, len(vals), T)
    terms = np.zeros((T, 32), F)
    terms[:, 0] = sig[pick]
    assert _stats(pp, vals[pick][:, None], 1)[2] == np.float64(_scalar_total(terms)) / T


@pytest.mark.parametrize("T", TOKENS)
def test_entropy_term_order(pp, T):
    E = 32
    rng = np.random.default_rng(100 + T)
    ks = 1 << rng.integers(0, 6, T)
    on = (np.arange(E)[None, :] - rng.integers(0, E, T)[:, None]) % E < ks[:, None]
    term = {}
    for k in (1, 2, 4, 8, 16, 32):  # k equal terms, k a power of two: their sum is exact
        term[k] = F(-_stats(pp, np.where(np.arange(E) < k, F(0), LOW)[None, :], E)[0] / k)
    terms = np.where(on, np.array([term[k] for k in ks], F)[:, None], F(0)).astype(F)
    assert _stats(pp, np.where(on, F(0), LOW), E)[0] == -np.float64(_scalar_total(terms)) / T


@pytest.mark.parametrize("T", TOKENS)
@pytest.mark.parametrize("E", [33, 200, 256])
def test_column_order(pp, T, E):
    rng = np.random.default_rng(200 + T + E)
    ks = rng.choice([3, 5, 7, 11, 13, 29, 31], T)
    on = np.argsort(rng.random((T, E)), 1).argsort(1) < ks[:, None]
    p = np.where(on, (F(1) / ks.astype(F)).astype(F)[:, None], F(0)).astype(F)
    part = np.stack([_in_turn(groups) for groups in _blocks(p)])
    n, col = len(part), []
    for q in range(4):  # the quarters of the parts, eight at a time pairwise
        c, b, b1 = np.zeros(E, F), q * n // 4, (q + 1) * n // 4
        while b + 8 <= b1:
            v = part[b:b + 8]
            c = (c + (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])))).astype(F)
            b += 8
        for i in range(b, b1):
            c = (c + part[i]).astype(F)
        col.append(c)
    f = (((col[0] + col[1]) + (col[2] + col[3])) / F(T)).astype(F)
    assert _stats(pp, np.where(on, F(0), LOW), E)[1] == np.float64(E) * np.float64(_tree1024((f * f).astype(F)))
