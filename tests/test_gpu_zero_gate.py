"""A selected expert whose gate weight is zero: y = 0 * FFN_e(x), which is NaN
where the activation is not finite and nothing otherwise (bf16, 5 tokens and
more: every batched path alike).  Tokens that did not select it are untouched."""
import numpy as np
import pytest

from parity import Y_TOL, layer_inputs, rel_err_per_token, to_host
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["llama3_8b_batched", "gpt2m_gelu_bf16"])
@pytest.mark.parametrize("T", [5, 8, 64, 300])
def test_zero_gate_of_an_infinite_activation(pp, T, name):
    import torch
    E, zero = 24, 7
    w, L = layer_inputs(name, T, d=256, E=E)
    x, Wg, Wu, Wd = (None if a is None else dev(a) for a in (L.x, L.Wg, L.Wu, L.Wd))
    x = x.abs() + 1  # every product of a row of one sign overflows alike
    desc = pp.make_desc(w.d_model, E, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, T)
    ids = np.full((T, E), -1, np.int32)
    ids[:, 0], ids[:, 1] = np.arange(T) % 5, zero
    has = np.arange(T) % 3 == 0
    counts = np.where(has, 2, 1).astype(np.int32)
    gates = np.zeros((T, E), np.float32)
    gates[:, 0] = 0.7
    sel = pp.Selection(dev(ids), dev(counts), dev(gates))
    plain, inf = torch.empty_like(x), torch.empty_like(x)
    pp.pp_sparse_ffn(desc, x, T, Wg, Wu, Wd, sel, plain, ws)
    Wu = Wu.clone()
    Wu[64 * zero:64 * zero + 64] = 3.0e38
    if Wg is not None:
        Wg = Wg.clone()
        Wg[64 * zero:64 * zero + 64] = 1.0
    pp.pp_sparse_ffn(desc, x, T, Wg, Wu, Wd, sel, inf, ws)
    torch.cuda.synchronize()
    assert pp.pp_get_device_status(ws) == pp.PP_OK
    a, b = to_host(plain), to_host(inf)
    assert np.isfinite(a).all()
    assert np.isnan(b[has]).all()
    assert rel_err_per_token(b[~has], a[~has]).max() <= Y_TOL["bf16"]
