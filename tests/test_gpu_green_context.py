"""A stream that owns fewer SMs than the device has (a green context): calls of
5 to 256 tokens, whose kernel wants all its CTAs resident at once, run there on
a smaller grid; the same workspace serves both grids in turn (the grid barrier's
counter and every ring go on where the previous call left them)."""
import ctypes

import pytest

from parity import Y_TOL, f32, layer_inputs, rel_err_per_token, to_host
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu
SMS = 16


class GreenStream:
    """A non-blocking stream on `sms` SMs of device 0."""

    def __init__(self, sms):
        cu = self.cu = ctypes.CDLL("libcuda.so.1")
        d, whole, part, rest = ctypes.c_int(), *(ctypes.create_string_buffer(512) for _ in range(3))
        desc, n = ctypes.c_void_p(), ctypes.c_uint(1)
        self.ctx, self.handle = ctypes.c_void_p(), ctypes.c_void_p()
        steps = [lambda: cu.cuDeviceGet(ctypes.byref(d), 0),
                 lambda: cu.cuDeviceGetDevResource(d, whole, 1),  # the device's SMs
                 lambda: cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), whole, rest, 0, sms),
                 lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
                 lambda: cu.cuGreenCtxCreate(ctypes.byref(self.ctx), desc, d, 1),
                 lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(self.handle), self.ctx, 1, 0)]
        for i, step in enumerate(steps):
            try:
                rc = step()
            except AttributeError:
                rc = -1
            if rc != 0:
                pytest.skip("no green context here: step %d returned %d" % (i, rc))

    def close(self):
        self.cu.cuStreamDestroy_v2(self.handle)
        self.cu.cuGreenCtxDestroy(self.ctx)


@pytest.mark.parametrize("name,d,E", [("llama3_8b_batched", 1536, 140), ("gpt2m_gelu_bf16", 1024, 64)])
def test_fewer_sms_than_the_device(pp, name, d, E):
    import torch
    Ts = (64, 5, 200)
    w, L = layer_inputs(name, max(Ts), d=d, E=E)
    x, Wr, Wg, Wu, Wd = (None if a is None else dev(a) for a in (L.x, L.Wr, L.Wg, L.Wu, L.Wd))
    desc = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
    ws = pp.alloc_workspace(desc, max(Ts))
    torch.cuda.synchronize()
    green = GreenStream(SMS)
    try:
        for T in Ts * 2:
            outs = []
            for stream in (None, green.handle.value):
                sel, y = pp.Selection.empty(T, E, "cuda"), torch.zeros_like(x[:T])
                torch.cuda.synchronize()
                pp.pp_layer(desc, x, T, Wr, Wg, Wu, Wd, f32(0.8), sel, y, ws, stream=stream)
                torch.cuda.synchronize()
                assert pp.pp_get_device_status(ws) == pp.PP_OK
                outs.append((sel, to_host(y)))
            (s0, y0), (s1, y1) = outs
            assert torch.equal(s0.ids, s1.ids) and torch.equal(s0.counts, s1.counts)
            assert torch.equal(s0.logits.view(torch.int32), s1.logits.view(torch.int32))
            assert rel_err_per_token(y1, y0).max() <= Y_TOL["bf16"] / 2  # other partial tiles, so other roundings
    finally:
        torch.cuda.synchronize()
        green.close()
