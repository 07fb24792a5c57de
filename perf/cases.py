"""The work a user of this library has it do, as measurable cases.

A case is one pass of a serving or preprocessing program over the library's
public entry points (``paper_2605_28283_gb300.binding``).  Shapes, value
distributions and rule parameters come from ``workloads.WORKLOADS`` and from
the shapes of the parity tests.

Kinds of case:

``layer``    ``layers`` back-to-back layers of a model on ``tokens`` tokens
             each.  ``entry`` is "layer" (pp_layer) or "chained"
             (pp_layer_chained).  With ``graph`` the pass is one replay of a
             CUDA graph captured when the program sets up, which is how a
             serving loop issues a step of many small launches; without it
             every call is issued by itself.
``route``    routing diagnostics of a batch: pp_route, then the FFN-sparsity
             accumulators (pp_sparsity_stats) and the router statistics
             (pp_router_stats) of what it returned.
``permute``  repacking one layer's weights into experts (pp_moefy_permute).
"""
import math

import numpy as np
import torch

from paper_2605_28283_gb300 import binding as pp
from paper_2605_28283_gb300 import workloads as wl

EPS_NORM = 1e-5    # RMSNorm epsilon of the chained step
EPS_STATS = 1e-9   # epsilon of the entropy term


def _layer(name, model, tokens, p, layers, graph, rule="min_prefix", gate="sigmoid", entry="layer", d=0, experts=0):
    w = wl.WORKLOADS[model]
    return {"name": name, "kind": "layer", "model": model, "d": d or w.d_model, "experts": experts or w.n_experts,
            "tokens": tokens, "p": p, "rule": rule, "gate": gate, "layers": layers, "graph": graph, "entry": entry}


def listed():
    return [
        # one token through all layers of a 7B model: the decode step of an interactive session
        _layer("decode_7b_b1", "llama2_7b_decode", 1, 0.7, 32, True),
        # four sessions decoded together, with the residual and norm between the layers as a model has them;
        # the rule of the paper's equation, at a larger mass
        _layer("decode_8b_b4_chained", "llama3_8b_batched", 4, 0.9, 8, True, rule="paper", entry="chained"),
        # the paper's own decode model, a few sequences at once (beam of four): small layers, latency
        _layer("decode_gpt2m_b4", "gpt2m_gelu_bf16", 4, 0.7, 24, True),
        # the same model serving sixteen sequences
        _layer("batch_gpt2m_b16", "gpt2m_gelu_bf16", 16, 0.7, 24, True),
        # a lightly loaded 8B server
        _layer("batch_8b_b8", "llama3_8b_batched", 8, 0.7, 8, True),
        # a fully loaded 8B server
        _layer("batch_8b_b64", "llama3_8b_batched", 64, 0.7, 8, True),
        # a short prompt of odd length, fixed expert budget, experts summed unweighted
        _layer("prompt_7b_t333_topk", "llama2_7b_decode", 333, 6.0, 1, False, rule="topk", gate="none"),
        # the prompt of one long sequence
        _layer("prefill_13b_t2048", "llama2_13b_prefill", 2048, 0.7, 1, False),
        # a prefill batch of four long sequences: the largest call
        _layer("prefill_13b_t8192", "llama2_13b_prefill", 8192, 0.7, 1, False),
        # the tiny fp32 model, one eager call: the smallest layers, 32-bit throughout
        _layer("tiny_f32_t64", "tiny_relu_f32", 64, 0.9, 1, False),
        # how sparse a validation batch routes (counts, entropy, balance)
        {"name": "route_stats_13b_t2048", "kind": "route", "model": "llama2_13b_prefill", "d": 5120, "experts": 216,
         "tokens": 2048, "p": 0.7, "rule": "min_prefix", "gate": "sigmoid"},
        # MoEfication of one 7B layer
        {"name": "permute_7b", "kind": "permute", "model": "llama2_7b_decode", "d": 4096, "experts": 172},
    ]


def _logint(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _rule(rng, experts, most=0.95):
    """(rule, parameter, gate): the cumulative-mass rule mostly, the others as the paper compares with them."""
    u = rng.random()
    if u < 0.7:
        return "min_prefix", round(rng.uniform(0.3, most), 3), "sigmoid"
    if u < 0.8:
        return "paper", round(rng.uniform(0.3, most), 3), "sigmoid"
    if u < 0.9:
        return "topk", float(rng.randint(1, max(1, min(16, experts // 4)))), rng.choice(["sigmoid", "none"])
    return "lte", round(rng.uniform(0.9, 0.995), 3), "none"


def draw(rng):
    kind = rng.choices(["decode", "batch", "prefill", "f32", "route", "permute"], [28, 30, 20, 10, 7, 5])[0]
    bf16 = ["gpt2m_gelu_bf16", "llama2_7b_decode", "llama3_8b_batched", "llama2_13b_prefill"]
    if kind == "f32":
        d, experts = rng.choice([(256, 16), (256, 16), (64, 5), (512, 24), (1024, 33)])
        rule, p, gate = _rule(rng, experts)
        return {"kind": "layer", "model": "tiny_relu_f32", "d": d, "experts": experts, "tokens": _logint(rng, 1, 512),
                "p": p, "rule": rule, "gate": gate, "layers": rng.choice([1, 1, 4]), "graph": rng.random() < 0.5,
                "entry": "layer"}
    w = wl.WORKLOADS[rng.choice(bf16)]
    d, experts = w.d_model, w.n_experts
    if rng.random() < 0.25:  # widths no named model has, down to the edges of what is supported
        d, experts = 8 * _logint(rng, 25, 1024), rng.randint(3, 256)
    if kind == "permute":
        return {"kind": "permute", "model": w.name, "d": d, "experts": experts}
    rule, p, gate = _rule(rng, experts)
    if kind == "route":
        return {"kind": "route", "model": w.name, "d": d, "experts": experts, "tokens": _logint(rng, 1, 8192), "p": p,
                "rule": rule, "gate": gate}
    case = {"kind": "layer", "model": w.name, "d": d, "experts": experts, "p": p, "rule": rule, "gate": gate,
            "entry": "layer"}
    if kind == "decode":
        dense = rng.random() < 0.1  # every expert: the dense layer the sparse one is compared with
        if dense:
            case.update(rule="min_prefix", p=1.0)
        return dict(case, tokens=rng.randint(1, 4), layers=rng.randint(1, 4 if dense else 16), graph=True,
                    entry=rng.choice(["layer", "layer", "chained"]))
    if kind == "batch":
        return dict(case, tokens=_logint(rng, 5, 128), layers=rng.randint(1, 4), graph=True)
    if rule in ("min_prefix", "paper"):
        case["p"] = round(rng.uniform(0.3, 0.8), 3)
    if rule == "topk":
        case["p"] = min(p, 8.0)
    if rule == "lte":
        case["p"] = max(p, 0.98)
    most = 8192 if case["rule"] in ("min_prefix", "paper") and case["p"] <= 0.65 else 2048
    return dict(case, tokens=_logint(rng, 129, most), layers=1, graph=False)


# ---------------------------------------------------------------- inputs
def _workload(case):
    return wl.scaled(wl.WORKLOADS[case["model"]], case["d"], case["experts"])


def _tensors(case, seed):
    """One dict per layer: Wr, Wg (or None), Wu, Wd and the layer's x [tokens, d]."""
    w = _workload(case)
    out = []
    for layer in range(case.get("layers", 1)):
        t = wl.device_layer(w, case.get("tokens", 1), seed, layer, "cuda")
        t["x"] = t["x"][0].contiguous()
        if case.get("entry") == "chained":
            gen = torch.Generator(device="cuda")
            gen.manual_seed((seed * 7919 + layer) & 0x7FFFFFFF)
            rand = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.float32)
            t["y_prev"] = (0.5 * rand(case["tokens"], w.d_model)).to(t["x"].dtype)
            t["gamma"] = (1.0 + 0.1 * rand(w.d_model)).to(t["x"].dtype)
        out.append(t)
    return out


def _perm(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed & 0x7FFFFFFF)
    return torch.randperm(64 * case["experts"], generator=gen, device="cuda").to(torch.int32)


def prepare(case, seed):
    w = _workload(case)
    state = {"case": case, "layers": _tensors(case, seed)}
    if case["kind"] == "permute":
        state["desc"] = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act)
        t = state["layers"][0]
        state["perm"] = _perm(case, seed)
        state["out"] = [None if v is None else torch.empty_like(v) for v in (t["Wg"], t["Wu"], t["Wd"])]
        state["ws"] = pp.alloc_workspace(state["desc"], 0)
        return state
    state["desc"] = pp.make_desc(w.d_model, w.n_experts, w.dtype, w.act, case["gate"], case["rule"])
    state["ws"] = pp.alloc_workspace(state["desc"], case["tokens"])
    if case["kind"] == "route":
        state["sel"] = pp.Selection.empty(case["tokens"], w.n_experts, "cuda")
        state["acc"] = torch.zeros(w.n_experts + 2, dtype=torch.int64, device="cuda")
        state["stats"] = torch.zeros(3, dtype=torch.float64, device="cuda")
        return state
    first = state["layers"][0]["x"]
    state["y"] = torch.empty((case["layers"], *first.shape), dtype=first.dtype, device="cuda")
    state["x"] = torch.empty_like(state["y"]) if case["entry"] == "chained" else None
    if case["graph"]:
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            _layers(state)  # load the kernels before the capture
            stream.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"], stream=stream):
                _layers(state)
        torch.cuda.current_stream().wait_stream(stream)
    return state


def _layers(state):
    case = state["case"]
    for i, t in enumerate(state["layers"]):
        if case["entry"] == "chained":
            pp.pp_layer_chained(state["desc"], t["x"], t["y_prev"], t["gamma"], EPS_NORM, case["tokens"], t["Wr"],
                                t["Wg"], t["Wu"], t["Wd"], case["p"], None, state["x"][i], state["y"][i], state["ws"])
        else:
            pp.pp_layer(state["desc"], t["x"], case["tokens"], t["Wr"], t["Wg"], t["Wu"], t["Wd"], case["p"], None,
                        state["y"][i], state["ws"])


def run(state):
    case = state["case"]
    t = state["layers"][0]
    if case["kind"] == "permute":
        pp.pp_moefy_permute(state["desc"], state["perm"], t["Wg"], t["Wu"], t["Wd"], *state["out"], state["ws"])
        return state["out"]
    if case["kind"] == "route":
        sel = state["sel"]
        state["acc"].zero_()
        pp.pp_route(state["desc"], t["x"], case["tokens"], t["Wr"], case["p"], sel, state["ws"])
        pp.pp_sparsity_stats(sel.counts, case["tokens"], case["experts"], state["acc"])
        pp.pp_router_stats(state["desc"], sel.logits, case["tokens"], EPS_STATS, state["stats"], state["ws"])
        return {"ids": sel.ids, "counts": sel.counts, "gates": sel.gates, "logits": sel.logits, "acc": state["acc"],
                "stats": state["stats"]}
    if case["graph"]:
        state["graph"].replay()
    else:
        _layers(state)
    return {"y": state["y"]} if state["x"] is None else {"y": state["y"], "x": state["x"]}


# ------------------------------------------------------------- necessary work
def _expected_selection(case):
    """(activated experts per token, distinct experts per layer) of logits with the workload's spread: sampled."""
    w = _workload(case)
    rng = np.random.Generator(np.random.PCG64(12345))
    T, E = case["tokens"], case["experts"]
    n = min(T, 256)
    ks, us = [], []
    for _ in range(4):
        std = rng.uniform(*w.router_std)
        if not w.rms_norm_x:
            std = w.router_std[0]
        g = rng.standard_normal((n, E)) * std
        k = np.empty(n, int)
        order = np.argsort(-g, axis=1)
        mass = np.cumsum(np.take_along_axis(np.exp(g - g.max(1, keepdims=True)), order, 1), 1)
        below = (mass < case["p"] * mass[:, -1:]).sum(1)
        if case["rule"] == "topk":
            k[:] = min(E, max(1, int(case["p"])))
        elif case["rule"] == "lte":
            k[:] = (1.0 / (1.0 + np.exp(-g)) > case["p"]).sum(1)
        elif case["p"] >= 1.0:
            k[:] = E
        elif case["rule"] == "paper":
            k[:] = np.maximum(1, below)
        else:
            k[:] = np.minimum(E, below + 1)
        hit = np.zeros((n, E), bool)
        np.put_along_axis(hit, order, np.arange(E)[None, :] < k[:, None], 1)
        ks.append(k.mean())
        missed = (1.0 - hit.mean(0)) ** T if T > n else ~hit.any(0)
        us.append(E - missed.sum())
    return float(np.mean(ks)), float(np.mean(us))


def work(case):
    w = _workload(case)
    d, E = case["d"], case["experts"]
    esz = 2 if w.dtype == "bf16" else 4
    mats = 3 if w.gated else 2
    if case["kind"] == "permute":
        return {"bytes": 2 * mats * 64 * E * d * esz + 4 * 64 * E, "flops": 0}
    T = case["tokens"]
    router_flops = 2 * T * E * d
    if case["kind"] == "route":
        return {"bytes": (T * d + E * d) * esz + 12 * T * E + 4 * T + 8 * (E + 2) + 24, "flops": router_flops}
    k, u = _expected_selection(case)
    rows = T * d * esz
    nbytes = E * d * esz + u * mats * 64 * d * esz + 2 * rows + (2 * rows + d * esz if case["entry"] == "chained" else 0)
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * (router_flops + 2 * T * k * mats * 64 * d)}


# ------------------------------------------------------------------ 64 bits
def _select64(g, case):
    """(order [T, E], counts [T]) of fp64 logits, equal logits by the lower index."""
    E = g.shape[1]
    order = torch.sort(-g, dim=1, stable=True).indices
    if case["rule"] == "topk":
        return order, torch.full((g.shape[0],), min(E, max(1, int(case["p"]))), device=g.device)
    p = float(np.float32(case["p"]))
    if case["rule"] == "lte":
        return order, (torch.sigmoid(g) > p).sum(1)
    if p >= 1.0:
        return order, torch.full((g.shape[0],), E, device=g.device)
    mass = torch.softmax(g, 1).gather(1, order).cumsum(1)
    below = (mass < p).sum(1)
    return order, below.clamp(min=1) if case["rule"] == "paper" else (below + 1).clamp(max=E)


def _ffn64(t, x, g, case):
    w = _workload(case)
    order, counts = _select64(g, case)
    on = torch.zeros_like(g, dtype=torch.bool)
    on.scatter_(1, order, torch.arange(g.shape[1], device=g.device)[None, :] < counts[:, None])
    y = torch.zeros_like(x)
    for e in on.any(0).nonzero().flatten().tolist():
        rows = on[:, e].nonzero().flatten()
        xe, s = x[rows], slice(64 * e, 64 * e + 64)
        h = xe @ t["Wu"][s].double().T
        if w.act == "swiglu":
            h = h * torch.nn.functional.silu(xe @ t["Wg"][s].double().T)
        elif w.act == "relu":
            h = h.clamp(min=0.0)
        else:
            h = torch.nn.functional.gelu(h, approximate="tanh")
        if case["gate"] == "sigmoid":
            h = h * torch.sigmoid(g[rows, e])[:, None]
        y.index_add_(0, rows, h @ t["Wd"][:, s].double().T)
    return y


def exact(case, seed):
    layers = _tensors(case, seed)
    t = layers[0]
    if case["kind"] == "permute":
        perm = _perm(case, seed).long()
        return [None if t["Wg"] is None else t["Wg"][perm], t["Wu"][perm], t["Wd"][:, perm].contiguous()]
    if case["kind"] == "route":
        g = t["x"].double() @ t["Wr"].double().T
        order, counts = _select64(g, case)
        keep = torch.arange(g.shape[1], device=g.device)[None, :] < counts[:, None]
        gates = torch.sigmoid(g.gather(1, order)) if case["gate"] == "sigmoid" else torch.ones_like(g)
        prob = torch.softmax(g, 1)
        stats = torch.stack([-(prob * torch.log(prob + EPS_STATS)).sum(1).mean(),
                             g.shape[1] * prob.mean(0).square().sum(), torch.sigmoid(g).mean()])
        return {"ids": None, "counts": None, "gates": gates * keep, "logits": g, "acc": None, "stats": stats}
    ys, xs = [], []
    for t in layers:
        x = t["x"].double()
        if case["entry"] == "chained":
            x = x + t["y_prev"].double()
            x = x * torch.rsqrt(x.square().mean(1, keepdim=True) + EPS_NORM) * t["gamma"].double()
            xs.append(x)
            x = x.to(t["x"].dtype).double()  # the layer reads the stored x
        ys.append(_ffn64(t, x, x @ t["Wr"].double().T, case))
    return {"y": torch.stack(ys)} if not xs else {"y": torch.stack(ys), "x": torch.stack(xs)}
