"""The work this framework is measured on: EAT MoE-layer calls through the public binding.

Layers have the shapes of `paper_2609_33614_gb300.workloads` (the toy fp32 layer and the layers
shaped like Mixtral-8x7B, OLMoE, Qwen1.5-MoE and DeepSeek-V2-Lite) with their input recipe: router
weights N(0, 0.02^2) plus a per-expert logit bias, expert weights N(0, 0.02^2), hidden states
N(0, 1).  A case names the shape, the expert-weight type, the entry point, the number of tokens of
a call and the routing options; every draw follows from the seed.

History: a serving handle has routed many tokens before the call that is measured.  "warm" gives
the handle the accounts such traffic leaves (the top-K counts and probabilities of sampled tokens,
scaled up, and typical output norms); "fresh" is a handle just created (a first prompt).
"""
from __future__ import annotations

import math

import torch

from paper_2609_33614_gb300 import eat, workloads as W

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.bfloat16}
HISTORY_TOKENS = 2048   # sampled tokens behind a warm history
HISTORY_SCALE = 512     # how many such samples the handle has seen


def _case(name, shape, weights, entry, tokens, history="warm", router="eat", sign=0,
          temporal=False, returns="y"):
    return dict(name=name, shape=shape, weights=weights, entry=entry, tokens=tokens,
                history=history, router=router, sign=sign, temporal=temporal, returns=returns)


def listed():
    return [
        # routing alone for a decode batch, from the caller's own buffers (a serving process that
        # keeps all device memory in its pool): the smallest call of the library
        _case("route_noalloc_olmoe_32", "olmoe", "bf16", "route_noalloc", 32),
        # the fp32 layer: a short step, and a long ragged one; a program that checkpoints the
        # expert history with its state reads the accounts back
        _case("toy_f32_64", "toy", "f32", "forward", 64, "fresh", returns="y+accounts"),
        _case("toy_f32_1999", "toy", "f32", "forward", 1999, returns="y+accounts"),
        # one sequence being generated: weights of two experts streamed for one token
        _case("mixtral_decode_1", "mixtral", "bf16", "forward", 1),
        # a full decode batch on e4m3 weights
        _case("mixtral_fp8_decode_64", "mixtral", "fp8", "forward", 64, sign=-1),
        # decode batch of many small experts; the program reads the routing for its statistics
        _case("olmoe_decode_32", "olmoe", "bf16", "forward", 32, sign=1, returns="y+routing"),
        # decode batch with always-on shared experts and per-sequence threshold smoothing
        _case("dsv2l_decode_128", "dsv2l", "bf16", "forward", 128, temporal=True),
        # a decode batch of a program that keeps its hidden states in page-locked host memory
        _case("host_olmoe_decode_48", "olmoe", "bf16", "host", 48),
        # one chunk of a chunked prefill (or a large ragged batch), with shared experts
        _case("qwen_chunk_333", "qwen", "bf16", "forward", 333),
        # a prompt batch, first on its handle
        _case("olmoe_prefill_4096", "olmoe", "bf16", "forward", 4096, "fresh",
              returns="y+accounts"),
        # a ragged prompt batch on e4m3 weights
        _case("olmoe_fp8_prefill_3001", "olmoe", "fp8", "forward", 3001),
        # the largest prompt batch
        _case("dsv2l_prefill_16384", "dsv2l", "bf16", "forward", 16384),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


# The ranges behind the listed cases: (shapes, weight types, entry point, tokens from, to).  The
# Mixtral-shaped layer ends at 2048 tokens and e4m3 layers at 4096, so that no draw costs more than
# the largest listed case.
RANGES = [
    (("olmoe", "qwen", "mixtral", "dsv2l"), ("bf16",), "route_noalloc", 1, 1024),
    (("olmoe", "qwen", "mixtral", "dsv2l"), ("bf16",), "route", 1, 4096),
    (("toy",), ("f32",), "forward", 1, 4096),
    (("mixtral", "olmoe", "qwen", "dsv2l"), ("bf16", "fp8"), "forward", 1, 128),
    (("mixtral", "olmoe", "qwen", "dsv2l"), ("bf16", "fp8"), "forward", 1, 128),
    (("mixtral", "olmoe", "qwen", "dsv2l"), ("bf16", "fp8"), "host", 1, 1024),
    (("mixtral", "olmoe", "qwen", "dsv2l"), ("bf16", "fp8"), "forward", 129, 1023),
    (("olmoe", "qwen", "dsv2l"), ("bf16",), "forward", 1024, 16384),
    (("mixtral",), ("bf16",), "forward", 1024, 2048),
    (("olmoe", "qwen", "dsv2l"), ("fp8",), "forward", 1024, 4096),
]


def draw(rng):
    shapes, weights, entry, lo, hi = rng.choice(RANGES)
    case = _case("", rng.choice(shapes), rng.choice(weights), entry, _log_int(rng, lo, hi),
                 rng.choice(("warm", "warm", "fresh")),
                 rng.choice(("eat", "eat", "eat", "eat", "topk", "topp")),
                 rng.choice((-1, 0, 1)))
    if entry == "forward":
        case["temporal"] = rng.random() < 0.25
        case["returns"] = rng.choice(("y", "y", "y+routing", "y+accounts"))
    del case["name"]
    return case


# ------------------------------------------------------------------------------------- inputs
def _gen(device, seed, k):
    return torch.Generator(device).manual_seed(1_000_003 * (seed + 1) + 7919 * k)


def _normal(shape, std, seed, k, dtype, device):
    t = torch.randn(*shape, generator=_gen(device, seed, k), device=device, dtype=torch.float32)
    return t.mul_(std).to(dtype)


def _router(s, seed, device):
    """Router weights and the per-expert logit bias of the shape's recipe."""
    w = _normal((s.n_experts, s.d_model), 0.02, seed, 1, torch.float32, "cpu")
    g = _gen("cpu", seed, 2)
    if s.bias == "zipf":
        rank = torch.randperm(s.n_experts, generator=g).double() + 1.0
        pi = rank.pow(-s.zipf_s)
        b = (pi / pi.sum()).log().float()
    else:
        b = torch.randn(s.n_experts, generator=g) * (0.6 if s.bias == "depth" else 0.5)
    return w.to(device), b.to(device)


def _tokens(s, n, seed, k, device):
    return _normal((n, s.d_model), 1.0, seed, k, s.xdtype, device)


def _probs(s, x, wr, br):
    z = (x.double() @ wr.double().T + br.double()) / s.temperature
    return torch.softmax(z, dim=1)


def _history(case, s, wr, br, seed):
    """Accounts N, P_total, C_s before the call (int64, fp64, fp64)."""
    E, dev = s.n_experts, wr.device
    if case["history"] == "fresh":
        z = torch.zeros(E, dtype=torch.float64, device=dev)
        return z.to(torch.int64), z, z.clone()
    p = _probs(s, _tokens(s, HISTORY_TOKENS, seed, 3, dev), wr, br)
    top, idx = p.topk(s.max_k, dim=1)
    n = torch.bincount(idx.flatten(), minlength=E)
    onehot = torch.zeros_like(p).scatter_(1, idx, top)
    P = onehot.sum(0) * HISTORY_SCALE
    # ||W_d (silu(g) * u)||: g, u ~ N(0, v) with v = 0.02^2 d; E[silu(g)^2] by quadrature
    v = 4e-4 * s.d_model
    t = torch.linspace(-8, 8, 1601, dtype=torch.float64)
    gs = torch.exp(-t * t / 2)
    e2 = float(((torch.nn.functional.silu(t * math.sqrt(v)) ** 2 * gs).sum() / gs.sum()))
    norm = math.sqrt(4e-4 * s.d_model * s.d_ff * e2 * v)
    jitter = torch.randn(E, generator=_gen("cpu", seed, 4), dtype=torch.float64).to(dev)
    C = norm * (1.0 + 0.01 * jitter) * (n > 0)
    return n * HISTORY_SCALE, P, C


def _fp8(w):
    """Per-row e4m3 weights and their fp32 scales (row maximum / 448)."""
    amax = w.abs().amax(dim=-1)
    scale = torch.where(amax > 0, amax.float() / 448.0, torch.ones_like(amax, dtype=torch.float32))
    q = torch.empty(w.shape, dtype=torch.float8_e4m3fn, device=w.device)
    for e in range(w.shape[0]):
        q[e] = (w[e].float() / scale[e].unsqueeze(-1)).to(torch.float8_e4m3fn)
    return q, scale


def _weights(case, s, seed, device):
    """Expert weights (gate, up, down; shared gate, up, down or None) and their scales."""
    E, d, F, S, Fs = s.n_experts, s.d_model, s.d_ff, s.n_shared, s.d_ff_shared
    shapes = [("w_gate", (E, F, d)), ("w_up", (E, F, d)), ("w_down", (E, d, F))]
    if S:
        shapes += [("ws_gate", (S, Fs, d)), ("ws_up", (S, Fs, d)), ("ws_down", (S, d, Fs))]
    out, scales = {}, {}
    for k, (name, shp) in enumerate(shapes):
        w = _normal(shp, 0.02, seed, 10 + k, DTYPES[case["weights"]], device)
        if case["weights"] == "fp8":
            w, scales[name + "_scale"] = _fp8(w)
        out[name] = w
    return out, scales


def _params(case, s):
    mode = {"eat": eat.EAT_ROUTER_EAT, "topk": eat.EAT_ROUTER_TOPK, "topp": eat.EAT_ROUTER_TOPP}
    return eat.eat_default_params(
        s.max_k, temperature=s.temperature, router_mode=mode[case["router"]],
        smoothing_mode=eat.EAT_SMOOTH_TEMPORAL if case["temporal"] else eat.EAT_SMOOTH_CALL)


class State:
    pass


def prepare(case, seed):
    s = W.SHAPES[case["shape"]]
    T, dev = case["tokens"], "cuda"
    st = State()
    st.case, st.shape = case, s
    wr, br = _router(s, seed, dev)
    N, P, C = _history(case, s, wr, br, seed)
    st.x = _tokens(s, T, seed, 5, dev)
    st.params = _params(case, s)
    if case["entry"] == "route_noalloc":
        st.wr, st.br, st.N, st.P, st.C = wr, br, N, P, C
        return st
    w, scales = _weights(case, s, seed, dev)
    st.layer = eat.EatLayer(wr, br, w["w_gate"], w["w_up"], w["w_down"], T, st.params,
                            w.get("ws_gate"), w.get("ws_up"), w.get("ws_down"), scales=scales)
    st.layer.set_accounts(N, P, C)
    if case["temporal"]:
        st.tau = torch.full((T,), float("nan"), dtype=torch.float32, device=dev)
        eat.eat_set_tau_state(st.layer.h, st.tau)
    if case["entry"] == "host":
        st.x_host = st.x.cpu().pin_memory()
        st.y_host = torch.empty_like(st.x_host).pin_memory()
    return st


def run(state):
    c = state.case
    if c["entry"] == "route_noalloc":
        s, T, dev = state.shape, c["tokens"], state.x.device
        idx = torch.empty(T, s.max_k, dtype=torch.int32, device=dev)
        w = torch.empty(T, s.max_k, dtype=torch.float32, device=dev)
        k = torch.empty(T, dtype=torch.int32, device=dev)
        eat.eat_route_noalloc(state.x, T, s.d_model, s.n_experts, eat.EAT_BF16, state.wr,
                              state.br, state.N, state.P, state.C, state.params, c["sign"],
                              idx, w, k)
        return {"idx": idx, "w": w, "k": k}
    if c["entry"] == "route":
        idx, w, k = state.layer.route(state.x, c["sign"])
        return {"idx": idx, "w": w, "k": k}
    if c["entry"] == "host":
        eat.eat_moe_forward_host(state.layer.h, state.x_host, c["tokens"], c["sign"],
                                 state.y_host)
        return {"y": state.y_host}
    if c["returns"] == "y+routing":
        y, idx, w, k = state.layer.forward(state.x, c["sign"], with_routing=True)
        out = {"y": y, "idx": idx, "w": w, "k": k}
    else:
        out = {"y": state.layer.forward(state.x, c["sign"])}
    if c["returns"] == "y+accounts":
        out["N"], out["P"], out["C"] = state.layer.accounts()
    if c["temporal"]:
        out["tau"] = state.tau
    return out


# ------------------------------------------------------------- 64-bit values (plain torch)
def _route64(case, s, p, N, P, C):
    """Selected experts (mask [T, E]), gates and final thresholds of a call, first on its
    thresholds' streams (Eq. 1-8 of the paper, the library's defaults)."""
    T, E = p.shape
    K = s.max_k
    order = torch.argsort(p, dim=1, descending=True, stable=True)
    rank = torch.empty_like(order).scatter_(
        1, order, torch.arange(E, device=p.device).expand(T, E).contiguous())
    mu = p.sum(1) / E
    sigma = torch.sqrt(((p - mu[:, None]) ** 2).sum(1) / E)
    tau = torch.maximum(0.5 * mu, mu - sigma)
    f = {1: 1.2, -1: 0.9, 0: 1.0}[case["sign"]]
    tau = 0.7 * f * tau + 0.3 * tau
    lo, hi = (torch.quantile(p, q, dim=1) for q in (0.1, 0.9))
    tau = torch.minimum(torch.maximum(tau, lo), hi)
    if case["router"] == "topk":
        sel = rank < K
    elif case["router"] == "topp":
        srt = p.gather(1, order)
        before = (torch.cumsum(srt, 1) - srt).gather(1, rank)
        sel = (rank < K) & (before < 0.6)
    else:
        n = N.double()
        a = n / n.sum() if float(n.sum()) > 0 else torch.zeros_like(n)
        b = torch.where(N > 0, P / n.clamp(min=1), torch.zeros_like(n))
        c = C / C.sum() if float(C.sum()) > 0 else torch.zeros_like(n)
        imp = 0.4 * p + 0.6 * (0.3 * a + 0.3 * b + 0.4 * c)
        by = torch.argsort(imp, dim=1, descending=True, stable=True)
        r = torch.empty_like(by).scatter_(
            1, by, torch.arange(E, device=p.device).expand(T, E).contiguous())
        cand = imp > tau[:, None]
        sel = torch.where(cand.any(1, keepdim=True), cand & (r < K), r == 0)
    g = torch.where(sel, p, torch.zeros_like(p))
    return sel, g / (g.sum(1, keepdim=True) + 1e-8), tau


def _expert64(x, w, names, scales, e):
    g, u, d = (w[n][e].double() * (scales[n + "_scale"][e].double()[:, None] if scales else 1.0)
               for n in names)
    return (torch.nn.functional.silu(x @ g.T) * (x @ u.T)) @ d.T


def exact(case, seed):
    s = W.SHAPES[case["shape"]]
    T, E, K = case["tokens"], s.n_experts, s.max_k
    dev = "cuda"
    wr, br = _router(s, seed, dev)
    N, P, C = _history(case, s, wr, br, seed)
    x = _tokens(s, T, seed, 5, dev).double()
    p = _probs(s, x, wr, br)
    sel, gate, tau = _route64(case, s, p, N, P, C)
    k = sel.sum(1)
    key = torch.where(sel, torch.arange(E, device=dev).expand(T, E), E).sort(1).values[:, :K]
    live = key < E
    idx = torch.where(live, key, -1).to(torch.int32)
    gk = gate.gather(1, key.clamp(max=E - 1)) * live
    routing = {"idx": idx, "w": gk, "k": k.to(torch.int32)}
    if case["entry"] in ("route_noalloc", "route"):
        return routing
    w, scales = _weights(case, s, seed, dev)
    y = torch.zeros_like(x)
    C2 = C.clone()
    for e in range(E):
        t = sel[:, e].nonzero().flatten()
        if t.numel():
            o = _expert64(x[t], w, ("w_gate", "w_up", "w_down"), scales, e)
            y[t] += gate[t, e, None] * o
            C2[e] = 0.05 * C[e] + 0.95 * o.norm(dim=1).mean()
    for e in range(s.n_shared):
        y += _expert64(x, w, ("ws_gate", "ws_up", "ws_down"), scales, e)
    if case["entry"] == "host":
        return {"y": y.cpu()}
    out = {"y": y}
    if case["returns"] == "y+routing":
        out.update(routing)
    if case["returns"] == "y+accounts":
        out["N"], out["P"], out["C"] = N + sel.sum(0), P + (p * sel).sum(0), C2
    if case["temporal"]:
        out["tau"] = tau
    return out


# ------------------------------------------------------------------------ work and tolerance
def work(case):
    s = W.SHAPES[case["shape"]]
    T, E, d, F = case["tokens"], s.n_experts, s.d_model, s.d_ff
    xb = 4 if case["weights"] == "f32" else 2
    route = {"bytes": E * d * 4 + T * d * xb + T * (s.max_k * 8 + 4), "flops": 2 * T * d * E}
    if case["entry"] in ("route_noalloc", "route"):
        return route
    # the experts a call activates: how often sampled tokens select each of them
    wr, br = _router(s, 0, "cpu")
    acc = _history(case, s, wr, br, 0)
    sel, _, _ = _route64(case, s, _probs(s, _tokens(s, 512, 0, 6, "cpu"), wr, br), *acc)
    f = sel.double().mean(0)
    union = float((1.0 - (1.0 - f) ** T).sum())
    acts = float(f.sum()) * T
    wb, sb = {"f32": (4, 0), "bf16": (2, 0), "fp8": (1, 4)}[case["weights"]]
    per = lambda width: 3 * d * width * wb + (2 * width + d) * sb
    nbytes = route["bytes"] + union * per(F) + T * d * xb
    flops = route["flops"] + acts * 6 * d * F
    if s.n_shared:
        nbytes += s.n_shared * per(s.d_ff_shared)
        flops += s.n_shared * T * 6 * d * s.d_ff_shared
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Relative 2-norm ("rel") and largest ("max") difference of an output, and the share of
    selected experts that may differ: about four times what the path shows against exact()."""
    # measured: gates and thresholds 1e-7 to 6e-7, fp32 outputs 6e-7 (largest 3.4e-6)
    if case["entry"] in ("route_noalloc", "route") or case["weights"] == "f32":
        return {"rel": 2.5e-6, "max": 1.5e-5, "differ": 1e-3}
    # bf16 activations and outputs, bf16 or e4m3 weights: 2.3e-3 to 2.9e-3 (largest 1.8e-2)
    return {"rel": 1.2e-2, "max": 7e-2, "differ": 1e-3}
