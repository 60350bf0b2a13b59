"""The measured cases of the ACE MoE layer: what a program that serves a mixture-of-experts
model calls, through the public entry points of `paper_2609_05228_gb300.ace`.

A case names an entry point ("kind") and the sizes and options of one pass:

  forward   ace_moe_forward       one layer on device buffers
  host      ace_moe_forward_host  one layer from and to page-locked host buffers
  stack     ace_stack_forward     a decoder's MoE layers in sequence, with residuals
  tables    ace_offline_tables_device  the GSP/RCR tables of a layer's weights

Layers follow the shapes of the repository's configurations: hidden 2048, 128 experts,
top-8, FFN 768; the large layer (4096, 256, 8, 2048); the tiny fp32 layer (256, 16, 4,
128); and generic ones around them. Inputs follow its recipe: x ~ N(0, 1), weights
~ N(0, 0.02^2), gamma ~ 1 + U(-0.1, 0.1), and for prompts a router bias that makes the
experts' popularity fall like Zipf's law.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_05228_gb300 import ace, synth

EPS = 1e-6


def _case(name, kind, T, shape, dtype="bf16", mode="ratio", value=0.5, fusion="max", zipf=False, layers=1):
    d, n, k, m = shape
    return {"name": name, "kind": kind, "tokens": T, "hidden": d, "experts": n, "top_k": k, "ffn": m, "dtype": dtype,
            "mode": mode, "value": value, "fusion": fusion, "zipf": zipf, "layers": layers}


QWEN = (2048, 128, 8, 768)
LARGE = (4096, 256, 8, 2048)
TINY = (256, 16, 4, 128)


def listed():
    return [
        # one user's next token: the smallest call, where latency and launches count
        _case("decode_1", "forward", 1, QWEN),
        # a few users; a fixed threshold, as a deployment that calibrated it once passes
        _case("decode_8_tau", "forward", 8, QWEN, mode="threshold", value=0.11),
        # a busy server's decode step
        _case("decode_64", "forward", 64, QWEN),
        # a decode step whose rows live in host memory (another device or process makes them)
        _case("decode_32_host", "host", 32, QWEN),
        # the MoE layers of a decoder, one decode step for a batch
        _case("stack4_decode_32", "stack", 32, QWEN, layers=4),
        # a large layer's decode step, skewed routing
        _case("large_decode_16", "forward", 16, LARGE, zipf=True),
        # one short prompt of odd length, a mild skip ratio
        _case("prefill_777", "forward", 777, QWEN, value=0.25, zipf=True),
        # a batch of prompts
        _case("prefill_4096", "forward", 4096, QWEN, zipf=True),
        # a large batch of prompts through a decoder's layers
        _case("stack4_prefill_16384", "stack", 16384, QWEN, layers=4),
        # a large layer's prompts
        _case("large_prefill_8192", "forward", 8192, LARGE, zipf=True),
        # the fp32 layer, as used to develop and check a model
        _case("tiny_f32_64", "forward", 64, TINY, dtype="f32"),
        # loading a model: the expert tables of one layer from its weights
        _case("tables_2048", "tables", 0, QWEN),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _cost(c):
    return c["tokens"] * c["top_k"] * c["hidden"] * c["ffn"] * c["layers"]


def draw(rng):
    kind = rng.choices(["decode", "prefill", "host", "stack", "f32", "narrow", "tables"], [5, 5, 1, 2, 1, 1, 1])[0]
    pick = rng.random()
    if pick < 0.35:
        shape = QWEN
    elif pick < 0.5 and kind != "stack":
        shape = LARGE
    else:
        n = _log_int(rng, 8, 256)
        shape = (256 * rng.randint(2, 16), n, rng.randint(1, min(n, 10)), 128 * rng.randint(1, 16))
    T = _log_int(rng, 1, 256) if kind in ("decode", "host") or (kind == "stack" and rng.random() < 0.5) else \
        _log_int(rng, 257, 16384)
    layers = rng.randint(2, 4) if kind == "stack" else 1
    if kind == "stack" and shape[1] > 128:
        shape = (shape[0], 128, shape[2], min(shape[3], 1024))
    dtype = "bf16"
    if kind == "f32":          # small layers on the CUDA cores
        n = _log_int(rng, 4, 64)
        shape = (64 * rng.randint(1, 16), n, rng.randint(1, min(n, 8)), 32 * rng.randint(1, 16))
        dtype, T = "f32", _log_int(rng, 1, 256)
    if kind == "narrow":       # bf16 sizes that are not whole tensor-core tiles
        n = _log_int(rng, 4, 64)
        shape = (64 * rng.randint(1, 16), n, rng.randint(1, min(n, 8)), 64 * rng.randint(1, 16))
        T = _log_int(rng, 1, 256)
    if kind == "tables":
        n = _log_int(rng, 8, 128)
        shape = (256 * rng.randint(2, 12), n, rng.randint(1, min(n, 8)), 64 * rng.randint(2, 24))
        T = 0
    if rng.random() < 0.75:
        mode, value = "ratio", rng.choice([0.0, 0.125, 0.25, 0.375, 0.5, 0.625])
    else:
        mode, value = "threshold", round(rng.uniform(0.5, 1.2) / shape[2], 4)
    fusion = "max" if rng.random() < 0.75 else rng.choice(["min", "mean", "gsp", "rcr", "score"])
    kinds = {"host": "host", "stack": "stack", "tables": "tables"}
    c = _case("", kinds.get(kind, "forward"), T, shape, dtype, mode, value, fusion, rng.random() < 0.5, layers)
    del c["name"]
    most = 0.5 * _cost(_case("", "forward", 8192, LARGE))
    while c["tokens"] > 1 and _cost(c) > most:
        c["tokens"] = int(c["tokens"] * 0.7)
    return c


# ----------------------------------------------------------------------- inputs


def _randn(shape, seed, tag, dtype, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + tag) & 0x7FFFFFFFFFFF)
    t = torch.randn(shape, generator=g, device="cuda", dtype=dtype)
    return t.mul_(scale) if scale != 1.0 else t


def _weights(c, seed, layer):
    """One layer's weights on the device (nn.Linear layouts) and its host tables."""
    d, n, m = c["hidden"], c["experts"], c["ffn"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    s = seed * 16 + layer
    rng = np.random.default_rng(s)
    bias = np.zeros(n, np.float32)
    if c["zipf"]:
        beta = synth.ZIPF_BETA_LARGE if d == 4096 else synth.ZIPF_BETA
        b = -beta * synth.ZIPF_S * np.log(rng.permutation(n) + 1.0)
        bias = (b - b.mean()).astype(np.float32)
    a_gsp, a_rcr = synth.make_tables(n, s)
    gamma = torch.from_numpy((1.0 + rng.uniform(-0.1, 0.1, d)).astype(np.float32)).cuda().to(dt)
    return {"router_w": _randn((n, d), s, 1, dt, 0.02), "router_b": torch.from_numpy(bias).cuda(),
            "w_gate": _randn((n, m, d), s, 2, dt, 0.02), "w_up": _randn((n, m, d), s, 3, dt, 0.02),
            "w_down": _randn((n, d, m), s, 4, dt, 0.02), "gamma": gamma, "a_gsp": a_gsp, "a_rcr": a_rcr}


def _tokens(c, seed):
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    return _randn((c["tokens"], c["hidden"]), seed * 16 + 15, 5, dt)


class _State:
    """What a serving program holds: the layers' handles and its buffers."""

    def __init__(self, case):
        self.case = case
        self.layers, self.stack = [], None

    def __del__(self):
        if self.stack:
            ace.ace_stack_destroy(self.stack)
        for h in self.layers:
            ace.ace_layer_destroy(h)


def prepare(case, seed):
    st = _State(case)
    if case["kind"] == "tables":
        st.w = _weights(case, seed, 0)
        return st
    for l in range(case["layers"]):
        w = _weights(case, seed, l)
        desc = ace.ace_layer_desc(case["hidden"], case["experts"], case["top_k"], case["ffn"], case["tokens"],
                                  ace.ACE_BF16 if case["dtype"] == "bf16" else ace.ACE_F32, EPS, EPS, 1.0, 1,
                                  int(case["zipf"]), int(case["kind"] == "stack"))
        torch.cuda.synchronize()
        st.layers.append(ace.ace_layer_create(desc, w["router_w"], w["router_b"], w["w_gate"], w["w_up"], w["w_down"],
                                              w["gamma"], w["a_gsp"], w["a_rcr"]))
        del w
    if case["kind"] == "stack":
        st.stack = ace.ace_stack_create(st.layers)
    st.x = _tokens(case, seed)
    if case["kind"] == "host":
        st.x = st.x.cpu().pin_memory()
        st.out = torch.empty_like(st.x).pin_memory()
    else:
        st.out = torch.empty_like(st.x)
    torch.cuda.empty_cache()
    return st


def run(state):
    c = state.case
    if c["kind"] == "tables":
        w = state.w
        return ace.ace_offline_tables_device(c["hidden"], c["experts"], c["ffn"], w["gamma"], w["router_w"], w["w_gate"],
                                             w["w_up"], w["w_down"], EPS)
    if c["kind"] == "stack":
        call, handle = ace.ace_stack_forward, state.stack
    else:
        call = ace.ace_moe_forward_host if c["kind"] == "host" else ace.ace_moe_forward
        handle = state.layers[0]
    call(handle, state.x, state.out, c["tokens"], c["mode"], c["value"], None, c["fusion"])
    return state.out


# ----------------------------------------------------------------------- what a pass needs


def _kept_share(c):
    """Share of the routed slots that is evaluated. Threshold mode: about half are skipped at
    tau = 0.88 / k, and the top slot of each token is kept."""
    k = c["top_k"]
    q = c["value"] if c["mode"] == "ratio" else min(1.0, 0.5 * (c["value"] * k / 0.88) ** 3)
    return max(1.0 / k, 1.0 - q)


def work(case):
    c = case
    d, n, k, m, T = c["hidden"], c["experts"], c["top_k"], c["ffn"], c["tokens"]
    E = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] == "tables":
        return {"bytes": float(n * 3 * d * m * E + n * d * E + 8 * n), "flops": float(n * (4 * d * d * m + 6 * d * m))}
    R = T * k * _kept_share(c)
    # distinct experts with a kept slot: expected, with equal or Zipf shares
    p = np.arange(1, n + 1, dtype=np.float64) ** (-synth.ZIPF_S if c["zipf"] else 0.0)
    D = min(R, float(np.sum(1.0 - np.exp(-R * p / p.sum()))))
    if T == 1:
        D = R
    one = D * 3 * d * m * E + n * d * E + 2 * T * d * E
    return {"bytes": float(one * c["layers"]), "flops": float((6 * d * m * R + 2 * d * n * T) * c["layers"])}


def tolerance(case):
    """Four times what the path differs by from exact(), or a little less: fp32 layers 2e-7 (sums of up to a few
    thousand fp32 products). bf16 layers 2.3e-3 to 2.9e-3 (the activations, the output and, above 256 tokens, the
    slot rows are rounded to bf16). Stacks 1.2e-2 to 1.9e-2: a layer's rounding moves the next layers' router
    logits, and slots near a boundary of the top-k or of the threshold change sides. The same happens to a slot
    whose score ties with the threshold up to fp32 rounding where the router's sums are taken in another order: it
    moves one token's row by that slot's share, which "max" leaves room for where such near-ties occur (large
    batches, stacks). Tables 4e-8: fp32 products accumulated over the FFN width, averaged over a matrix."""
    if case["kind"] == "tables":
        return {"rel": 1e-6, "max": 1e-5}
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 2e-5}
    if case["kind"] == "stack":
        return {"rel": 0.03, "max": 0.9}
    return {"rel": 1e-2, "max": 0.05 if case["tokens"] <= 256 else 0.9}


# ----------------------------------------------------------------------- the same in 64 bits


def _layer_exact(c, w, x):
    """x [T, d] (storage type) -> y [T, d] float64, the normalised rows rounded to the storage type as
    the layer stores them (its router and experts read those rows)."""
    T, d = x.shape
    k = c["top_k"]
    xd = x.double()
    h = xd / torch.sqrt((xd * xd).mean(1, keepdim=True) + EPS) * w["gamma"].double()
    h = h.to(x.dtype).double()
    z = h @ w["router_w"].double().T + w["router_b"].double()
    zk, ids = torch.topk(z, k, dim=1)
    g = torch.softmax(zk, dim=1)
    views = []
    for a in (w["a_gsp"], w["a_rcr"]):
        s = g * torch.from_numpy(a).cuda().double()[ids]
        views.append(s / (s.sum(1, keepdim=True) + EPS))
    pg, pr = views
    score = {"max": torch.maximum(pg, pr), "min": torch.minimum(pg, pr), "mean": (pg + pr) / 2, "gsp": pg, "rcr": pr,
             "score": g}[c["fusion"]]
    if c["mode"] == "threshold":
        skip = score < float(np.float32(c["value"]))
    else:
        n_cand = T * (k - 1)
        mq = min(n_cand, int(math.floor(float(np.float32(c["value"])) * T * k + 0.5)))
        if mq >= n_cand:
            skip = torch.ones_like(score, dtype=torch.bool)
        else:
            skip = score < torch.sort(score[:, 1:].reshape(-1)).values[mq]
            if mq == 0:
                skip = torch.zeros_like(skip)
    skip[:, 0] = False
    ghat = torch.where(skip, torch.zeros_like(g), g)
    ghat = ghat / (ghat.sum(1, keepdim=True) + EPS)
    y = torch.zeros(T, d, dtype=torch.float64, device=x.device)
    for e in range(c["experts"]):
        t, i = torch.nonzero((ids == e) & ~skip, as_tuple=True)
        if not len(t):
            continue
        he = h[t]
        act = torch.nn.functional.silu(he @ w["w_gate"][e].double().T) * (he @ w["w_up"][e].double().T)
        y.index_add_(0, t, ghat[t, i, None] * (act @ w["w_down"][e].double().T))
    return y


def exact(case, seed):
    c = case
    if c["kind"] == "tables":
        if work(c)["flops"] > 1e13:
            return None
        w = _weights(c, seed, 0)
        gam = w["gamma"].double()
        a = []
        for e in range(c["experts"]):
            G, U = (gam[:, None] * w[p][e].double().T for p in ("w_gate", "w_up"))
            D = w["w_down"][e].double().T
            up = torch.linalg.norm(U) * torch.linalg.norm(G @ D)
            gate = torch.linalg.norm(G) * torch.linalg.norm(U @ D)
            a.append(torch.sqrt(up * gate))
        gsp = torch.stack(a)
        r = w["router_w"].double()
        r = r - r.mean(0, keepdim=True)
        q = r / (torch.sqrt((r * r).mean(1, keepdim=True)) + EPS)
        a = []
        for e in range(c["experts"]):
            act = torch.nn.functional.silu(w["w_gate"][e].double() @ q[e]) * (w["w_up"][e].double() @ q[e])
            a.append(torch.linalg.norm(w["w_down"][e].double() @ act) / (torch.linalg.norm(q[e]) + EPS))
        rcr = torch.stack(a)
        return (gsp / (gsp.mean() + EPS)).cpu().numpy(), (rcr / (rcr.mean() + EPS)).cpu().numpy()
    x = _tokens(c, seed)
    for l in range(c["layers"]):
        w = _weights(c, seed, l)
        y = _layer_exact(c, w, x)
        out = x.double() + y if c["kind"] == "stack" else y
        x = out.to(x.dtype)       # layers of a stack hand on rows of the storage type
        del w
    return out.cpu() if c["kind"] == "host" else out
