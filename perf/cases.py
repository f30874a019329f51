"""Performance cases of the MoE layer forward, through the public Python API.

A case is one call that a program makes: a forward over resident experts
(``Plan.forward``: what a server with the layer's experts in device memory
does, from one decoded token to a long prefill), a forward over a pool smaller
than the layer (``Plan.forward_streamed``: experts staged from pinned host
windows in LRU waves), or a decode step of a stack of streamed layers
(``Plan.forward_streamed_stack``).

Inputs follow the benchmark's distributions: rows N(0, 1) in bf16, router,
expert and shared weights N(0, 0.02), 4-bit weights quantised from such
weights per group of 32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_23805_gb300 import api
from paper_2608_23805_gb300 import native as N

# The benchmark's layer (Qwen3-Next-shaped) and its tiny layer.
LARGE = {"hidden": 2048, "inter": 512, "experts": 512, "top_k": 10, "shared": True, "residual": False}
TINY = {"hidden": 256, "inter": 128, "experts": 16, "top_k": 2, "shared": False, "residual": False}
STACK_LAYERS = 48
SLOTS = 64  # pool of the streamed cases
CHUNK = 64  # experts generated at a time


def _case(kind, shape, tokens, weights, name=None, **kw):
    c = {"kind": kind, **shape, "tokens": tokens, "weights": weights, **kw}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a small layer over one batch: a smoke-sized model, all launches and latency
        _case("resident", TINY, 64, "bf16", "tiny_64"),
        # decoding one sequence, a few, and a full batch of them
        _case("resident", LARGE, 1, "bf16", "bf16_1"),
        _case("resident", LARGE, 37, "bf16", "bf16_37"),
        # a chunk of a prefill mixed with decode rows
        _case("resident", LARGE, 600, "bf16", "bf16_600"),
        # prefills: a long prompt, and the longest
        _case("resident", LARGE, 4096, "bf16", "bf16_4096"),
        _case("resident", LARGE, 32768, "bf16", "bf16_32768"),
        # the same with 4-bit experts
        _case("resident", LARGE, 8, "q4", "q4_8"),
        _case("resident", LARGE, 250, "q4", "q4_250"),
        _case("resident", LARGE, 4096, "q4", "q4_4096"),
        # a prefill whose experts do not fit the pool: staged in LRU waves
        _case("streamed", LARGE, 32768, "bf16", "bf16_32768_lru64"),
        _case("streamed", LARGE, 32768, "q4", "q4_32768_lru64"),
        # one decode step of a 48-layer stack that shares one 64-slot pool
        _case("stack", dict(TINY, residual=True), 64, "bf16", "decode48_64"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Resident calls of 1 to 32,768 rows over the benchmark's layer (either
    weight format) make up half; the rest are small and middle layers of
    other shapes, streamed prefills and decode stacks."""
    u = rng.random()
    weights = rng.choice(["bf16", "q4"])
    if u < 0.5:
        return _case("resident", LARGE, _log_int(rng, 1, 32768), weights)
    if u < 0.75:
        experts = rng.choice([16, 32, 48, 64, 96, 128, 256])
        shape = {"hidden": 256 * rng.randint(1, 8), "inter": 128 * rng.randint(1, 6), "experts": experts,
                 "top_k": rng.randint(1, min(10, experts)), "shared": rng.random() < 0.5,
                 "residual": rng.random() < 0.5}
        return _case("resident", shape, _log_int(rng, 1, 8192), weights)
    if u < 0.9:
        return _case("streamed", LARGE, _log_int(rng, 256, 32768), weights)
    return _case("stack", dict(TINY, residual=True), rng.randint(1, 64), "bf16")


# --------------------------------------------------------------------------
# inputs, from the seed alone
# --------------------------------------------------------------------------
def _layers(case):
    return STACK_LAYERS if case["kind"] == "stack" else 1


def _gen(*key):
    return torch.Generator(device="cuda").manual_seed(int(np.random.SeedSequence(key).generate_state(1, np.uint64)[0] >> 1))


def _randn(shape, gen, scale=1.0, dtype=torch.bfloat16):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype).mul_(scale)


def _quantise(w):
    """[n, rows, cols] -> (codes [n, rows, cols / 2] uint8, scales [n, rows, cols / 32] fp16):
    scale = absmax / 7, code = round(w / scale) + 8, the even column in the low nibble."""
    n, rows, cols = w.shape
    g = w.float().view(n, rows, cols // 32, 32)
    s = (g.abs().amax(-1) / 7).to(torch.float16)
    sf = s.float().clamp_min(1e-30)[..., None]
    q = (torch.round(g / sf) + 8).clamp_(0, 15).to(torch.uint8).view(n, rows, cols // 2, 2)
    return q[..., 0] | (q[..., 1] << 4), s


def _extents(case, seed, layer, lo, hi):
    """Experts lo .. hi - 1 (lo a multiple of CHUNK) as extent bytes [n, extent_bytes]."""
    H, I, n = case["hidden"], case["inter"], hi - lo
    gen = _gen(seed, 1, layer, lo)
    w13, w2 = _randn((n, 2 * I, H), gen, 0.02), _randn((n, H, I), gen, 0.02)
    if case["weights"] == "bf16":
        parts = [w13, w2]
    else:
        c13, s13 = _quantise(w13)
        c2, s2 = _quantise(w2)
        parts = [c13, c2, s13, s2]
    return torch.cat([p.contiguous().view(n, -1).view(torch.uint8) for p in parts], dim=1)


def _chunks(case):
    E = case["experts"]
    return [(lo, min(lo + CHUNK, E)) for lo in range(0, E, CHUNK)]


def _dense(case, ext):
    """Extent bytes [n, extent_bytes] -> (W13 [n, 2I, H], W2 [n, H, I]) in fp64."""
    H, I, n = case["hidden"], case["inter"], ext.shape[0]
    if case["weights"] == "bf16":
        w = ext.view(torch.bfloat16).double()
        return w[:, :2 * I * H].view(n, 2 * I, H), w[:, 2 * I * H:].view(n, H, I)
    HI = H * I
    cut = [0, HI, HI + HI // 2, HI + HI // 2 + HI // 8, HI + HI // 2 + HI // 8 + HI // 16]
    part = [ext[:, a:b].contiguous() for a, b in zip(cut, cut[1:])]

    def weights(codes, scales, rows, cols):
        codes = codes.view(n, rows, cols // 2)
        q = torch.stack([codes & 15, codes >> 4], dim=-1).view(n, rows, cols // 32, 32).double() - 8
        return (q * scales.view(torch.float16).view(n, rows, cols // 32, 1).double()).view(n, rows, cols)

    return weights(part[0], part[2], 2 * I, H), weights(part[1], part[3], H, I)


def _small_inputs(case, seed):
    """Rows, routers and the shared expert (None without one)."""
    T, H, I, E, L = case["tokens"], case["hidden"], case["inter"], case["experts"], _layers(case)
    gen = _gen(seed, 0)
    x = _randn((T, H), gen)
    routers = _randn((L, E, H), gen, 0.02, torch.float32)
    if not case["shared"]:
        return x, routers, None, None
    return x, routers, _randn((3 * I * H,), gen, 0.02), _randn((1, H), gen, 0.02, torch.float32)


class _Events:
    """The route events of a call's layers in one set of buffers, layer by layer."""

    def __init__(self, L, T, k, E):
        self.ids = torch.empty((L, T, k), dtype=torch.int32, device="cuda")
        self.weights = torch.empty((L, T, k), dtype=torch.float32, device="cuda")
        self.counts = torch.empty((L, E), dtype=torch.int32, device="cuda")
        self.gap = torch.empty((L, T), dtype=torch.float32, device="cuda")
        self.layers = [_Event(*(t[l] for t in (self.ids, self.weights, self.counts, self.gap))) for l in range(L)]

    def outputs(self):
        return {"ids": self.ids, "weights": self.weights, "counts": self.counts, "gap": self.gap}


class _Event:
    def __init__(self, ids, weights, counts, gap):
        self.c = N.msi_route_event(*(t.data_ptr() for t in (ids, weights, counts, gap)))


def prepare(case, seed):
    """A plan with its experts in pinned host windows (and, for a resident
    case, in its slots), the call's rows and the output buffers."""
    T, H, E, L = case["tokens"], case["hidden"], case["experts"], _layers(case)
    resident = case["kind"] == "resident"
    wdtype = N.MSI_W_BF16 if case["weights"] == "bf16" else N.MSI_W_Q4G32
    eb = int(N.lib().msi_extent_bytes(H, case["inter"], wdtype))
    windows = torch.empty((L * E, eb), dtype=torch.uint8, pin_memory=True)
    for l in range(L):
        for lo, hi in _chunks(case):
            windows[l * E + lo:l * E + hi].copy_(_extents(case, seed, l, lo, hi), non_blocking=True)
    x, routers, shared_w, gate_w = _small_inputs(case, seed)
    torch.cuda.synchronize()
    plan = api.Plan(n_layers=L, n_experts=E, top_k=case["top_k"], hidden=H, inter=case["inter"],
                    n_slots=E if resident else SLOTS, host_windows=windows, has_shared=case["shared"],
                    shared_w=shared_w, shared_gate_w=gate_w, wdtype=wdtype, early_staging=not resident)
    state = {"case": case, "plan": plan, "x": x, "routers": [routers[l] for l in range(L)],
             "ev": _Events(L, T, case["top_k"], E), "out": torch.empty_like(x),
             "stage": torch.cuda.Stream()}
    if case["kind"] == "stack":
        state["out_b"] = torch.empty_like(x)
    if resident:
        # the slots an earlier churn left the experts in: any order
        for e, slot in enumerate(np.random.default_rng(seed).permutation(E)):
            plan.stage(int(slot), 0, e)
        torch.cuda.synchronize()
        state["table"], state["gens"] = plan.slot_table(0)
    return state


def run(state):
    case, plan, ev = state["case"], state["plan"], state["ev"]
    if case["kind"] == "resident":
        out, _ = plan.forward(0, state["x"], state["routers"][0], state["table"], state["gens"],
                              out=state["out"], ev=ev.layers[0], residual=case["residual"])
    elif case["kind"] == "streamed":
        out, _ = plan.forward_streamed(0, state["x"], state["routers"][0], out=state["out"], ev=ev.layers[0],
                                       residual=case["residual"], stage_stream=state["stage"])
    else:
        out = plan.forward_streamed_stack(0, state["x"], state["routers"], state["out"], state["out_b"],
                                          ev.layers, residual=case["residual"], stage_stream=state["stage"])
    return {"out": out, **ev.outputs()}


def work(case):
    """Each needed expert's weights read once (for the streamed cases from the
    host: the bytes that cross to the device), rows in and out, the router;
    2 flops per multiply-add of the three projections of every routed row, the
    shared expert's and the router's."""
    T, H, I, E, k, L = (*(case[n] for n in ("tokens", "hidden", "inter", "experts", "top_k")), _layers(case))
    used = E * (1 - (1 - k / E) ** T)  # expected experts that some row selects
    per_weight = 2 if case["weights"] == "bf16" else 0.5625
    weight_bytes = used * 3 * H * I * per_weight + E * H * 4 + (3 * H * I * 2 + H * 4 if case["shared"] else 0)
    row_bytes = T * (4 * H + 8 * k + 4)
    flops = T * (6 * H * I * (k + case["shared"]) + 2 * H * E)
    return {"bytes": float(L * (weight_bytes + row_bytes)), "flops": float(L * flops)}


def tolerance(case):
    # bf16 outputs of bf16 intermediates (h, the expert outputs): each rounding
    # is up to 2^-9, and the outputs are 3e-3 (2-norm) from 64 bits; two paths
    # with their roundings apart differ by up to twice that.  A pair of logits
    # closer than their sums' rounding may change places: rarely, and each such
    # row moves two ids and two counts and mixes another expert's output in.
    # Through a stack a change of rounding travels on to all later layers.
    if case["kind"] == "stack":
        return {"rel": 0.014, "max": 0.9, "differ": 0.009}
    if case["tokens"] >= 1024:
        return {"rel": 6e-3, "max": 0.9, "differ": 0.009}
    return {"rel": 6e-3, "max": 0.3, "differ": 0.004}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------
def _exact_layer(case, seed, layer, x, router, shared_w, gate_w):
    T, H, I, k = case["tokens"], case["hidden"], case["inter"], case["top_k"]
    logits = x @ router.double().t()
    order = torch.sort(logits, dim=1, descending=True, stable=True)
    top, ids = order.values[:, :k], order.indices[:, :k]
    gap = top[:, k - 1] - order.values[:, k] if k < case["experts"] else torch.full_like(top[:, 0], math.inf)
    weights = torch.softmax(top, dim=1)

    def ffn(rows, w13, w2):
        gu = rows @ w13.t()
        return (torch.nn.functional.silu(gu[:, :I]) * gu[:, I:]) @ w2.t()

    out = torch.zeros((T, H), dtype=torch.float64, device="cuda")
    flat = ids.reshape(-1)
    by_expert = torch.argsort(flat, stable=True)
    counts = torch.bincount(flat, minlength=case["experts"])
    ends = torch.cumsum(counts, 0).tolist()
    for lo, hi in _chunks(case):
        if ends[hi - 1] == (ends[lo - 1] if lo else 0):
            continue
        w13, w2 = _dense(case, _extents(case, seed, layer, lo, hi))
        for e in range(lo, hi):
            at = by_expert[(ends[e - 1] if e else 0):ends[e]]
            if at.numel():
                t = at // k
                out.index_add_(0, t, ffn(x[t], w13[e - lo], w2[e - lo]) * weights.reshape(-1)[at, None])
        del w13, w2
    if case["shared"]:
        w = shared_w.double()
        y = ffn(x, w[:2 * I * H].view(2 * I, H), w[2 * I * H:].view(H, I))
        out += torch.sigmoid(x @ gate_w[0].double())[:, None] * y
    if case["residual"]:
        out += x
    return out, ids.to(torch.int32), weights, counts.to(torch.int32), gap


def exact(case, seed):
    x, routers, shared_w, gate_w = _small_inputs(case, seed)
    x, seen = x.double(), []
    for l in range(_layers(case)):
        # the next layer's input is this one's bf16 output
        out, *event = _exact_layer(case, seed, l, x, routers[l], shared_w, gate_w)
        seen.append(event)
        x = out.to(torch.bfloat16).double()
    ids, weights, counts, gap = (torch.stack([s[i] for s in seen]) for i in range(4))
    return {"out": out, "ids": ids, "weights": weights, "counts": counts, "gap": gap}
