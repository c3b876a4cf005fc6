"""The work whose speed counts: what a program that runs this MoE layer has it do, through its public entry points.

Two kinds of case:
  layer   `layers` different MoE layers called one after the other through MoELayer.forward, each on activations of its
          own (in a model, attention sits between them): a decode step for T = 1...16 tokens, a prefill above that.
          Decode goes through several layers, so that their weights come from HBM as in a model, not from L2.
  stack   `tokens` decode steps of OffloadedStack: `layers` stacked layers whose experts live in pinned host memory,
          `slots` of them per layer on the device, the others fetched on routing.

Widths, expert counts, ranks and token counts are those of synth/workloads.py, tests/ and bench.py; draw() takes others
from the same ranges.
"""
import math
import random

import numpy as np
import torch

import paper_2503_00245_b200 as P

MAX_DECODE_T = 16  # up to here a call is a decode step (several sequences at once), above a prefill


def _layer(name, d, f, T, *, E=8, k=2, r=0, xd="bf16", bias="none", layers=1):
    return {"name": name, "kind": "layer", "d": d, "f": f, "E": E, "k": k, "r": r, "xd": xd, "bias": bias, "T": T, "layers": layers}


def _stack(name, d, f, *, E, k, slots, layers, tokens, fp8=False, trace=False):
    return {"name": name, "kind": "stack", "d": d, "f": f, "E": E, "k": k, "slots": slots, "layers": layers, "tokens": tokens,
            "fp8": fp8, "trace": trace}


def listed():
    return [
        # the smallest call: fp32 activations, a layer of a toy model or a unit test; only latency
        _layer("tiny-decode-T1", 256, 512, 1, xd="f32", layers=4),
        # one sequence being generated on the 200M-active model class: the ordinary decode step
        _layer("wearable-decode-T1", 1024, 2816, 1, layers=4),
        # eight sequences decoded together on the same class
        _layer("wearable-decode-T8", 1024, 2816, 8, layers=4),
        # one sequence on the 1.4B-active class: the ordinary decode step of the large model
        _layer("phone-decode-T1", 2048, 5632, 1, bias="normal", layers=4),
        # weight-decomposed experts, one sequence: rank small, and the paper's rank of half the hidden width
        _layer("phone-wd128-decode-T1", 2048, 5632, 1, r=128, layers=4),
        _layer("phone-wd1024-decode-T1", 2048, 5632, 1, r=1024, layers=4),
        # the paper's own weight-decomposed widths (rank 800: no multiple of 64), an odd few sequences together
        _layer("paper-wd800-decode-T5", 1600, 4352, 5, r=800, layers=2),
        # prompts: an ordinary one, a ragged one at the paper's own widths, and the longest one with uneven expert load
        _layer("wearable-prefill-T512", 1024, 2816, 512),
        _layer("paper-prefill-T333", 1440, 3840, 333),
        _layer("phone-prefill-T2048", 2048, 5632, 2048, bias="normal"),
        # the long prompt with weight-decomposed experts
        _layer("phone-wd128-prefill-T2048", 2048, 5632, 2048, r=128),
        # experts in host memory: four of sixteen resident per layer, skewed routing, eight tokens generated
        _stack("wearable-offload-decode", 1024, 2816, E=16, k=2, slots=4, layers=4, tokens=8),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    """A case between the listed ones: widths over the whole range in steps of 8, other expert counts, any token count."""
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "wd-decode", "wd-prefill", "stack"])
    d = _log_int(rng, 256, 1024 if kind == "stack" else 2048, 8)
    f = max(64, min(5632, int(d * rng.uniform(2.0, 3.2)) // 8 * 8))
    E = rng.choice([2, 4, 8, 8, 8, 16])
    k = min(E, rng.choice([1, 2, 2, 2, 4]))
    bias = rng.choice(["none", "normal"])
    xd = "f32" if rng.random() < 0.15 else "bf16"
    if kind == "stack":
        E = rng.choice([8, 16])
        k = rng.choice([1, 2])
        c = _stack("", d, min(f, 2816), E=E, k=k, slots=rng.randint(k, 4), layers=rng.randint(2, 4), tokens=rng.randint(3, 8),
                   fp8=rng.random() < 0.3, trace=rng.random() < 0.3)
    else:
        r = 0
        if kind.startswith("wd"):
            r = min(_log_int(rng, 32, 1024, 8), d // 2 // 8 * 8)
        if kind.endswith("decode"):
            T = rng.choice([1, 1, rng.randint(2, MAX_DECODE_T)])
            layers = rng.choice([2, 3, 4]) if T == 1 else 2
            if T * d > 16384:
                xd = "bf16"  # many wide fp32 rows do not fit a decode step,
            if r and T > 1 and 32000 // f < 10:
                T = max(2, min(T, 32000 // f - 2))  # nor do many tokens with wide decomposed experts
        else:
            layers = 1
            T = _log_int(rng, MAX_DECODE_T + 1, 2048)
            T = max(MAX_DECODE_T + 1, min(T, 4096 // k))
        c = _layer("", d, f, T, E=E, k=k, r=r, xd=xd, bias=bias, layers=layers)
    del c["name"]
    return c


# ------------------------------------------------------------------ what a program has in hand before the call
def _normal(g, shape, sigma, dtype):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(sigma).to(dtype)


def _router(g, c, bias):
    w = _normal(g, (c["d"], c["E"]), c["d"] ** -0.5, torch.bfloat16)
    if bias == "none":
        return w, None
    if bias == "normal":
        return w, _normal(g, (c["E"],), 0.5, torch.float32)
    rank = torch.randperm(c["E"], generator=g, device="cuda").double() + 1.0  # "zipf": shares fall with rank ** -1.2
    return w, (-1.2 * torch.log(rank)).float()


def _dense(g, c):
    d, f, E, bf = c["d"], c["f"], c["E"], torch.bfloat16
    return P.pack_dense(_normal(g, (E, d, f), d ** -0.5, bf), _normal(g, (E, d, f), d ** -0.5, bf), _normal(g, (E, f, d), f ** -0.5, bf))


def _decomposed(g, c):
    d, f, E, r, bf = c["d"], c["f"], c["E"], c["r"], torch.bfloat16
    return P.pack_wd(_normal(g, (E, d, r), d ** -0.5, bf), _normal(g, (E, r, f), r ** -0.5, bf),
                     _normal(g, (E, d, r), d ** -0.5, bf), _normal(g, (E, r, f), r ** -0.5, bf),
                     _normal(g, (E, f, r), f ** -0.5, bf), _normal(g, (E, r, d), r ** -0.5, bf))


def _prepare_layers(c, g):
    xdt = torch.float32 if c["xd"] == "f32" else torch.bfloat16
    layers, xs = [], []
    for _ in range(c["layers"]):
        w, b = _router(g, c, c["bias"])
        experts = {"wd": _decomposed(g, c)} if c["r"] else {"dense": _dense(g, c)}
        layers.append(P.MoELayer(c["d"], c["f"], c["E"], c["k"], w, b, x_dtype=xdt, max_tokens=c["T"], **experts))
        xs.append(_normal(g, (c["T"], c["d"]), 1.0, xdt))
    return {"kind": "layer", "layers": layers, "xs": xs}


def _sticky_sets(rng, c):
    """Expert sets [token][layer][k] of a text whose routing changes slowly: a set keeps its members, or swaps one."""
    cur = [rng.sample(range(c["E"]), c["k"]) for _ in range(c["layers"])]
    out = []
    for _ in range(c["tokens"]):
        for s in cur:
            if rng.random() < 0.4:
                s[rng.randrange(c["k"])] = rng.choice([e for e in range(c["E"]) if e not in s])
        out.append([list(s) for s in cur])
    return out


def _prepare_stack(c, g, seed):
    def gen():
        for _ in range(c["layers"]):
            w, b = _router(g, c, "zipf")
            yield {"w_router": w, "b_router": b, "gud": _dense(g, c)}

    stack = P.OffloadedStack(c["d"], c["f"], c["E"], c["k"], c["slots"], gen(), fp8=c["fp8"])
    return {"kind": "stack", "stack": stack, "x": _normal(g, (c["tokens"], c["d"]), 1.0, torch.float32),
            "sets": _sticky_sets(random.Random(seed), c) if c["trace"] else None}


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return _prepare_stack(case, g, seed) if case["kind"] == "stack" else _prepare_layers(case, g)


def run(state):
    if state["kind"] == "layer":
        return [layer.forward(x) for layer, x in zip(state["layers"], state["xs"])]
    h = state["x"].clone()  # the embeddings of the tokens; every step turns its row into the stack's output
    if state["sets"] is not None:
        for t, sets in enumerate(state["sets"]):
            state["stack"].step_trace(h[t], sets)
        return {"h": h}
    chosen = [state["stack"].step(h[t]) for t in range(h.shape[0])]
    return {"h": h, "experts": np.array(chosen, dtype=np.int32)}


# ------------------------------------------------------------------ what one pass cannot do without
def _expected_experts(E, k, T):
    return E * (1.0 - (1.0 - k / E) ** T)  # distinct experts that T tokens select under even routing


def work(case):
    c = case
    d, f, E, k = c["d"], c["f"], c["E"], c["k"]
    if c["kind"] == "stack":
        # every token reads its experts' weights from HBM; what misses cost on the host link depends on the routing
        n = c["tokens"] * c["layers"]
        return {"bytes": n * (k * 6.0 * d * f + 2 * d * E) + 8.0 * d * c["tokens"], "flops": n * k * 6.0 * d * f}
    per_expert = 3.0 * c["r"] * (d + f) if c["r"] else 3.0 * d * f  # values
    xb = 4 if c["xd"] == "f32" else 2
    one = 2 * per_expert * _expected_experts(E, k, c["T"]) + 2 * d * E + 2 * xb * d * c["T"]
    return {"bytes": c["layers"] * one, "flops": c["layers"] * c["T"] * k * 2 * per_expert}


def tolerance(case):
    """About four times what the layer differs by from the same sums in 64 bits (measured over the listed and drawn cases):
    2e-7 to 3e-7 for fp32 rows whose hidden activations stay fp32 (one token, or decomposed experts in a decode step),
    1.7e-3 for bf16 rows there, the rounding of y alone, and 2.2e-3 to 2.9e-3 where the hidden activations, or a stacked
    layer's input, are rounded to bf16 as well."""
    if case["kind"] == "layer" and (case["T"] == 1 or (case["r"] and case["T"] <= MAX_DECODE_T)):
        return {"rel": 1e-5, "max": 1e-4} if case["xd"] == "f32" else {"rel": 7e-3, "max": 2e-2}
    return {"rel": 1.1e-2, "max": 5e-2}
