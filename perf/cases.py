"""Performance cases of the library: what a generative-recommendation server has it do, through the public entry points.

Two kinds of work:

* ``generate``: a batch of requests is admitted (their post-prefill states go to the shared-state store), every decode
  call selects or takes its parents, updates the ancestry index and decodes every layer, and at the end the requests are
  released.  One pass is a whole generation, so every chain depth from 1 to ``steps`` is in it.
* ``prefill``: the prompts of a batch of requests are turned into shared states, one call per (request, layer), and the
  states are read back (what a prefill worker hands to a decode worker).

Keys of a ``generate`` case: requests, layers, heads (key heads), v_heads (value heads; equal to heads unless grouped),
dk, dv, dtype (records and queries), out (outputs), beam, steps, parents ("uniform" / "zipf" with exponent zipf: a parent
map that the caller holds; "select": the library's own beam selection over ``codes`` codes feeds the index), fused (append
and decode in one call), delta (the (alpha, delta, k) record format), graph (the generation is captured once in a CUDA
graph and replayed).  Keys of a ``prefill`` case: requests, layers, heads, dk, dv, dtype, tokens.
"""
from __future__ import annotations

import math

import torch

import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

_ELEM = {"bf16": 2, "fp32": 4}
_TORCH = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _generate(name, **kw):
    case = dict(name=name, kind="generate", requests=1, layers=1, heads=32, v_heads=0, dk=128, dv=128, dtype="bf16", out="bf16",
                beam=512, steps=4, parents="uniform", zipf=0.0, codes=0, fused=True, delta=False, graph=False)
    case.update(kw)
    case["v_heads"] = case["v_heads"] or case["heads"]
    return case


def _prefill(name, **kw):
    case = dict(name=name, kind="prefill", requests=1, layers=1, heads=32, dk=128, dv=128, dtype="bf16", tokens=4096)
    case.update(kw)
    return case


def listed():
    return [
        # The smallest call: eight beams, two 32 x 32 heads in fp32 (a tiny model, or a latency probe). Launches and host time.
        _generate("tiny_beam8_fp32", heads=2, dk=32, dv=32, dtype="fp32", out="fp32", beam=8, steps=3),
        # One user, a narrow beam over a four-token semantic id, one layer: an interactive request.
        _generate("one_user_beam128", heads=16, beam=128),
        # One user, a wide beam through a sixteen-layer decoder, selection on the device, calls issued eagerly.
        _generate("one_user_beam512_16layers", layers=16, parents="select", codes=256),
        # A large batch of wide beams whose parents are spread evenly: many distinct ancestors.
        _generate("batch8_beam1024", requests=8, beam=1024, steps=6),
        # The full decode stack, beams that share ancestors, the generation replayed as a CUDA graph: a loaded server.
        _generate("stack16_beam512_graph", requests=4, layers=16, steps=8, parents="zipf", zipf=1.5, graph=True),
        # Narrow heads.
        _generate("heads64_beam512", requests=4, layers=2, dk=64, dv=64, steps=8, parents="zipf", zipf=1.5),
        # Wide heads.
        _generate("heads256_beam512", requests=4, layers=2, dk=256, dv=256, parents="zipf", zipf=1.5),
        # fp32 records and outputs, append and decode as separate calls (the caller decodes a layer more than once, or late).
        _generate("fp32_separate_append", requests=2, layers=2, heads=16, dtype="fp32", out="fp32", beam=256, fused=False),
        # Grouped value heads with wide values, a ragged beam, selection on the device over a larger codebook.
        _generate("grouped_wide_beam333", requests=3, layers=2, heads=8, v_heads=16, dv=256, beam=333, steps=5, parents="select", codes=512),
        # The (alpha, delta, k) record format.
        _generate("delta_records_beam200", requests=2, layers=2, beam=200, steps=6, parents="zipf", zipf=1.2, delta=True),
        # A long user history of one layer.
        _prefill("prefill_16384", tokens=16384),
        # Two short histories of odd length, narrow heads, fp32.
        _prefill("prefill_1021_fp32", requests=2, heads=16, dk=64, dv=64, dtype="fp32", tokens=1021),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.2:
        case = _prefill("", requests=rng.randint(1, 3), layers=rng.randint(1, 3), heads=rng.choice([2, 8, 16, 32]), dtype=rng.choice(["bf16", "bf16", "fp32"]),
                        tokens=_log_int(rng, 24, 16384))
        case["dk"] = case["dv"] = rng.choice([32, 64, 128, 128])
        while case["requests"] * case["layers"] * case["heads"] * case["tokens"] > 32 * 16384:     # no more than the long history
            if case["requests"] * case["layers"] == 1:
                case["tokens"] = case["tokens"] * 2 // 3
            elif case["layers"] > 1:
                case["layers"] -= 1
            else:
                case["requests"] -= 1
        del case["name"]
        return case
    case = _generate("", requests=rng.randint(1, 8), layers=_log_int(rng, 1, 16), heads=rng.choice([4, 8, 16, 24, 32]), beam=_log_int(rng, 8, 1024),
                     steps=rng.randint(2, 8), fused=rng.random() < 0.8, graph=rng.random() < 0.3)
    case["dk"], case["dv"] = rng.choice([(128, 128)] * 5 + [(64, 64)] * 2 + [(256, 256), (128, 256), (128, 512), (256, 512), (32, 32)])
    case["dtype"] = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    case["out"] = rng.choice([case["dtype"], case["dtype"], "fp32"])
    case["v_heads"] = case["heads"]
    if (case["dk"], case["dv"]) in ((64, 64), (128, 128), (128, 256)) and rng.random() < 0.25:
        case["heads"] //= 2                                                                       # two value heads per key head
    elif case["dk"] == case["dv"] <= 128 and rng.random() < 0.15:
        case["delta"] = case["fused"] = True
    case["parents"] = rng.choice(["uniform", "zipf", "select"])
    if case["parents"] == "zipf":
        case["zipf"] = round(rng.uniform(1.1, 1.6), 2)
    elif case["parents"] == "select":
        case["codes"] = rng.choice([128, 256, 512, 1000])
    limit = work(_largest())["bytes"]
    while work(case)["bytes"] > limit:
        case["layers" if case["layers"] > 1 else "requests"] -= 1
    del case["name"]
    return case


def _largest():
    return next(c for c in listed() if c["name"] == "stack16_beam512_graph")


def _widths(case):
    """Beam width of every decode call: selection from the root finds at most ``codes`` candidates."""
    first = min(case["beam"], case["codes"]) if case["parents"] == "select" else case["beam"]
    return [first] + [case["beam"]] * (case["steps"] - 1)


# ---- inputs ------------------------------------------------------------------------------------------------------------
def _unit(gen, shape, dtype):
    """N(0, 1) vectors, L2-normalised, in the storage dtype."""
    x = torch.randn(shape, generator=gen, device="cuda")
    x /= torch.linalg.vector_norm(x, dim=-1, keepdim=True)
    return x.to(dtype)


def _normal(gen, shape, dtype):
    return torch.randn(shape, generator=gen, device="cuda").to(dtype)


def _gates(gen, shape):
    alpha = 0.9 + 0.1 * torch.rand(shape, generator=gen, device="cuda")
    return alpha, torch.sigmoid(torch.randn(shape, generator=gen, device="cuda"))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return _prepare_prefill(case, gen) if case["kind"] == "prefill" else _prepare_generate(case, seed, gen)


def _prepare_prefill(case, gen):
    R, L, H, dk, dv, T = (case[n] for n in ("requests", "layers", "heads", "dk", "dv", "tokens"))
    dtype = _TORCH[case["dtype"]]
    cfg = P.make_config(R, L, H, dk, dv, 8, 1, case["dtype"], case["dtype"], R * 8)
    prompts = {}
    for r in range(R):
        for layer in range(L):
            prompts[r, layer] = (_unit(gen, (T, H, dk), dtype), _normal(gen, (T, H, dv), dtype), *_gates(gen, (T, H)))
    return {"case": case, "ctx": P.Onela(cfg), "prompts": prompts}


def _prepare_generate(case, seed, gen):
    R, L, H, Hv, dk, dv = (case[n] for n in ("requests", "layers", "heads", "v_heads", "dk", "dv"))
    dtype, widths = _TORCH[case["dtype"]], _widths(case)
    cfg = P.make_config(R, L, H, dk, dv, case["beam"], case["steps"], case["dtype"], case["out"], R * sum(widths),
                        P.FLAG_GTR_DELTA if case["delta"] else 0, 0 if Hv == H else Hv)
    s = {"case": case, "ctx": P.Onela(cfg), "widths": widths, "parents": [None], "tokens": [], "outs": []}
    # a state whose products with unit vectors are of the values' order
    s["S0"] = 0.3 * torch.randn((R, L, Hv, dv, dk), generator=gen, device="cuda")
    for W in widths:
        layers = []
        for _ in range(L):
            layers.append((_unit(gen, (R, W, H, dk), dtype), _normal(gen, (R, W, Hv, dv), dtype), *_gates(gen, (R, W, Hv)),
                           _unit(gen, (R, W, H, dk), dtype)))
        s["tokens"].append(layers)
        s["outs"].append(torch.empty((L, R, W, Hv, dv), dtype=_TORCH[case["out"]], device="cuda"))
    s["out_of"] = [[o[layer] for layer in range(L)] for o in s["outs"]]
    if case["parents"] == "select":
        # candidate log-probabilities of every call, and where selection leaves its results
        C, W_prev = case["codes"], 1
        s["logp"], s["codes"], s["scores"], s["parents"] = [], [], [torch.zeros((R, 1), device="cuda")], []
        for W in widths:
            s["logp"].append(torch.log_softmax(torch.randn((R, W_prev, C), generator=gen, device="cuda"), dim=-1))
            s["parents"].append(torch.empty((R, W), dtype=torch.int32, device="cuda"))
            s["codes"].append(torch.empty((R, W), dtype=torch.int32, device="cuda"))
            s["scores"].append(torch.empty((R, W), device="cuda"))
            W_prev = W
    else:
        law = inputs.Workload("", R, 1, 1, dk, dv, case["dtype"], 0, case["beam"], case["steps"], case["parents"], case["zipf"], seed)
        for t in range(1, case["steps"]):
            s["parents"].append(torch.stack([inputs.parents(law, r, t) for r in range(R)]).cuda())
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _generation(s)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _generation(s)
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------------
def _generation(s):
    case, ctx = s["case"], s["ctx"]
    R, select, fused = case["requests"], case["parents"] == "select", case["fused"]
    ctx.onela_init_shared_states(0, R, s["S0"])
    for t, W in enumerate(s["widths"]):
        if select:
            ctx.onela_select_beams(0, R, s["scores"][t], s["logp"][t], case["codes"], W, s["parents"][t], s["codes"][t], s["scores"][t + 1])
        ctx.onela_reorder_beams(0, R, s["parents"][t] if t else None, W)
        for layer, (k, v, alpha, beta, q) in enumerate(s["tokens"][t]):
            out = s["out_of"][t][layer]
            if fused:
                ctx.onela_append_decode_step(0, R, layer, k, v, alpha, beta, q, out)
            else:
                ctx.onela_append_records(0, R, layer, k, v, alpha, beta)
                ctx.onela_decode_step(0, R, layer, q, out)
    for r in range(R):
        ctx.onela_release_request(r)


def run(state):
    ctx = state["ctx"]
    if state["case"]["kind"] == "prefill":
        states = []
        for (r, layer), (k, v, alpha, beta) in state["prompts"].items():
            ctx.onela_prefill_shared_state(r, layer, k, v, alpha, beta)
            states.append(ctx.onela_export_shared_state(r, layer))
        return states
    if state["case"]["graph"]:
        state["graph"].replay()
    else:
        _generation(state)
    if state["case"]["parents"] == "select":
        return {"outs": state["outs"], "parents": state["parents"], "codes": state["codes"], "scores": state["scores"][1:]}
    return state["outs"]


# ---- what a pass cannot do without -------------------------------------------------------------------------------------
def _distinct(case, t):
    """Expected number of distinct records, per request, on the live chains of decode call t (their own included)."""
    W = case["beam"]
    p = [1.0 / i ** case["zipf"] for i in range(1, W + 1)] if case["parents"] == "zipf" else [1.0] * W
    total = sum(p)
    n = count = _widths(case)[t]
    for _ in range(t):
        n = sum(1.0 - (1.0 - x / total) ** n for x in p)
        count += n
    return count


def work(case):
    R, L, H, dk, dv = (case[n] for n in ("requests", "layers", "heads", "dk", "dv"))
    es = _ELEM[case["dtype"]]
    if case["kind"] == "prefill":
        rows = R * L * case["tokens"] * H                         # tokens read, states written; S k and the rank-one update
        return {"bytes": rows * ((dk + dv) * es + 8) + R * L * H * dk * dv * 4, "flops": rows * 4 * dk * dv}
    Hv, eo = case["v_heads"], _ELEM[case["out"]]
    state = R * L * Hv * dk * dv
    nbytes, flops = 2 * 4 * state, 0                              # admission: states read and stored
    slot = H * dk * es + Hv * (dv * es + 8)                       # one record slot of one layer, all heads
    for t, W in enumerate(_widths(case)):
        older = _distinct(case, t) - W
        # states, queries, the call's tokens (read, and stored as records), the older records, outputs, ancestry rows
        nbytes += 4 * state + R * L * W * (H * dk * es + 2 * slot + Hv * dv * eo) + R * L * older * slot + R * L * W * (t + 1) * 4
        flops += R * L * W * Hv * (2 * dk * dv + 2 * (t + 1) * (2 * dk + dv))
        if case["parents"] == "select":
            nbytes += R * (1 if t == 0 else _widths(case)[t - 1]) * case["codes"] * 4 + R * W * 12
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "prefill":
        return {"rel": 1e-5}                                      # fp32 sums
    if case["out"] == "bf16" or (case["delta"] and case["dtype"] == "bf16"):
        return {"rel": 5e-3}                                      # bf16 outputs, or replayed records rounded to bf16
    if case["dk"] == 32:
        return {"rel": 1e-5}                                      # fp32 throughout
    return {"rel": 1e-3}                                          # the product with the state has fp16 operands (2^-11 per element)
