"""Workloads of the BlockFFN layer as a decoding program runs them, for timing.

A case is a dict of plain values:

  kind    what the program does in one pass:
            "stack"    every FFN layer of a model on one chunk: residual h += FFN(bf16(h)) from layer
                       to layer, each layer's x is what the layer before left
            "chunks"   one layer call per chunk for chunks that do not depend on one another (x is
                       promised stable), over several copies of the weights
            "call"     a single layer through the Layer class, routing results included
            "pieces"   router, chunk union, expert stage and reuse ratio by their own entry points, on
                       one chunk per layer (a program that looks at the routing between them)
            "noalloc"  the expert stage of every layer for a caller that may not allocate, union
                       lists given
  graph   the pass was captured into a CUDA graph when the program started (a decoding loop) or is
          enqueued call by call
  router  the layer's own router gives the scores, or they are given
  d, E, d_e, L, layers   hidden size, experts, expert width, tokens of the chunk, layers (or calls)
  active, union   share of the experts one token activates, and of those any token of the chunk does

Shapes are those of the paper's model table and of the benchmark's configurations, the values those
of inputs.py: x ~ N(0, 1) with a component that neighbouring tokens share, weights with standard
deviation 1 / sqrt(fan in), gain ~ U(0.5, 1.5), scores |N(0, 1)| + 0.05 where active. Token sparsity
is 80 to 88 %, the union of a chunk about 30 % of the experts, as the paper reports for its models.
In a stack the down projections are scaled by 1/E, so that the running hidden state keeps its scale
and with it the sparsity.
"""
import math
from statistics import NormalDist

import torch

from paper_2507_08771_b200 import binding as B

_N = NormalDist()


def listed():
    def case(name, kind, d, E, d_e, L, layers, active, union, router=True, graph=True):
        return {"name": name, "kind": kind, "d": d, "E": E, "d_e": d_e, "L": L, "layers": layers,
                "active": active, "union": union, "router": router, "graph": graph}

    return [
        # The smallest call there is, one layer of the tiny configuration with everything a user of
        # the Layer class gets back: latency and launches.
        case("tiny_layer_call", "call", 256, 16, 64, 4, 1, 0.5, 0.94, graph=False),
        # The smallest model of the table on a short chunk, enqueued call by call: launches on the
        # host against short kernels.
        case("small_stack_5tok_calls", "stack", 768, 48, 64, 5, 16, 0.2, 0.30, graph=False),
        # Ordinary decoding, one token, 0.8B shape.
        case("decode_1tok_0p8b", "stack", 1536, 48, 128, 1, 32, 0.16, 0.16),
        # Verification of an 8-token draft, the 24-layer configuration with its routers on.
        case("verify_8tok_64e", "stack", 2048, 64, 128, 8, 24, 0.2, 0.30),
        # A ragged chunk on the 1.2B shape (width 1792, 56 experts).
        case("verify_13tok_1p2b", "stack", 1792, 56, 128, 13, 35, 0.18, 0.30),
        # A 32-token draft tree on the 2.8B shape: the largest.
        case("tree_32tok_2p8b", "stack", 2048, 128, 128, 32, 36, 0.1245, 0.3086),
        # The 24-layer configuration as the benchmark has it: scores known before the pass.
        case("scores_8tok_64e", "stack", 2048, 64, 128, 8, 24, 0.2, 0.30, router=False),
        # Independent chunks, scores given, 0.8B shape: the benchmark's headline configuration.
        case("chunks_8tok_0p8b", "chunks", 1536, 48, 128, 8, 46, 0.2, 0.30, router=False),
        # Independent chunks of 16 tokens with the router on.
        case("chunks_16tok_64e", "chunks", 2048, 64, 128, 16, 26, 0.2, 0.30),
        # Router, union, experts and reuse ratio one by one, call by call.
        case("pieces_24tok_64e", "pieces", 2048, 64, 128, 24, 8, 0.2, 0.30, graph=False),
        # A width and an expert width that are no multiples of the tensor-core tiles.
        case("off_grid_8tok", "stack", 1000, 40, 96, 8, 12, 0.2, 0.30),
        # The expert stage for a caller that may not allocate, call by call.
        case("noalloc_8tok_64e", "noalloc", 2048, 64, 128, 8, 8, 0.2, 0.30, router=False, graph=False),
    ]


def draw(rng):
    def spread(lo, hi):     # whole numbers, even over their logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("stack", "stack", "stack", "stack", "chunks", "chunks", "call", "pieces", "off_grid", "noalloc"))
    L, E, d_e = spread(1, 32), spread(16, 128), rng.choice((64, 128, 128, 128, 256))
    d = 64 * spread(4, 32)
    router = kind in ("call", "pieces", "off_grid") or (kind != "noalloc" and rng.random() < 0.7)
    graph = kind in ("stack", "chunks", "off_grid") and rng.random() < 0.75
    if kind == "off_grid":
        kind, d, d_e, E = "stack", 8 * spread(40, 250), 8 * rng.randrange(6, 22), spread(16, 64)
        layers = rng.randrange(2, 2 + max(3, min(10, 64 // L)))
    elif kind in ("noalloc", "pieces", "call"):
        if kind == "noalloc":
            d_e = min(d_e, 128)
            E = min(E, B.NOALLOC_SCRATCH_BYTES // (4 * L * d_e))
        layers = 1 if kind == "call" else rng.randrange(2, 9)
    else:
        layers = rng.randrange(12, 37)
    active = round(rng.uniform(0.12, 0.2), 3)
    union = active if L == 1 else round(max(active * 1.05, min(0.3 + rng.uniform(-0.05, 0.1), 1 - (1 - active) ** L)), 3)
    case = {"kind": kind, "d": d, "E": E, "d_e": d_e, "L": L, "layers": layers, "active": active,
            "union": union, "router": router, "graph": graph}
    while work(case)["bytes"] > 1.4e9:       # no more than the largest listed one
        case["layers"] = case["layers"] * 3 // 4
    return case


# ---- routing statistics ----------------------------------------------------------------
def _expected_union(active, rho, L, steps=200):
    """Share of the experts any of L tokens activates: logits sqrt(rho) c + sqrt(1 - rho) z over a
    threshold that one token passes with probability `active`."""
    t, none = _N.inv_cdf(1.0 - active), 0.0
    for i in range(steps):
        c = _N.inv_cdf((i + 0.5) / steps)
        none += _N.cdf((t - math.sqrt(rho) * c) / math.sqrt(1.0 - rho)) ** L
    return 1.0 - none / steps


def _rho(case):
    """The tokens' shared component that gives the case's union."""
    lo, hi = 0.0, 0.995
    if case["L"] == 1:
        return 0.0
    for _ in range(20):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if _expected_union(case["active"], mid, case["L"]) > case["union"] else (lo, mid)
    return 0.5 * (lo + hi)


def _union_size(case):
    return min(case["E"], max(1, round(case["union"] * case["E"])))


# ---- inputs ----------------------------------------------------------------------------
def _normal(gen, shape, std):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)


def _scores(gen, n, case):
    """n score matrices with a union of exactly the case's size, float32 [n][L][E]."""
    L, E, u = case["L"], case["E"], _union_size(case)
    p = min(1.0, case["active"] * E / u)
    members = torch.rand(n, E, device="cuda", generator=gen).argsort(1)[:, :u]
    hit = torch.rand(n, L, u, device="cuda", generator=gen) < p
    lucky = torch.randint(L, (n, 1, u), device="cuda", generator=gen)
    hit |= (torch.arange(L, device="cuda").view(1, L, 1) == lucky) & ~hit.any(1, keepdim=True)
    vals = torch.empty(n, L, u, device="cuda").normal_(generator=gen).abs_() + 0.05
    return torch.zeros(n, L, E, device="cuda").scatter_(2, members.view(n, 1, u).expand(n, L, u), vals * hit)


def _layer_weights(gen, case, residual):
    d, E, d_e = case["d"], case["E"], case["d_e"]
    t = {"U": _normal(gen, (E, d_e, d), d ** -0.5),
         "D": _normal(gen, (E, d, d_e), d_e ** -0.5 * (1.0 / E if residual else 1.0))}
    if case["router"]:
        t["W_r"] = _normal(gen, (E, d), d ** -0.5)
        t["gain"] = torch.empty(E, device="cuda").uniform_(0.5, 1.5, generator=gen)
        t["bias"] = torch.full((E,), -_N.inv_cdf(1.0 - case["active"]), device="cuda")
    return B.DeviceWeights(B.make_weights(t.get("W_r"), t.get("gain"), t.get("bias"), t["U"], t["D"]), t)


def _tokens(gen, n, case):
    """n chunks of hidden states, bf16 [n][L][d]."""
    rho, L, d = _rho(case), case["L"], case["d"]
    c = torch.empty(n, 1, d, device="cuda").normal_(generator=gen)
    z = torch.empty(n, L, d, device="cuda").normal_(generator=gen)
    return (math.sqrt(rho) * c + math.sqrt(1.0 - rho) * z).to(torch.bfloat16)


def prepare(case, seed):
    """Weights, handle, buffers and this pass's chunk(s); for a captured pass also its graph."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, L, d, E, n = case["kind"], case["L"], case["d"], case["E"], case["layers"]
    residual = kind in ("stack", "noalloc")
    s = {"case": case, "weights": [_layer_weights(gen, case, residual) for _ in range(n)],
         "x0": _tokens(gen, 1 if residual else n, case)}
    if not case["router"]:
        s["scores"] = [t.clone() for t in _scores(gen, n, case)]        # (each 16-byte aligned)
    if kind == "noalloc":
        s["cfg"] = B.Config(d, E, case["d_e"], L, 1e-6, 0, 0)
        mask = (torch.stack(s["scores"]) != 0).any(1)
        s["n_union"] = mask.sum(1, dtype=torch.int32)
        order = torch.where(mask, 0, E) + torch.arange(E, device="cuda")
        s["ids"] = torch.where(torch.arange(E, device="cuda") < s["n_union"].view(n, 1), order.argsort(1), -1).int()
    else:
        s["layer"] = B.Layer(d, E, case["d_e"], L_max=L)
    if kind == "pieces":
        s["scores"] = [torch.zeros(L, E, device="cuda") for _ in range(n)]
        s["tok_mask"] = torch.zeros(n, L, (E + 31) // 32, dtype=torch.int32, device="cuda")
        s["ids"] = torch.zeros(n, E, dtype=torch.int32, device="cuda")
        s["n_union"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["reuse"] = torch.zeros(2, dtype=torch.float64, device="cuda")
    if residual:
        s["h"] = torch.zeros(L, d, device="cuda")                                      # fp32 residual
        s["x"] = torch.zeros(2, L, d, dtype=torch.bfloat16, device="cuda")             # its rounding, alternating
    else:
        s["out"] = torch.zeros(n, L, d, device="cuda")
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _enqueue(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _enqueue(s)
    return s


# ---- one pass --------------------------------------------------------------------------
def _enqueue(s):
    case = s["case"]
    kind, L, router, weights = case["kind"], case["L"], case["router"], s["weights"]
    if kind == "chunks":
        h, stats = s["layer"].h, s["layer"].stats
        for i, w in enumerate(weights):
            if router:
                B.blockffn_layer_forward(h, w.struct, s["x0"][i], L, s["out"][i], None, stats, B.CALL_INDEPENDENT_X)
            else:
                B.blockffn_layer_forward_scores(h, w.struct, s["x0"][i], s["scores"][i], L, s["out"][i], None, stats,
                                                B.CALL_INDEPENDENT_X)
        return
    if kind == "pieces":
        h, stats = s["layer"].h, s["layer"].stats
        s["reuse"].zero_()
        for i, w in enumerate(weights):
            x, scores, ids, n_union = s["x0"][i], s["scores"][i], s["ids"][i], s["n_union"][i:i + 1]
            B.blockffn_router(h, w.struct, x, L, scores, s["tok_mask"][i])
            B.blockffn_chunk_union(h, scores, L, None, ids, n_union, stats)
            B.blockffn_expert_ffn(h, w.struct, x, scores, L, ids, n_union, s["out"][i])
            B.blockffn_reuse_ratio(h, scores, L, s["reuse"])
        return
    # a chunk through the layers: the residual starts as the chunk's hidden states; the weights, and
    # scores that are given, do not change while the pass runs
    flags = B.CALL_ACCUMULATE | B.CALL_INDEPENDENT
    s["h"].copy_(s["x0"][0])
    s["x"][0].copy_(s["x0"][0])
    for i, w in enumerate(weights):
        x, x_next = s["x"][i % 2], s["x"][(i + 1) % 2]
        if kind == "noalloc":
            B.blockffn_expert_ffn_noalloc(s["cfg"], w.struct, x, s["scores"][i], L, s["ids"][i], s["n_union"][i:i + 1],
                                          s["h"], x_next, flags)
        elif router:
            B.blockffn_layer_forward(s["layer"].h, w.struct, x, L, s["h"], x_next, s["layer"].stats, flags)
        else:
            B.blockffn_layer_forward_scores(s["layer"].h, w.struct, x, s["scores"][i], L, s["h"], x_next,
                                            s["layer"].stats, flags)


def run(s):
    case = s["case"]
    if case["kind"] == "call":
        r = s["layer"].forward(s["weights"][0], s["x0"][0])
        return {"out": r.out, "scores": r.scores, "tok_mask": r.tok_mask, "union_mask": r.union_mask,
                "union_ids": r.union_ids, "n_union": r.n_union}
    if case["graph"]:
        s["graph"].replay()
    else:
        _enqueue(s)
    if case["kind"] == "chunks":
        return s["out"]
    if case["kind"] == "pieces":
        return {k: s[k] for k in ("out", "scores", "tok_mask", "ids", "n_union", "reuse")}
    return {"h": s["h"], "x": s["x"][case["layers"] % 2]}


# ---- what a pass cannot do without ------------------------------------------------------
def work(case):
    L, d, E, d_e, n = case["L"], case["d"], case["E"], case["d_e"], case["layers"]
    if case["router"]:
        u = case["union"] * E
        per_layer = 2 * E * d + 8 * E                       # router weights, gain and bias
    else:
        u, per_layer = _union_size(case), 4 * L * E         # scores
    chunks = n if case["kind"] in ("chunks", "call", "pieces") else 1
    return {"bytes": n * (u * 4 * d_e * d + per_layer) + chunks * 6 * L * d,
            "flops": n * (4 * L * u * d_e * d + (2 * L * E * d if case["router"] else 0))}


def tolerance(case):
    """Against a float64 evaluation the calls of this file are off by: 1.7e-3 (largest element 1e-2)
    for a layer whose intermediate is rounded to bf16; up to 4e-3 (2e-2) for a stack, whose x is
    rounded between layers as well, so that a router in it sees slightly different logits; 3e-4 (8e-3,
    one bf16 step of x) for a stack whose intermediate stays float32. About four times that."""
    fp32 = case["kind"] == "noalloc" or case["d"] % 64 or case["d_e"] & (case["d_e"] - 1)
    if case["kind"] != "noalloc" and case["kind"] != "stack":
        return {"rel": 7e-3, "max": 0.05, "differ": 2e-3}
    if fp32:
        return {"rel": 1e-3, "max": 0.03}
    return {"rel": 1.2e-2, "max": 0.06}


def exact(case, seed):
    """The outputs in float64 (what is stored in bf16 between layers is rounded to it). Masks,
    lists and the ratio of two counts have no such value."""
    s = prepare(dict(case, graph=False), seed)
    kind, L, d = case["kind"], case["L"], case["d"]
    h, x, outs, all_scores = s["x0"][0].double(), s["x0"][0].double(), [], []
    for i, w in enumerate(s["weights"]):
        t = w.tensors
        if kind not in ("stack", "noalloc"):
            x = s["x0"][i].double()
        if case["router"]:
            a = torch.relu(x @ t["W_r"].double().T + t["bias"].double())
            sc = t["gain"].double() * a / (a.square().mean(1, keepdim=True) + 1e-6).sqrt()
        else:
            sc = s["scores"][i].double()
        out = torch.zeros(L, d, dtype=torch.float64, device="cuda")
        for e in (sc != 0).any(0).nonzero().flatten().tolist():
            z = x @ t["U"][e].double().T
            out += (sc[:, e:e + 1] * z * torch.sigmoid(z)) @ t["D"][e].double().T
        h = h + out
        x = h.to(torch.bfloat16).double()
        outs.append(out)
        all_scores.append(sc)
    if kind == "call":
        return {"out": outs[0], "scores": all_scores[0], "tok_mask": None, "union_mask": None,
                "union_ids": None, "n_union": None}
    if kind == "chunks":
        return torch.stack(outs)
    if kind == "pieces":
        return {"out": torch.stack(outs), "scores": torch.stack(all_scores), "tok_mask": None,
                "ids": None, "n_union": None, "reuse": None}
    return {"h": h, "x": x}
