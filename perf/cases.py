"""The calls a user of the library makes, over the range of sizes, types and options they are made with.

A case is one pass through a public entry point: a verify layer on device or on host buffers, a residual stack
of layers, or the oracle ranking of a tree.  Inputs follow the repository's synthetic recipe (unit-RMS hidden
states, router rows ~ N(0, 1/d) with a bias of -slope * ln(rank) that makes the routing heavy-tailed, expert
weights ~ N(0, 1/d)) but are drawn by the GPU's generator, because a state of several GB is made many times.
"""
import math
import random

import numpy as np
import torch

from paper_2602_16052_b200 import moespec
from paper_2602_16052_b200.synth import CONFIGS

_DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
_POLICIES = {"substitution": moespec.SUBSTITUTION, "truncation": moespec.TRUNCATION}
_SHORTLISTS = {"all": moespec.FROM_ALL, "union": moespec.FROM_UNION, "static": moespec.STATIC}


def _case(shape, M, B, name=None, entry="layer", dtype="bf16", out="fp32", policy="substitution", shortlist="all",
          renormalize=True, layers=1):
    """shape names a layer shape of the repository; M tree tokens, B kept experts."""
    c = {"shape": shape, "entry": entry, "M": M, "B": B, "dtype": dtype, "out": out, "policy": policy,
         "shortlist": shortlist, "renormalize": renormalize, "layers": layers}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest layer in use: launches and latency are what it costs
        _case("tiny", 15, 8, "tiny fp32 15 tokens", dtype="fp32"),
        # a decode step without a draft (or whose draft was refused): one token
        _case("olmoe", 1, 32, "one token", out="bf16"),
        # the usual draft tree at the usual budget
        _case("olmoe", 63, 32, "tree of 63, budget 32"),
        # the same call as a program with its activations in pinned host memory makes it
        _case("olmoe", 63, 32, "tree of 63 from host", entry="host"),
        # the other policy, candidate set and gating, in the 16-bit type that many checkpoints are stored in
        _case("olmoe", 127, 48, "tree of 127 fp16", dtype="fp16", out="fp16", policy="truncation", shortlist="union",
              renormalize=False),
        # a tree that is wider than one tile of tokens
        _case("olmoe", 255, 32, "tree of 255", out="bf16"),
        # many narrow experts behind a wide router
        _case("qwen3", 100, 64, "128 experts", out="bf16"),
        # few wide experts: a small tree against two GB of weights
        _case("mixtral", 15, 6, "wide experts", out="bf16"),
        # all MoE blocks of a 16-layer model, one pass per verification step, each layer's shortlist fixed beforehand
        # from earlier traffic (ranked by the router, near ties at the cut would differ after a few layers)
        _case("olmoe", 31, 32, "stack of 16", entry="stack", out="bf16", shortlist="static", layers=16),
        # a chunk of a prompt before the first draft, no budget: every expert, many tokens each
        _case("olmoe", 2048, 64, "prompt of 2048", out="bf16"),
        # the full-precision layer that 16-bit ones are checked against
        _case("olmoe", 63, 32, "tree of 63 fp32", dtype="fp32"),
        # which experts a budget should have kept for this tree
        _case("olmoe", 63, 32, "oracle ranking", entry="ranking"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["layer"] * 6 + ["host", "stack", "ranking"])
    shape = "olmoe" if entry != "layer" else rng.choice(["tiny", "olmoe", "olmoe", "olmoe", "qwen3", "mixtral"])
    N = CONFIGS[shape].n_experts
    top = {"layer": {"tiny": 127, "olmoe": 2048, "qwen3": 1024, "mixtral": 127}[shape], "host": 255, "stack": 127,
           "ranking": 127}[entry]
    M = _log_int(rng, 1 if entry != "ranking" else 15, top)
    B = rng.randint(max(2, N // 4), N) if entry != "ranking" else rng.randint(16, 32)
    dtype = "fp32" if shape == "tiny" else rng.choice(["bf16", "bf16", "fp16"])
    if entry == "layer" and shape == "olmoe" and M <= 127 and rng.random() < 0.25:
        dtype = "fp32"
    out = dtype if entry == "stack" else rng.choice([dtype, "fp32"])
    plain = entry in ("stack", "ranking")
    shortlist = {"stack": "static", "ranking": "all"}.get(entry) or rng.choice(["all", "all", "union", "static"])
    return _case(shape, M, B, entry=entry, dtype=dtype, out=out,
                 policy="substitution" if plain else rng.choice(["substitution", "substitution", "truncation"]),
                 shortlist=shortlist, renormalize=True if plain else rng.random() < 0.7,
                 layers=rng.randint(3, 16) if entry == "stack" else 1)


def _inputs(case, seed):
    """Hidden states and, per layer, router, bias, experts and the fixed ordering of a static shortlist."""
    cfg, dt = CONFIGS[case["shape"]], _DTYPES[case["dtype"]]
    dev = torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    normal = lambda *s: torch.empty(s, dtype=dt, device=dev).normal_(0.0, 1.0 / math.sqrt(cfg.d), generator=g)
    h = torch.randn(case["M"], cfg.d, device=dev, generator=g)
    h = (h / h.square().mean(1, keepdim=True).sqrt()).to(dt)
    layers = []
    for l in range(case["layers"]):
        order = list(range(cfg.n_experts))          # experts by popularity
        random.Random(seed * 1000 + l).shuffle(order)
        bias = torch.empty(cfg.n_experts)
        for r, e in enumerate(order):
            bias[e] = -cfg.slope * math.log(r + 1)
        layers.append({"router": normal(cfg.n_experts, cfg.d), "bias": bias.to(dev), "order": order,
                       "gate": normal(cfg.n_experts, cfg.f, cfg.d), "up": normal(cfg.n_experts, cfg.f, cfg.d),
                       "down": normal(cfg.n_experts, cfg.d, cfg.f)})
    return h, layers


def prepare(case, seed):
    cfg, M = CONFIGS[case["shape"]], case["M"]
    h, weights = _inputs(case, seed)
    layers = []
    for w in weights:
        layer = moespec.Layer(w["router"], w["bias"], w["gate"], w["up"], w["down"], max_M=M, max_k=cfg.k,
                              policy=_POLICIES[case["policy"]], shortlist=_SHORTLISTS[case["shortlist"]],
                              renormalize=case["renormalize"], residual=case["entry"] == "stack",
                              out_dtype=_DTYPES[case["out"]])
        if case["shortlist"] == "static":
            layer.set_static_ranking(w["order"])
        layers.append(layer)
    state = {"entry": case["entry"], "layer": layers[0], "k": cfg.k, "B": case["B"], "hidden": h,
             "out": torch.empty(M, cfg.d, dtype=_DTYPES[case["out"]], device=h.device)}
    if case["entry"] == "stack":
        state["stack"] = moespec.Stack(layers)
    if case["entry"] == "host":
        state["hidden"] = h.cpu().pin_memory()
        state["out"] = torch.empty(M, cfg.d, dtype=_DTYPES[case["out"]]).pin_memory()
    return state


def run(state):
    k, B, h, out = state["k"], state["B"], state["hidden"], state["out"]
    if state["entry"] == "layer":
        return state["layer"].verify_layer(h, k, B, out=out)
    if state["entry"] == "host":
        return state["layer"].verify_layer_host(h, k, B, out)
    if state["entry"] == "stack":
        return state["stack"].verify_stack(h, k, B, out=out)
    order, objective, gold = state["layer"].oracle_ranking(h, k, B, out_star=out)
    return {"order": np.asarray(order), "objective": objective, "gold": gold, "out_star": out}


def _routed(case):
    """(experts with rows, rows) of one layer, from logits of the distribution the inputs give."""
    cfg, M = CONFIGS[case["shape"]], case["M"]
    z = np.random.RandomState(7).randn(M, cfg.n_experts) - cfg.slope * np.log(np.arange(1, cfg.n_experts + 1))
    natural = np.argsort(-z, axis=1)[:, :cfg.k]
    if case["entry"] == "ranking":
        return len(np.unique(natural)), M * cfg.k
    p = np.exp(z)
    score = (p / p.sum(1, keepdims=True)).sum(0)
    if case["shortlist"] == "union":
        score[np.setdiff1d(np.arange(cfg.n_experts), natural)] = -1.0
    kept = np.arange(case["B"]) if case["shortlist"] == "static" else np.argsort(-score)[:case["B"]]
    kept = kept[score[kept] >= 0]
    if case["policy"] == "truncation":
        rows = natural[np.isin(natural, kept)]
    else:
        rows = kept[np.argsort(-z[:, kept], axis=1)[:, :cfg.k]].ravel()
    return len(np.unique(rows)), rows.size


def work(case):
    cfg, M = CONFIGS[case["shape"]], case["M"]
    size, out_size = (torch.empty(0, dtype=_DTYPES[case[t]]).element_size() for t in ("dtype", "out"))
    active, rows = _routed(case)
    layer = (active * 3 * cfg.f + cfg.n_experts) * cfg.d * size
    return {"bytes": case["layers"] * layer + M * cfg.d * (size + out_size),
            "flops": case["layers"] * (rows * 6 * cfg.d * cfg.f + 2 * M * cfg.n_experts * cfg.d)}


def tolerance(case):
    if case["entry"] == "ranking":
        return {"rel": 1.5e-2, "max": 0.15, "differ": 0.2}
    if case["entry"] == "stack":
        return {"rel": 0.16, "max": 0.6}      # a rounding that flips a near tie of two experts grows from layer to layer
    if case["dtype"] == "fp32":
        return {"rel": 2e-6, "max": 2e-5}
    return {"rel": 1.2e-2, "max": 0.1} if case["dtype"] == "bf16" else {"rel": 1.5e-3, "max": 1.5e-2}


def _assign(case, cfg, z, order):
    """Kept experts [M, k] (-1: none) and their mixing weights, from fp64 logits."""
    p = torch.softmax(z, 1)
    natural = z.topk(cfg.k, 1).indices
    if case["entry"] == "ranking":
        kept = torch.ones(cfg.n_experts, dtype=torch.bool, device=z.device)
    else:
        if case["shortlist"] == "static":
            best = torch.tensor(order[:case["B"]], device=z.device)
        else:
            score = p.sum(0)
            n = min(case["B"], cfg.n_experts)
            if case["shortlist"] == "union":
                seen = torch.zeros_like(score, dtype=torch.bool)
                seen[natural.unique()] = True
                score = torch.where(seen, score, torch.full_like(score, -1.0))
                n = min(n, int(seen.sum()))
            best = score.topk(n).indices
        kept = torch.zeros(cfg.n_experts, dtype=torch.bool, device=z.device)
        kept[best] = True
    if case["policy"] == "truncation" and case["entry"] != "ranking":
        idx = torch.where(kept[natural], natural, torch.full_like(natural, -1))
        total = p.gather(1, natural).sum(1, keepdim=True)
    else:
        idx = torch.where(kept, z, torch.full_like(z, -math.inf)).topk(min(cfg.k, int(kept.sum())), 1).indices
        total = p.gather(1, idx).sum(1, keepdim=True)
    w = p.gather(1, idx.clamp(min=0)) / (total if case["renormalize"] else 1.0)
    return idx, torch.where(idx >= 0, w, torch.zeros_like(w))


def _terms(case, cfg, x, w):
    """Weighted expert outputs [M, k, d] in 64 bits."""
    x = x.double()
    idx, wgt = _assign(case, cfg, x @ w["router"].double().T + w["bias"].double(), w["order"])
    terms = torch.zeros(idx.shape + (cfg.d,), dtype=torch.float64, device=x.device)
    for e in idx[idx >= 0].unique().tolist():
        t, s = (idx == e).nonzero(as_tuple=True)
        hid = torch.nn.functional.silu(x[t] @ w["gate"][e].double().T) * (x[t] @ w["up"][e].double().T)
        terms[t, s] = wgt[t, s, None] * (hid @ w["down"][e].double().T)
    return idx, terms


def exact(case, seed):
    cfg = CONFIGS[case["shape"]]
    x, layers = _inputs(case, seed)
    if case["entry"] == "stack":
        for w in layers:          # the stream between layers is held in the layers' type by definition
            x = (x.double() + _terms(case, cfg, x, w)[1].sum(1)).to(x.dtype)
        return x.double()
    idx, terms = _terms(case, cfg, x, layers[0])
    if case["entry"] != "ranking":
        return terms.sum(1)
    # greedy: each step adds the expert that leaves the smallest squared distance to the unpruned output
    gram = terms @ terms.transpose(1, 2)
    left = torch.ones_like(idx, dtype=torch.float64)          # terms not yet covered
    gold, objective = gram.sum(), []
    member = torch.nn.functional.one_hot(idx, cfg.n_experts).double()
    taken = torch.zeros(cfg.n_experts, dtype=torch.bool, device=x.device)
    err = gold
    for _ in range(case["B"]):
        gain = 2.0 * (gram * left[:, None, :]).sum(2) - gram.diagonal(dim1=1, dim2=2)
        total = torch.einsum("tk,tkn->n", gain, member).masked_fill(taken, -math.inf)
        pick = int(total.argmax())
        err = err - total[pick]
        objective.append(err)
        taken[pick] = True
        left = left * (1.0 - member[:, :, pick])
    return {"order": None, "objective": torch.stack(objective).cpu().numpy(), "gold": float(gold),
            "out_star": terms.sum(1)}
