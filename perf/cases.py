"""Performance cases of balanced-butterfly counting on one GPU.

Each case is one use of the library through its public entry points: one
resident graph counted again, a graph built from its edge list and counted, a
replayed plan over many resident graphs, a served group of requests built as
one union, and the per-vertex and per-edge counts. Graphs are drawn on the GPU
from a seed, with the shapes of the repository's own workloads (`synth/`) over
their range of sizes:

* ``uniform``    endpoints uniform on both sides, iid signs;
* ``ratings``    Chung-Lu, 20 edges per U and 100 per V vertex, gamma 2.1 / 1.9,
                 expected degree at most m / 1000, P(+) = 0.8;
* ``polarized``  Chung-Lu, 15 edges per U and 150 per V vertex, gamma 2.0 / 1.8,
                 expected degree at most m / 300, two camps;
* ``request``    a large served request: Chung-Lu, 13.6 edges per vertex with
                 one vertex in five on the U side, gamma 2.0 / 1.8, two camps;
* ``small``      a small served or batched graph: Chung-Lu, gamma 2.2 on both
                 sides, P(+) = 0.6.
"""
import math
import random

import numpy as np
import torch

import paper_2609_21848_gb300 as dbbc
from paper_2609_21848_gb300 import autotune

# name, gamma of U and V, degree cap as a share of m, sign model, tuning record
MODELS = {
    "uniform": dict(gammas=None, cap=None, camps=False, p=0.5, tuning=None),
    "ratings": dict(gammas=(2.1, 1.9), cap=1e-3, camps=False, p=0.8, tuning=None),
    "polarized": dict(gammas=(2.0, 1.8), cap=1 / 300, camps=True, p=0.9, tuning="polarized-20m-2m-300m"),
    "request": dict(gammas=(2.0, 1.8), cap=None, camps=True, p=0.9, tuning="batch-4096"),
    "small": dict(gammas=(2.2, 2.2), cap=None, camps=False, p=0.6, tuning="batch-4096"),
}


def _graph_case(name, kind, model, n_u, n_v, m, repeats=0.0, host=False):
    c = {"kind": kind, "model": model, "n_u": n_u, "n_v": n_v, "m": m, "repeats": repeats, "host": host}
    return {"name": name, **c} if name else c


def _group_case(name, kind, graphs, first):
    c = {"kind": kind, "model": "small", "graphs": graphs, "first": first}
    return {"name": name, **c} if name else c


def listed():
    return [
        # a dashboard or a service asks a small resident graph again: launches and one read-back
        _graph_case("count-resident-20k", "count", "uniform", 2_000, 3_000, 20_000),
        # the smallest whole request, its edge list already on the GPU
        _graph_case("step-uniform-20k", "step", "uniform", 2_000, 3_000, 20_000),
        # one small request with its arrays in ordinary host memory, ragged sizes
        _graph_case("step-host-151k", "step", "small", 9_973, 7_211, 151_313, host=True),
        # a rating log in which one row in seven repeats an earlier pair (the latest sign counts)
        _graph_case("step-repeats-2m", "step", "ratings", 100_003, 20_011, 2_000_003, repeats=0.15),
        # a mid-size resident graph counted again
        _graph_case("count-resident-1m", "count", "ratings", 50_021, 10_007, 1_000_003),
        # a large served request, already built, in its counting lane
        _graph_case("count-request-9m", "count", "request", 134_999, 539_993, 9_180_017),
        # the 20M-edge rating graph, built and counted
        _graph_case("step-ratings-20m", "step", "ratings", 1_000_000, 200_000, 20_000_000),
        # the largest single graph: the repository's default benchmark
        _graph_case("step-polarized-300m", "step", "polarized", 20_000_000, 2_000_000, 300_000_000),
        # the butterflies of every vertex (the input of tip decomposition)
        _graph_case("vertices-4m", "vertices", "ratings", 200_017, 40_009, 4_000_037),
        # the butterflies of every edge (the input of wing decomposition), queried on the GPU
        _graph_case("edges-20m", "edges", "ratings", 1_000_000, 200_000, 20_000_000),
        # many small resident graphs counted by one replayed plan
        _group_case("batch-1024", "batch", 1024, 0),
        # a group of small requests from pinned host memory: one union build, counts per request
        _group_case("union-host-200", "union", 200, 4_000),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "step", "step", "step", "vertices", "edges", "batch", "union"])
    if kind == "batch":
        return _group_case(None, kind, _log_uniform(rng, 16, 1024), rng.randrange(100_000))
    if kind == "union":
        return _group_case(None, kind, _log_uniform(rng, 2, 400), rng.randrange(100_000))
    model = rng.choice(["uniform", "ratings", "polarized", "request", "small"])
    # per-vertex and per-edge counts are asked of the graphs that are analysed, not of served ones
    if kind in ("vertices", "edges") and model in ("request", "small"):
        model = "ratings"
    hi = {"uniform": 4_000_000, "ratings": 20_000_000, "polarized": 100_000_000, "request": 20_000_000,
          "small": 200_000}[model]
    if kind in ("vertices", "edges"):
        hi = min(hi, 20_000_000)
    lo = {"request": 1_000_000, "small": 500}.get(model, 20_000)
    m = _log_uniform(rng, lo, hi)
    wide = math.exp(rng.uniform(-0.4, 0.4))  # the sides vary around the model's shape
    if model == "uniform":
        n_u, n_v = m / 10 * wide, m / 7 / wide
    elif model == "ratings":
        n_u, n_v = m / 20 * wide, m / 100 / wide
    elif model == "polarized":
        n_u, n_v = m / 15 * wide, m / 150 / wide
    elif model == "request":
        n_u, n_v = m / 13.6 / 5 * wide, m / 13.6 * 4 / 5 / wide
    else:
        n_u, n_v = _log_uniform(rng, 100, 20_000), _log_uniform(rng, 100, 20_000)
    n_u, n_v = max(100, int(n_u)), max(100, int(n_v))
    m = min(m, n_u * n_v // 2)
    repeats = rng.choice([0.0, 0.0, 0.02, 0.2]) if kind == "step" and m <= 20_000_000 else 0.0
    host = kind == "step" and m <= 5_000_000 and rng.random() < 0.4
    return _graph_case(None, kind, model, n_u, n_v, m, repeats, host)


# ---------------------------------------------------------------- inputs
def _side_weights(n, gamma, m, cap, dev):
    """Chung-Lu expected degrees min(cap, c (i+1)^(-1/(gamma-1))) summing to m, as
    whole multiples of 2^-20 (whole numbers add up the same in any order)."""
    raw = torch.arange(1, n + 1, dtype=torch.float64, device=dev).pow_(-1.0 / (gamma - 1.0))
    whole = (raw * 2.0**36).to(torch.int64)
    suffix = whole.sum() - whole.cumsum(0) + whole
    scale = (m - cap * torch.arange(n, dtype=torch.float64, device=dev)).clamp_(min=0) / suffix.double() * 2.0**36
    fits = scale * raw <= cap
    k = int(fits.to(torch.uint8).argmax()) if bool(fits.any()) else n - 1
    d = (scale[k] * raw).clamp_(max=cap)
    d[:k] = cap
    return (d * 2.0**20).to(torch.int64).clamp_(min=1)


def _endpoints(k, n, cum, total, gen, dev):
    if cum is None:
        return torch.randint(n, (k,), generator=gen, device=dev)
    return torch.searchsorted(cum, torch.randint(total, (k,), generator=gen, device=dev), right=True)


def _edges(model, n_u, n_v, m, gen, dev):
    """m distinct (u, v) pairs in random order with their signs (int32, int32, int8)."""
    p = MODELS[model]
    cums = [None, None]
    totals = [0, 0]
    if p["gammas"]:
        for i, (n, other) in enumerate(((n_u, n_v), (n_v, n_u))):
            cap = float(min(other, max(2.0, p["cap"] * m) if p["cap"] else 1_000_000))
            cums[i] = _side_weights(n, p["gammas"][i], float(m), cap, dev).cumsum_(0)
            totals[i] = int(cums[i][-1])
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    tries = 0
    while keys.numel() < m:
        k = int((m - keys.numel()) * (1.15 + 0.5 * tries)) + 64
        if tries >= 6:  # a nearly complete corner: fill up uniformly
            new = torch.randint(n_u * n_v, (k,), generator=gen, device=dev)
        else:
            new = _endpoints(k, n_u, cums[0], totals[0], gen, dev) * n_v
            new += _endpoints(k, n_v, cums[1], totals[1], gen, dev)
        keys = torch.unique(torch.cat([keys, new]))
        tries += 1
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=dev)[:m]]
    u = torch.randperm(n_u, generator=gen, device=dev).to(torch.int32)[keys // n_v]
    v = torch.randperm(n_v, generator=gen, device=dev).to(torch.int32)[keys % n_v]
    same = torch.rand(m, generator=gen, device=dev) < p["p"]
    if p["camps"]:
        cu = torch.rand(n_u, generator=gen, device=dev) < 0.5
        cv = torch.rand(n_v, generator=gen, device=dev) < 0.5
        same = same == (cu[u] == cv[v])
    return u, v, torch.where(same, 1, -1).to(torch.int8)


def _coo(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(dev).manual_seed(seed)
    m, extra = case["m"], int(case["m"] * case["repeats"])
    u, v, s = _edges(case["model"], case["n_u"], case["n_v"], m - extra, gen, dev)
    if extra:  # repeated pairs with signs of their own, anywhere in the log
        again = torch.randint(m - extra, (extra,), generator=gen, device=dev)
        sign = torch.where(torch.rand(extra, generator=gen, device=dev) < 0.5, 1, -1).to(torch.int8)
        order = torch.randperm(m, generator=gen, device=dev)
        u, v, s = (torch.cat(x)[order] for x in ((u, u[again]), (v, v[again]), (s, sign)))
    return u.contiguous(), v.contiguous(), s.contiguous()


def _group_sizes(case):
    """(n_u, n_v, m) of every graph of a group: the batched workload's ranges."""
    sizes = []
    for i in range(case["graphs"]):
        rng = random.Random(1_000_003 * case["first"] + i)
        n_u, n_v = _log_uniform(rng, 100, 20_000), _log_uniform(rng, 100, 20_000)
        sizes.append((n_u, n_v, min(_log_uniform(rng, 500, 200_000), n_u * n_v // 2)))
    return sizes


def _group(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(dev).manual_seed(seed)
    return [_edges("small", n_u, n_v, m, gen, dev) + (n_u, n_v) for n_u, n_v, m in _group_sizes(case)]


def prepare(case, seed):
    """The edge list, the built graph or the plan that a user's program holds."""
    dbbc.lib()
    autotune.apply_saved(MODELS[case["model"]]["tuning"])
    kind = case["kind"]
    if kind == "batch":
        graphs = [dbbc.dbbc_graph_from_coo(*g) for g in _group(case, seed)]
        return {"kind": kind, "plan": dbbc.dbbc_batch_create(graphs)}
    if kind == "union":
        graphs = _group(case, seed)
        u, v, s = (torch.cat([g[i] for g in graphs]).cpu().pin_memory() for i in range(3))
        offsets = np.concatenate([[0], np.cumsum([g[0].numel() for g in graphs])]).astype(np.int64)
        return {"kind": kind, "args": (u, v, s, offsets, np.array([g[3] for g in graphs], np.int32),
                                       np.array([g[4] for g in graphs], np.int32))}
    u, v, s = _coo(case, seed)
    if kind == "step":
        if case["host"]:
            u, v, s = (x.cpu().numpy() for x in (u, v, s))
        return {"kind": kind, "args": (u, v, s, case["n_u"], case["n_v"])}
    state = {"kind": kind, "graph": dbbc.dbbc_graph_from_coo(u, v, s, case["n_u"], case["n_v"])}
    if kind == "edges":
        state["query"] = (u, v)
    return state


def run(state):
    kind = state["kind"]
    if kind == "count":
        return dbbc.dbbc_count(state["graph"])
    if kind == "step":
        return dbbc.count_coo(*state["args"])
    if kind == "batch":
        return dbbc.dbbc_batch_count(state["plan"])
    if kind == "union":
        with dbbc.dbbc_graph_from_coo_multi(*state["args"]) as g:
            return dbbc.dbbc_count_components(g)
    if kind == "vertices":
        return dbbc.dbbc_count_vertices(state["graph"])
    balanced, unbalanced = dbbc.dbbc_count_edges(state["graph"], *state["query"])
    return balanced.view(torch.int64), unbalanced.view(torch.int64)


def work(case):
    """Bytes: edge lists are 9 bytes an edge, a resident graph 8 bytes an edge (its
    two rows' entries) and 12 bytes a vertex, every count 8 bytes. The wedges
    that are aggregated depend on the graph that is drawn and are not counted."""
    if case["kind"] in ("batch", "union"):
        sizes = _group_sizes(case)
        m, n = sum(x[2] for x in sizes), sum(x[0] + x[1] for x in sizes)
        return {"bytes": (8 * m + 12 * n if case["kind"] == "batch" else 9 * m) + 16 * len(sizes), "flops": 0}
    m, n = case["m"], case["n_u"] + case["n_v"]
    resident = 8 * m + 12 * n
    return {"bytes": {"count": resident + 16, "step": 9 * m + 16, "vertices": resident + 16 * n,
                      "edges": resident + 24 * m}[case["kind"]], "flops": 0}


def exact(case, seed):
    """The totals of a small graph from dense products: with S = A A^T and T = |A| |A|^T
    of the sign matrix A, a pair of U vertices has (T + S) / 2 symmetric and
    (T - S) / 2 asymmetric wedges."""
    if case["kind"] not in ("count", "step") or case["n_u"] > 4096 or case["n_u"] * case["n_v"] > 40_000_000:
        return None
    u, v, s = (x.cpu().numpy() for x in _coo(case, seed))
    dense = np.zeros((case["n_u"], case["n_v"]), np.float64)
    dense[u, v] = s  # of repeated pairs the last stays
    a = torch.from_numpy(dense).cuda()
    signed, plain = a @ a.T, a.abs() @ a.abs().T
    sym, asym = ((plain + signed) / 2).triu(1), ((plain - signed) / 2).triu(1)
    balanced = (sym * (sym - 1) + asym * (asym - 1)).sum() / 2
    return int(round(float(balanced))), int(round(float((sym * asym).sum())))
