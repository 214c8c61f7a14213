"""What a user of this library has it do, as cases that can be timed: graphs and
batches of the kinds the method is used on, taken through the public entry
points of the Python binding.

The graphs are the ones the tests and the benchmark use -- planted partitions
(small graphs with clear communities), R-MAT (social networks), Chung-Lu with
weights 1..4 (web graphs), grids with shortcuts (road networks), k-mer paths,
and an interaction stream -- drawn on the device from the seed alone.  Every
case runs the deterministic schedule, whose results are the same from run to
run; the asynchronous one gives another partition on every run.

Byte counts are the CSR entries (4-byte ID and weight) and offsets read once
and the outputs written once; the arithmetic is integer.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_11658_gb300 as L
from paper_2405_11658_gb300 import synth as S
from paper_2405_11658_gb300 import synth_device as D

DEV = "cuda"


def listed():
    return [
        # quality check of a small graph's labels where no context exists: two
        # short kernels and two reads, all latency
        {"name": "modularity_small", "op": "modularity_noalloc", "graph": "planted", "n": 10_000, "blocks": 20,
         "deg_in": 5.0, "deg_out": 4.75, "gamma": 1.0},
        # quality of a given labelling of a large graph: one pass over the CSR
        {"name": "modularity_rmat22", "op": "modularity", "graph": "rmat", "scale": 22, "ef": 16, "gamma": 1.0},
        # one small graph alone on the GPU: launches and synchronisations count
        {"name": "static_planted_1e4", "op": "static", "graph": "planted", "n": 10_000, "blocks": 20, "deg_in": 5.0,
         "deg_out": 4.75, "gamma": 1.0, "subsets": 8},
        # many small graphs of uneven size per call, Static and updates mixed
        {"name": "batch_64_small", "op": "batch", "graph": "planted", "count": 64, "n": 10_000, "n_min": 1_000,
         "gamma": 1.0, "subsets": 8, "frac": 1e-3},
        # social network, clustered from scratch
        {"name": "static_rmat22", "op": "static", "graph": "rmat", "scale": 22, "ef": 16, "gamma": 1.0, "subsets": 8},
        # web graph with weights, clustered from scratch: the largest case
        {"name": "static_chung_lu", "op": "static", "graph": "chung_lu", "n": 6_250_000, "m": 125_000_000,
         "gamma": 1.0, "subsets": 8},
        # road network, clustered from scratch: short rows, many iterations
        {"name": "static_grid_5000", "op": "static", "graph": "grid", "side": 5_000, "gamma": 1.0, "subsets": 8},
        # web graph after a batch of 1e-5 |E|, K and Sigma at hand (Dynamic Frontier)
        {"name": "df_chung_lu", "op": "update", "mode": "DF", "graph": "chung_lu", "n": 1_562_500, "m": 31_250_000,
         "frac": 1e-5, "gamma": 1.0, "subsets": 8},
        # k-mer graph after a batch of 1e-4 |E| (Delta-screening)
        {"name": "ds_kmer_1e7", "op": "update", "mode": "DS", "graph": "kmer", "n": 10_000_000, "frac": 1e-4,
         "gamma": 1.0, "subsets": 8},
        # social network after a batch of 1e-3 |E|, a resolution that needs the
        # wide scores, more colour classes (Naive-dynamic)
        {"name": "nd_rmat18_gamma", "op": "update", "mode": "ND", "graph": "rmat", "scale": 18, "ef": 16, "frac": 1e-3,
         "gamma": 1153434 / 1048576, "subsets": 32},
        # an interaction stream: four consecutive batches applied and followed by DF
        {"name": "stream_df", "op": "stream", "n": 285_000, "events": 1_957_500, "frac": 1e-4, "batches": 4,
         "gamma": 1.0, "subsets": 8},
        # a large batch (1e-2 |E|) applied to a web graph
        {"name": "apply_chung_lu", "op": "apply", "graph": "chung_lu", "n": 1_562_500, "m": 31_250_000, "frac": 1e-2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, kinds, most):
    """A graph family and its size, at most `most` CSR entries."""
    kind = rng.choice(kinds)
    if kind == "planted":
        n = _log_int(rng, 300, min(200_000, most // 10))
        return {"graph": kind, "n": n, "blocks": max(2, n // rng.randint(150, 900)),
                "deg_in": round(rng.uniform(4.0, 20.0), 2), "deg_out": round(rng.uniform(1.0, 6.0), 2)}
    if kind == "rmat":
        ef = rng.randint(8, 32)
        top = max(10, int(math.log2(most / (2 * ef))))
        return {"graph": kind, "scale": rng.randint(10, min(22, top)), "ef": ef}
    if kind == "chung_lu":
        m = _log_int(rng, 50_000, most // 2)
        return {"graph": kind, "n": max(2_000, int(m / rng.uniform(6.0, 20.0))), "m": m}
    if kind == "grid":
        return {"graph": kind, "side": _log_int(rng, 40, min(5_000, int(math.sqrt(most / 4))))}
    return {"graph": "kmer", "n": _log_int(rng, 5_000, min(20_000_000, most // 3))}


def draw(rng):
    op = rng.choice(["static", "static", "static", "update", "update", "update", "batch", "stream", "apply",
                     "modularity", "modularity_noalloc"])
    gamma = rng.choice([1.0, 1.0, 0.5, 0.75, 1.25, 1153434 / 1048576])
    subsets = rng.choice([8, 8, 8, 32])
    every = ["planted", "rmat", "chung_lu", "grid", "kmer"]
    if op == "static":
        return {"op": op, **_draw_graph(rng, every, 200_000_000), "gamma": gamma, "subsets": subsets}
    if op == "update":
        c = {"op": op, "mode": rng.choice(["DF", "DF", "DS", "ND"]), **_draw_graph(rng, every, 100_000_000)}
        return {**c, "frac": math.exp(rng.uniform(math.log(1e-6), math.log(1e-2))), "gamma": gamma, "subsets": subsets}
    if op == "batch":
        n = _log_int(rng, 500, 16_000)
        return {"op": op, "graph": "planted", "count": rng.randint(8, 96), "n": n, "n_min": max(50, n // 20),
                "gamma": gamma, "subsets": subsets, "frac": math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))}
    if op == "stream":
        n = _log_int(rng, 5_000, 285_000)
        return {"op": op, "n": n, "events": int(n * rng.uniform(5.0, 8.0)), "batches": rng.randint(1, 4),
                "frac": math.exp(rng.uniform(math.log(1e-5), math.log(1e-3))), "gamma": gamma, "subsets": subsets}
    if op == "apply":
        return {"op": op, **_draw_graph(rng, ["chung_lu", "grid", "kmer"], 100_000_000),
                "frac": math.exp(rng.uniform(math.log(1e-6), math.log(1e-1)))}
    if op == "modularity":
        return {"op": op, **_draw_graph(rng, every, 150_000_000), "gamma": gamma}
    c = _draw_graph(rng, ["planted", "rmat", "grid", "kmer"], 2_000_000)
    return {"op": op, **c, "gamma": gamma}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _unique_keys(u, v, n):
    """Sorted distinct keys a * n + b (a < b) of the pairs, loops dropped."""
    keep = u != v
    return torch.unique(torch.minimum(u, v)[keep] * n + torch.maximum(u, v)[keep])


def _planted(n, blocks, deg_in, deg_out, seed):
    g = _generator(seed)
    size = max(2, n // blocks)
    mi, mo = int(n * deg_in / 2), int(n * deg_out / 2)
    b = torch.randint(0, max(1, n // size), (mi,), generator=g, device=DEV) * size
    ui = (b + torch.randint(0, size, (mi,), generator=g, device=DEV)).clamp_(max=n - 1)
    vi = (b + torch.randint(0, size, (mi,), generator=g, device=DEV)).clamp_(max=n - 1)
    uo = torch.randint(0, n, (mo,), generator=g, device=DEV)
    vo = torch.randint(0, n, (mo,), generator=g, device=DEV)
    return n, _unique_keys(torch.cat([ui, uo]), torch.cat([vi, vo]), n)


def _rmat(scale, ef, seed, a=0.57, b=0.19, c=0.19):
    g = _generator(seed)
    n = 1 << scale
    m = ef * n
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device=DEV)
        u = (u << 1) | (r >= a + b)
        v = (v << 1) | (((r >= a) & (r < a + b)) | (r >= a + b + c))
    return n, _unique_keys(u, v, n)


def _grid(side, seed, remove=0.05, shortcuts=0.001):
    g = _generator(seed)
    n = side * side
    ids = torch.arange(n, device=DEV).reshape(side, side)
    u = torch.cat([ids[:, :-1].reshape(-1), ids[:-1, :].reshape(-1)])
    v = torch.cat([ids[:, 1:].reshape(-1), ids[1:, :].reshape(-1)])
    keep = torch.rand(u.numel(), generator=g, device=DEV) >= remove
    k = max(1, round(shortcuts * n))
    su = torch.randint(0, n, (k,), generator=g, device=DEV)
    sv = torch.randint(0, n, (k,), generator=g, device=DEV)
    return n, _unique_keys(torch.cat([u[keep], su]), torch.cat([v[keep], sv]), n)


def _kmer(n, seed, mean_path=64.0, degree=2.1):
    g = _generator(seed)
    perm = torch.randperm(n, generator=g, device=DEV)
    keep = torch.rand(n - 1, generator=g, device=DEV) >= 1.0 / mean_path
    u, v = perm[:-1][keep], perm[1:][keep]
    extra = max(0, int(degree * n / 2) - u.numel())
    eu = torch.randint(0, n, (extra,), generator=g, device=DEV)
    ev = torch.randint(0, n, (extra,), generator=g, device=DEV)
    return n, _unique_keys(torch.cat([u, eu]), torch.cat([v, ev]), n)


def _edges(case, seed):
    """(n, sorted edge keys, weights) of the case's graph."""
    kind = case["graph"]
    if kind == "chung_lu":
        keys, w = D.chung_lu_edges(case["n"], case["m"], 2.1, 1, 4, seed=seed, device=DEV)
        return case["n"], keys, w
    if kind == "planted":
        n, keys = _planted(case["n"], case["blocks"], case["deg_in"], case["deg_out"], seed)
    elif kind == "rmat":
        n, keys = _rmat(case["scale"], case["ef"], seed)
    elif kind == "grid":
        n, keys = _grid(case["side"], seed)
    else:
        n, keys = _kmer(case["n"], seed)
    return n, keys, torch.ones(keys.numel(), dtype=torch.int32, device=DEV)


def _graph(case, seed):
    n, keys, w = _edges(case, seed)
    if case.get("op") == "apply" and case["graph"] != "chung_lu":
        # the same number of edges from every seed, so that the new graph's
        # arrays have one size (Chung-Lu graphs do by themselves)
        m = int((1.8 if case["graph"] == "grid" else 1.0) * n)
        keep = torch.randperm(keys.numel(), generator=_generator(seed + 2), device=DEV)[:m].sort().values
        keys, w = keys[keep], w[keep]
    return L.Graph(*D.csr_from_edges(n, keys, w)), keys, w


def _batch(g, keys, w, frac, seed):
    """A random batch of frac |E| updates (80% insertions), at least two."""
    size = max(2, round(frac * keys.numel()))
    dels, ins = D.random_batch(g.n, keys, w, size, seed)
    return L.Edges(*(x.contiguous() for x in dels)), L.Edges(*(x.contiguous() for x in ins))


def _opts(case):
    return L.Opts(gamma=case.get("gamma", 1.0), det_subsets=case.get("subsets", 8))


def _labels(g, seed):
    """A labelling to score: about sqrt(n) groups of neighbouring IDs, a tenth
    of the vertices moved to another group."""
    gen = _generator(seed + 1)
    k = max(1, math.isqrt(g.n))
    lab = torch.arange(g.n, device=DEV) // max(1, g.n // k)
    move = torch.rand(g.n, generator=gen, device=DEV) < 0.1
    other = torch.randint(0, k, (g.n,), generator=gen, device=DEV)
    return torch.where(move, other, lab).to(torch.int32)


def prepare(case, seed):
    op = case["op"]
    if op == "stream":
        return _prepare_stream(case, seed)
    if op == "batch":
        return _prepare_batch(case, seed)
    g, keys, w = _graph(case, seed)
    st = {"op": op, "graph": g, "opts": _opts(case)}
    if op in ("modularity", "modularity_noalloc"):
        st["labels"] = _labels(g, seed)
        st["gamma"] = case["gamma"]
    if op == "modularity_noalloc":
        return st
    spare = 0
    if op in ("update", "apply"):
        st["dels"], st["ins"] = _batch(g, keys, w, case["frac"], seed + 1)
        spare = 2 * st["ins"].count + 1024
    del keys, w
    torch.cuda.empty_cache()
    st["ctx"] = L.Context(max_n=g.n, max_nnz=g.nnz + spare)
    if op == "update":
        # what the previous step of the user's program left: C, K and Sigma of
        # the old graph, and the new graph
        memb, _ = st["ctx"].static(g, st["opts"], want_q=False)
        memb, K, Sigma, _ = st["ctx"].update(g, memb, None, None, "ND", st["opts"], want_q=False)
        st["graph"] = st["ctx"].apply_batch(g, st["dels"], st["ins"])
        st["mode"] = case["mode"]
        st["prior"], st["K"], st["Sigma"] = memb, K, Sigma
    return st


def _prepare_stream(case, seed):
    src, dst = S.temporal_stream(case["n"], case["events"], seed=seed)
    (off, idx, w), rest = S.temporal_split(case["n"], src, dst)
    size = max(2, round(case["frac"] * case["events"]))
    batches = [L.Edges.from_numpy(b) for b in S.temporal_batches(rest, size, case["batches"])]
    g = L.Graph.from_numpy(off, idx, w)
    ctx = L.Context(max_n=g.n, max_nnz=g.nnz + 2 * size * len(batches) + 1024)
    opts = _opts(case)
    memb, _ = ctx.static(g, opts, want_q=False)
    memb, K, Sigma, _ = ctx.update(g, memb, None, None, "ND", opts, want_q=False)
    return {"op": "stream", "graph": g, "ctx": ctx, "opts": opts, "batches": batches, "prior": memb, "K": K,
            "Sigma": Sigma}


def _batch_sizes(case):
    """Vertices of each graph of the call: log-spaced, the largest first."""
    k, hi, lo = case["count"], case["n"], case["n_min"]
    return [int(round(hi * (lo / hi) ** (i / max(1, k - 1)))) for i in range(k)]


def _prepare_batch(case, seed):
    graphs, batches = [], []
    for i, n in enumerate(_batch_sizes(case)):
        g, keys, w = _graph({"graph": "planted", "n": n, "blocks": max(2, n // 500), "deg_in": 5.0, "deg_out": 4.75},
                            seed * 1009 + i)
        graphs.append(g)
        batches.append(_batch(g, keys, w, case["frac"], seed * 1009 + i))
    opts = _opts(case)
    total_n = sum(g.n for g in graphs)
    total_nnz = sum(g.nnz for g in graphs) + sum(2 * b[1].count for b in batches)
    handle = L.Batch(max_graphs=len(graphs), max_total_n=total_n, max_total_nnz=total_nnz)
    priors, _ = handle.run([{"graph": g} for g in graphs], opts)
    # every other graph is clustered from scratch, the rest updated by DF, DS
    # and ND in turn after a batch
    out = torch.empty(total_n, dtype=torch.int32, device=DEV)
    ctx = L.Context(max_n=max(g.n for g in graphs), max_nnz=max(g.nnz + 2 * b[1].count for g, b in zip(graphs, batches)))
    items, at = [], 0
    for i, (g, (dels, ins)) in enumerate(zip(graphs, batches)):
        it = {"graph": g, "out": out[at:at + g.n]}
        if i % 2:
            it.update(graph=ctx.apply_batch(g, dels, ins), mode=("DF", "DS", "ND")[i // 2 % 3], prior=priors[i],
                      dels=dels, ins=ins)
        items.append(it)
        at += g.n
    ctx.close()
    return {"op": "batch", "handle": handle, "items": items, "opts": opts, "out": out}


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    op = state["op"]
    if op == "modularity_noalloc":
        return L.modularity_noalloc(state["graph"], state["labels"], state["gamma"])
    if op == "batch":
        _, res = state["handle"].run(state["items"], state["opts"])
        return {"membership": state["out"], "q": np.array([r["q"] for r in res]),
                "status": np.array([r["status"] for r in res]), "passes": np.array([r["passes"] for r in res])}
    ctx = state["ctx"]
    if op == "modularity":
        return ctx.modularity(state["graph"], state["labels"], state["gamma"])
    if op == "static":
        memb, q = ctx.static(state["graph"], state["opts"])
        return {"membership": memb, "q": q}
    if op == "update":
        memb, K, Sigma, q = ctx.update(state["graph"], state["prior"], state["dels"], state["ins"], state["mode"],
                                       state["opts"], prior_K=state["K"], prior_Sigma=state["Sigma"])
        return {"membership": memb, "K": K, "Sigma": Sigma, "q": q}
    if op == "apply":
        g = ctx.apply_batch(state["graph"], state["dels"], state["ins"])
        return {"off": g.off, "idx": g.idx, "w": g.w}
    g, memb, K, Sigma = state["graph"], state["prior"], state["K"], state["Sigma"]
    qs = []
    for ins in state["batches"]:
        g = ctx.apply_batch(g, None, ins)
        memb, K, Sigma, q = ctx.update(g, memb, None, ins, "DF", state["opts"], prior_K=K, prior_Sigma=Sigma)
        qs.append(q)
    # the graph's entry arrays differ in size between streams; its row offsets
    # and weighted degrees are here, and whole graphs come from the apply case
    return {"off": g.off, "membership": memb, "K": K, "Sigma": Sigma, "q": np.array(qs)}


def _size(case):
    """(vertices, CSR entries) of the case's graph, as expected from its parameters."""
    kind = case.get("graph")
    if kind == "planted":
        return case["n"], case["n"] * (case["deg_in"] + case["deg_out"])
    if kind == "rmat":
        n = 1 << case["scale"]
        return n, 1.9 * case["ef"] * n
    if kind == "chung_lu":
        return case["n"], 2.0 * case["m"]
    if kind == "grid":
        return case["side"] ** 2, 3.8 * case["side"] ** 2
    return case["n"], 2.1 * case["n"]


def work(case):
    op = case["op"]
    if op == "batch":
        n = sum(_batch_sizes(case))
        return {"bytes": (8 + 4) * n + 8 * 9.75 * n, "flops": 0}
    if op == "stream":
        # each batch: the graph read and written by its application, read by
        # the update with C, K and Sigma, which are written again
        n, nnz = case["n"], 0.7 * case["events"]
        return {"bytes": case["batches"] * (3 * (8 * n + 8 * nnz) + 2 * 20 * n), "flops": 0}
    n, nnz = _size(case)
    csr = 8 * (n + 1) + 8 * nnz
    if op in ("modularity", "modularity_noalloc"):
        return {"bytes": csr + 4 * n, "flops": 0}
    if op == "static":
        return {"bytes": csr + 4 * n, "flops": 0}
    pairs = case["frac"] * nnz / 2
    if op == "update":
        return {"bytes": csr + 2 * 20 * n + 12 * pairs, "flops": 0}
    return {"bytes": 2 * csr + 12 * pairs + 16 * 0.8 * pairs, "flops": 0}


def exact(case, seed):
    """Eq. 1 from exact integer sums for the modularity cases.  The other cases
    return partitions of a greedy method, whose modularity has no value of its
    own, and whole numbers."""
    if not case["op"].startswith("modularity"):
        return None
    n, keys, w = _edges(case, seed)
    gen = _generator(seed + 1)
    k = max(1, math.isqrt(n))
    lab = torch.arange(n, device=DEV) // max(1, n // k)
    move = torch.rand(n, generator=gen, device=DEV) < 0.1
    lab = torch.where(move, torch.randint(0, k, (n,), generator=gen, device=DEV), lab)
    w = w.to(torch.int64)
    u, v = keys // n, keys % n
    two_m = 2 * int(w.sum())
    inside = 2 * int(w[lab[u] == lab[v]].sum())
    sigma = torch.zeros(n, dtype=torch.int64, device=DEV)
    sigma.index_add_(0, lab[u], w)
    sigma.index_add_(0, lab[v], w)
    squares = sum(int(s) ** 2 for s in sigma[sigma > 0].tolist())
    return float(torch.tensor(inside / two_m - case["gamma"] * squares / (two_m * two_m), dtype=torch.float64))
