"""The resident-block pass (csrc/team.cuh) at the edges of its degree tiers, of
its proposal lists and of its barrier kinds, against the oracle.  All
arithmetic is integer and the schedule is deterministic, so every comparison
is exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
from paper_2405_11658_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2405_11658_gb300 as L  # noqa: E402

# one below, at and above the last degree of every tier
EDGES = (7, 8, 9, 15, 16, 17, 31, 32, 33, 127, 128, 129, 255, 256, 257, 2047, 2048, 2049)
HUBS = (8191, 8192, 8193, 10240, 10241, 20000)


def tiers_graph(n, wmax, seed):
    """A random graph with, for every degree of EDGES (and, where it has the
    vertices, of HUBS), three vertices of about that degree: star centres over
    random leaves."""
    rng = np.random.default_rng(seed)
    us, vs = [rng.integers(0, n, 3 * n)], [rng.integers(0, n, 3 * n)]
    centre = n
    for d in EDGES + (HUBS if n >= HUBS[-1] else ()):
        for _ in range(3):
            us.append(np.full(d, centre))
            vs.append(rng.choice(n, d, replace=False))
            centre += 1
    u, v = np.concatenate(us), np.concatenate(vs)
    return S.edges_to_csr(centre, u, v, rng.integers(1, wmax + 1, len(u)))


def check(g, opts, ctx, batch_seed=5):
    oo = O.LeidenOpts(**opts)
    lo = L.Opts(**opts)
    ref = O.static(*g, oo)
    G = L.Graph.from_numpy(*g)
    memb, q = ctx.static(G, lo)
    st = ctx.stats()
    assert np.array_equal(memb.cpu().numpy(), ref.membership) and q == ref.q
    k = ref.stats["passes"]
    assert st["passes"] == k
    for name in ("iters", "nv", "nnz", "moves", "refine_moves"):
        assert st[name][:k] == ref.stats[name], name
    dels, ins = S.random_batch(*g, 30, seed=batch_seed)
    gt = O.apply_batch(*g, dels, ins)
    Gt = ctx.apply_batch(G, L.Edges.from_numpy(dels), L.Edges.from_numpy(ins))
    for mode in ("DF", "DS", "ND"):
        r = O.update(*gt, ref.membership, None, None, dels, ins, mode, oo)
        m2, K2, S2, q2 = ctx.update(Gt, memb, L.Edges.from_numpy(dels), L.Edges.from_numpy(ins), mode, lo)
        assert np.array_equal(m2.cpu().numpy(), r.membership) and q2 == r.q, mode


@pytest.mark.parametrize("n,wmax,opts", [
    (2500, 1, {}),                                    # one cluster
    (2500, 1, {"det_subsets": 1}),                    # whole level per sub-sweep: block lists overflow
    (2500, 1 << 20, {"gamma": 1153434 / 1048576}),    # 128-bit scores
    (30000, 3, {"det_subsets": 256}),                 # the whole grid, almost empty classes
    (30000, 1, {"det_subsets": 2}),
])
def test_tier_edges(n, wmax, opts):
    g = tiers_graph(n, wmax, 3)
    with L.Context(max_n=len(g[0]), max_nnz=len(g[1]) + 4096) as ctx:
        check(g, opts, ctx)


@pytest.mark.parametrize("n", [1, 2, 3, 40, 130, 600])
def test_smallest_levels(n):
    # a single block, then clusters of a few
    g = S.erdos_renyi(n, min(1.0, 12.0 / n), n, wmax=3) if n > 1 else S.edges_to_csr(1, [], [])
    with L.Context(max_n=len(g[0]), max_nnz=len(g[1]) + 64) as ctx:
        ref = O.static(*g, O.LeidenOpts())
        memb, q = ctx.static(L.Graph.from_numpy(*g), L.Opts())
        assert np.array_equal(memb.cpu().numpy(), ref.membership) and q == ref.q


def test_same_result_as_the_multi_kernel_path():
    # a context with a tier table of its own runs one launch per tier instead
    g = S.chung_lu(40000, 300000, 2.1, 1, 4, seed=9)
    tiers = L.default_tiers()
    tiers[0]["threads"] = 128
    with L.Context(max_n=len(g[0]), max_nnz=len(g[1])) as ctx:
        G = L.Graph.from_numpy(*g)
        a, qa = ctx.static(G)
        sa = ctx.stats()
        la = L.kernel_launches()
        ctx.static(G)
        la = L.kernel_launches() - la
        ctx.set_tiers(tiers)
        lb = L.kernel_launches()
        b, qb = ctx.static(G)
        lb = L.kernel_launches() - lb
        sb = ctx.stats()
    assert torch.equal(a, b) and qa == qb
    for name in ("passes", "iters", "nv", "nnz", "moves", "refine_moves", "move_scanned_entries",
                 "move_scanned_vertices", "move_bytes"):
        assert sa[name] == sb[name], name
    assert la < lb / 5   # the two paths really differ


@pytest.mark.parametrize("count", [1, 7, 20, 45, 90, 160])
def test_batch_cluster_sizes(count):
    # clusters of 16, 8, 4, 2 blocks for the largest graphs, single blocks for
    # the others: each graph as on a context
    sizes = [int(20 + 6000 * 0.96 ** k) for k in range(count)]
    graphs = [S.erdos_renyi(n, 8 / n, n, wmax=3) if n < 400 else S.planted_partition(n, max(2, n // 300), 0.02, 5 / n, n)
              for n in sizes]
    with L.Context(max_n=8192, max_nnz=1 << 19) as ctx, \
            L.Batch(max_graphs=count, max_total_n=sum(len(g[0]) for g in graphs),
                    max_total_nnz=sum(len(g[1]) for g in graphs)) as batch:
        gs = [L.Graph.from_numpy(*g) for g in graphs]
        outs, res = batch.run([{"graph": g} for g in gs])
        for g, out, r in zip(gs, outs, res):
            memb, q = ctx.static(g)
            st = ctx.stats()
            assert r["status"] == 0 and torch.equal(out, memb) and r["q"] == q
            for name in ("passes", "iters", "nv", "nnz", "moves", "refine_moves", "changed0"):
                assert r[name] == st[name], name


@pytest.mark.parametrize("opts", [{"det_subsets": 1}, {"gamma": 1153434 / 1048576, "det_subsets": 1}, {}])
def test_batch_with_hub_rows(opts):
    # more than 8192 distinct candidates: the hub tables of the batch workspace
    g = tiers_graph(30000, 1 << 12, 4)
    ref = O.static(*g, O.LeidenOpts(**opts))
    with L.Batch(max_graphs=3, max_total_n=3 * len(g[0]), max_total_nnz=3 * len(g[1])) as batch:
        G = L.Graph.from_numpy(*g)
        outs, res = batch.run([{"graph": G}] * 3, L.Opts(**opts))
        for out, r in zip(outs, res):
            assert r["status"] == 0 and np.array_equal(out.cpu().numpy(), ref.membership) and r["q"] == ref.q


@pytest.mark.parametrize("size", [2, 4, 5, 8, 9, 16, 17, 23, 24, 45, 46, 60])
def test_aggregation_tier_edges(size):
    # cliques joined in a ring: communities of total degree size * (size - 1)
    # + 2, on both sides of the aggregation tiers' limits 16, 64, 256, 512 and
    # 2048 (a context with a tier table of its own aggregates through them)
    a, b = np.triu_indices(size, 1)
    count = 300
    base = np.arange(count) * size
    u, v = (base[:, None] + a).ravel(), (base[:, None] + b).ravel()
    g = S.edges_to_csr(count * size, np.concatenate([u, base + size - 1]), np.concatenate([v, np.roll(base, -1)]),
                       np.random.default_rng(size).integers(1, 1 << (22 if size < 40 else 18), len(u) + count))  # 2m < 2^40
    ref = O.static(*g, O.LeidenOpts())
    tiers = L.default_tiers()
    tiers[0]["threads"] = 128
    with L.Context(max_n=count * size, max_nnz=len(g[1])) as ctx:
        ctx.set_tiers(tiers)
        memb, q = ctx.static(L.Graph.from_numpy(*g))
        st = ctx.stats()
    assert np.array_equal(memb.cpu().numpy(), ref.membership) and q == ref.q
    for name in ("iters", "nv", "nnz", "moves", "refine_moves"):
        assert st[name][:ref.stats["passes"]] == ref.stats[name], name
