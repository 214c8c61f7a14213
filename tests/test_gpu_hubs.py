"""Levels with more hub rows (more than 8192 candidates) than one colour class
or the workspace was first sized for.  All arithmetic is integer, so every
comparison is exact."""
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


def circulant(n, half):
    """Vertex i joined to i - half .. i + half (on the device), weights 1..3."""
    d = torch.cat([torch.arange(-half, 0), torch.arange(1, half + 1)]).cuda()
    i = torch.arange(n, device="cuda")[:, None]
    idx = torch.sort((i + d) % n, dim=1)[0]
    w = 1 + (i + idx) % 3
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * (2 * half)
    return L.Graph(off, idx.reshape(-1).to(torch.int32), w.reshape(-1).to(torch.int32))


def test_more_hubs_in_a_class_than_the_block_keeps_bits_for():
    # 16400 rows of 8194 candidates in one class (16384 bits a block): a batch
    # holds the tables of all of them, a context with its own tier table takes
    # the multi-kernel path
    g = circulant(16400, 4097)
    opts = L.Opts(det_subsets=1, max_passes=1, max_iters=2)
    tiers = L.default_tiers()
    tiers[0]["threads"] = 128
    with L.Context(max_n=g.n, max_nnz=g.nnz) as ctx:
        ctx.set_tiers(tiers)
        memb, q = ctx.static(g, opts)
        st = ctx.stats()
    torch.cuda.empty_cache()
    with L.Batch(max_graphs=1, max_total_n=g.n, max_total_nnz=g.nnz) as batch:
        outs, res = batch.run([{"graph": g}], opts)
    r = res[0]
    assert r["status"] == 0
    assert r["iters"] == st["iters"] and r["moves"] == st["moves"] and r["refine_moves"] == st["refine_moves"]
    assert torch.equal(outs[0], memb) and r["q"] == q


def test_hub_tables_beyond_the_scratch():
    # 600 centres over 8400 of 10000 leaves, one class: 600 tables of 20480
    # slots need more than the context's 1.0e7 scratch slots, so the level
    # falls back to the multi-kernel path; the batch has room for them
    rng = np.random.default_rng(1)
    leaves = np.concatenate([rng.choice(10000, 8400, replace=False) for _ in range(600)])
    centres = np.repeat(10000 + np.arange(600), 8400)
    g = S.edges_to_csr(10600, leaves, centres, rng.integers(1, 4, len(leaves)))
    opts = dict(det_subsets=1)
    ref = O.static(*g, O.LeidenOpts(**opts))
    G = L.Graph.from_numpy(*g)
    with L.Context(max_n=G.n, max_nnz=G.nnz) as ctx:
        memb, q = ctx.static(G, L.Opts(**opts))
        st = ctx.stats()
        # launches a further iteration takes: none on the resident pass
        launches = []
        for iters in (1, 2):
            n0 = L.kernel_launches()
            ctx.static(G, L.Opts(max_passes=1, max_iters=iters, tol=0.0, **opts))
            launches.append(L.kernel_launches() - n0)
            assert ctx.stats()["iters"] == [iters]
        assert launches[1] > launches[0]
    assert np.array_equal(memb.cpu().numpy(), ref.membership) and q == ref.q
    k = ref.stats["passes"]
    for name in ("iters", "nv", "nnz", "moves", "refine_moves"):
        assert st[name][:k] == ref.stats[name], name
    with L.Batch(max_graphs=1, max_total_n=G.n, max_total_nnz=G.nnz) as batch:
        outs, res = batch.run([{"graph": G}], L.Opts(**opts))
    assert res[0]["status"] == 0 and np.array_equal(outs[0].cpu().numpy(), ref.membership) and res[0]["q"] == ref.q
