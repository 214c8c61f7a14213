"""Every shape of the batch kernel (tests/batch_shapes.py; which batch gets which
is checked in test_host_launches.py) gives each graph the result of a context.
All arithmetic is integer, so every comparison is exact."""
from __future__ import annotations

import pytest

from paper_2405_11658_gb300 import synth as S

from tests.batch_shapes import SHAPES

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2405_11658_gb300 as L  # noqa: E402


def graph(size, seed):
    """About `size` vertices + entries, nine entries a vertex, communities of 100."""
    n = size // 10
    g = S.planted_partition(n, max(2, n // 100), min(1.0, 6.0 / 100 if n >= 200 else 12.0 / n), 3.0 / n, seed)
    # near enough to be on the same side of every line of the rule (6144 the lowest)
    assert size < 6144 or abs(len(g[0]) + len(g[1]) - size) < 0.07 * size, (size, len(g[0]), len(g[1]))
    return L.Graph.from_numpy(*g)


@pytest.mark.parametrize("opts", [{}, {"gamma": 1153434 / 1048576, "det_subsets": 32}])
@pytest.mark.parametrize("name", list(SHAPES))
def test_every_shape_gives_the_results_of_a_context(name, opts):
    sizes = SHAPES[name][0]
    made = {s: [graph(s, k) for k in range(min(3, sizes.count(s)))] for s in set(sizes)}
    gs = [made[s][k % len(made[s])] for k, s in enumerate(sizes)]
    o = L.Opts(**opts)
    want = {}
    with L.Context(max_n=max(g.n for g in gs), max_nnz=max(g.nnz for g in gs)) as ctx:
        for g in {id(g): g for g in gs}.values():
            memb, q = ctx.static(g, o)
            want[id(g)] = (memb, q, ctx.stats())
    with L.Batch(max_graphs=len(gs), max_total_n=sum(g.n for g in gs), max_total_nnz=sum(g.nnz for g in gs)) as batch:
        outs, res = batch.run([{"graph": g} for g in gs], o)
    for g, out, r in zip(gs, outs, res):
        memb, q, st = want[id(g)]
        assert r["status"] == 0 and torch.equal(out, memb) and r["q"] == q
        for field in ("passes", "iters", "nv", "nnz", "moves", "refine_moves", "changed0"):
            assert r[field] == st[field], field
