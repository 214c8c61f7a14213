"""Per-pass times of a run's statistics: every pass that aggregates has the time
of its aggregation in t_agg_ms, and t_pass_ms covers the pass's phases, whether
the aggregation is part of the resident pass or follows it in launches of its
own (the uniform policy; levels beyond the resident pass's table)."""
from __future__ import annotations

import pytest

from paper_2405_11658_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2405_11658_gb300 as L  # noqa: E402


@pytest.mark.parametrize("name", ["tiered", "uniform", "large"])
def test_pass_times_include_the_aggregation(name):
    g = S.rmat(18, 16, seed=2) if name == "large" else S.rmat(13, 16, seed=2)   # large: 7e6 entries
    with L.Context(max_n=len(g[0]), max_nnz=len(g[1])) as ctx:
        ctx.set_agg_policy(name == "uniform")
        G = L.Graph.from_numpy(*g)
        ctx.static(G)
        ctx.static(G)
        st = ctx.stats()
    k = st["passes"]
    assert k >= 2
    for p in range(k - 1):   # every pass but the last aggregates
        assert st["t_agg_ms"][p] > 0.0, p
        # the phases are on the device clock, the pass on the host's: 2% for
        # their rates, 10 us for the clock's resolution
        assert st["t_pass_ms"][p] * 1.02 + 0.01 >= st["t_move_ms"][p] + st["t_refine_ms"][p] + st["t_agg_ms"][p], p
    assert sum(st["t_pass_ms"][:k]) <= st["total_ms"]
