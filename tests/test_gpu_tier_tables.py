"""DET on the multi-kernel path -- a context with a tier table of its own, which
the autotuner's candidates and the resident pass's fallbacks take as well --
at the edges of the degree tiers, with every update mode, both score widths and
other class counts than the default, against the oracle (exact)."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2405_11658_gb300 as L  # noqa: E402
from tests.test_gpu_team import check, tiers_graph  # noqa: E402


def tables():
    a = L.default_tiers()
    a[0]["threads"] = 128
    b = [t for t in L.default_tiers() if t["kind"] != "block"]   # hubs from the end of the group tiers on
    b[0]["threads"] = 128
    return {"default_shapes": a, "early_hubs": b}


@pytest.mark.parametrize("table", ["default_shapes", "early_hubs"])
@pytest.mark.parametrize("n,wmax,opts", [
    (2500, 1, {}),
    (2500, 1, {"det_subsets": 1}),
    (2500, 1 << 20, {"gamma": 1153434 / 1048576}),                       # 128-bit scores
    (30000, 3, {"det_subsets": 256}),                                    # rows beyond the block tier
    (30000, 1 << 12, {"gamma": 1153434 / 1048576, "det_subsets": 32}),   # 128-bit scores on them
])
def test_tier_edges_on_the_multi_kernel_path(table, n, wmax, opts):
    g = tiers_graph(n, wmax, 3)
    with L.Context(max_n=len(g[0]), max_nnz=len(g[1]) + 4096) as ctx:
        ctx.set_tiers(tables()[table])
        check(g, opts, ctx)
