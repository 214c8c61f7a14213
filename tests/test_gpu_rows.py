"""The pass that checks a CSR and sums its rows or takes the terms of Eq. 1
(rows_k in csrc/misc.cu), where its pieces can go wrong: rows longer than a
piece, runs of empty rows, pieces that end with a row, and malformed inputs.
Integer sums, so every comparison is exact."""
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


def star(leaves, n):
    return S.edges_to_csr(n, np.zeros(leaves, np.int64), np.arange(1, leaves + 1))


def path(n):
    return S.edges_to_csr(n, np.arange(n - 1), np.arange(1, n))


GRAPHS = {
    "one_vertex": lambda: path(1),
    "two_vertices": lambda: path(2),
    "no_entries": lambda: S.edges_to_csr(1000, [], []),
    # items (rows + entries) of 1, 2 and 3 pieces of 256, one less and one more
    **{f"path_{n}": (lambda n=n: path(n)) for n in (85, 86, 87, 170, 171, 172, 257)},
    "star": lambda: star(20000, 20001),
    "star_then_empty": lambda: star(5000, 60000),
    "heavy_first_rows": lambda: S.rmat(13, 32, seed=1),
    "mean_degree_8": lambda: S.erdos_renyi(1500, 8 / 1500, 2, wmax=5),
    "mean_degree_9": lambda: S.erdos_renyi(1500, 9.2 / 1500, 2, wmax=5),
    "grid": lambda: S.grid(90, 0.05, 0.001, seed=3),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_sums_and_terms(name):
    off, idx, w = GRAPHS[name]()
    n = len(off) - 1
    rng = np.random.default_rng(n)
    K = np.bincount(np.repeat(np.arange(n), np.diff(off)), weights=w, minlength=n).astype(np.int64)
    with L.Context(max_n=n, max_nnz=len(idx)) as ctx:
        g = L.Graph.from_numpy(off, idx, w)
        for lab in (np.zeros(n), np.arange(n), rng.integers(0, n, n), np.arange(n) // 7):
            lab = lab.astype(np.int32)
            t = torch.from_numpy(lab).cuda()
            want = O.modularity(off, idx, w, lab)[0] if len(idx) else 0.0
            assert ctx.modularity(g, t) == want
            assert L.modularity_noalloc(g, t) == want
        _, k_out, _, _ = ctx.update(g, torch.arange(n, dtype=torch.int32, device="cuda"), None, None, "ND")
        assert np.array_equal(k_out.cpu().numpy(), K)


@pytest.mark.parametrize("fault", ["offset_falls", "offset_beyond", "offset_first", "offset_last", "column_high",
                                   "column_negative", "weight_zero", "label_high", "label_negative"])
def test_malformed_inputs_are_refused(fault):
    off, idx, w = (a.copy() for a in S.rmat(11, 8, seed=4))
    n = len(off) - 1
    lab = np.arange(n, dtype=np.int32)
    if fault == "offset_falls":
        off[n // 2] = off[n // 2 + 40]
        off[n // 2 + 1] = off[n // 2] - 5
    elif fault == "offset_beyond":
        off[n // 3] = len(idx) + 10
    elif fault == "offset_first":
        off[0] = 1
    elif fault == "offset_last":
        off[n] -= 1
    elif fault == "column_high":
        idx[-1] = n
    elif fault == "column_negative":
        idx[len(idx) // 2] = -3
    elif fault == "weight_zero":
        w[0] = 0
    elif fault == "label_high":
        lab[n - 1] = n
    else:
        lab[5] = -1
    g = L.Graph.from_numpy(off, idx, w)
    t = torch.from_numpy(lab).cuda()
    with L.Context(max_n=n, max_nnz=len(idx)) as ctx:
        calls = [lambda: ctx.modularity(g, t), lambda: L.modularity_noalloc(g, t)]
        if not fault.startswith("label"):
            calls.append(lambda: ctx.static(g))
        calls.append(lambda: ctx.update(g, t, None, None, "DF"))
        for call in calls:
            with pytest.raises(L.LeidenError) as e:
                call()
            assert e.value.code == -1
        good = S.rmat(11, 8, seed=4)
        assert np.array_equal(ctx.static(L.Graph.from_numpy(*good))[0].cpu().numpy(), O.static(*good).membership)
