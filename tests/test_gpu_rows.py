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
    with L.Context(max_n=n, max_nnz=len(idx) + 8) as ctx:
        calls = [lambda: ctx.modularity(g, t), lambda: L.modularity_noalloc(g, t)]
        if not fault.startswith("label"):
            calls.append(lambda: ctx.static(g))
            calls.append(lambda: ctx.apply_batch(g, None, L.Edges.from_numpy(([0], [n - 1], [1]))))
        calls.append(lambda: ctx.update(g, t, None, None, "DF"))
        for call in calls:
            with pytest.raises(L.LeidenError) as e:
                call()
            assert e.value.code == -1
        good = S.rmat(11, 8, seed=4)
        assert np.array_equal(ctx.static(L.Graph.from_numpy(*good))[0].cpu().numpy(), O.static(*good).membership)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_batch_application_reads_any_alignment(shift):
    # entry arrays that start 4, 8 or 12 bytes past a 16-byte boundary
    off, idx, w = S.chung_lu(3000, 15000, 2.1, 1, 4, seed=5)
    big_i = torch.zeros(len(idx) + 8, dtype=torch.int32, device="cuda")
    big_w = torch.zeros(len(idx) + 8, dtype=torch.int32, device="cuda")
    big_i[shift:shift + len(idx)] = torch.from_numpy(idx).cuda()
    big_w[shift:shift + len(idx)] = torch.from_numpy(w).cuda()
    g = L.Graph(torch.from_numpy(off).cuda(), big_i[shift:shift + len(idx)], big_w[shift:shift + len(idx)])
    dels, ins = S.random_batch(off, idx, w, 200, seed=6)
    want = O.apply_batch(off, idx, w, dels, ins)
    with L.Context(max_n=g.n, max_nnz=g.nnz + 1024) as ctx:
        got = ctx.apply_batch(g, L.Edges.from_numpy(dels), L.Edges.from_numpy(ins))
    for a, b in zip((got.off, got.idx, got.w), want):
        assert np.array_equal(a.cpu().numpy(), b)


def heavy_batch(n, hub_deg, hub_ins, hub_dels, seed, repeats=1):
    """A graph whose vertex 0 has hub_deg neighbours, and a batch that inserts
    hub_ins edges at it (each listed `repeats` times) and deletes hub_dels."""
    rng = np.random.default_rng(seed)
    nb = rng.choice(np.arange(1, n), hub_deg + hub_ins, replace=False)
    u = np.concatenate([np.zeros(hub_deg, np.int64), rng.integers(1, n, 2 * n)])
    v = np.concatenate([nb[:hub_deg], rng.integers(1, n, 2 * n)])
    g = S.edges_to_csr(n, u, v, rng.integers(1, 9, len(u)))
    off, idx, w = g
    pick = rng.choice(off[1], hub_dels, replace=False)
    dels = (np.zeros(hub_dels, np.int32), idx[pick], w[pick])
    # new neighbours, repeats of them, and some of the old ones reweighted
    t = np.concatenate([np.repeat(nb[hub_deg:], repeats), np.setdiff1d(idx[:off[1]], idx[pick])[:hub_ins // 3]])
    t = rng.permutation(t).astype(np.int32)
    ins = (np.zeros(len(t), np.int32), t, rng.integers(1, 5, len(t)).astype(np.int32))
    return g, dels, ins


@pytest.mark.parametrize("hub_deg,hub_ins,hub_dels,repeats", [
    (40, 8, 4, 1), (40, 16, 1, 1), (40, 17, 0, 1),              # around the serial limit of 16 updates
    (256, 3, 0, 1), (257, 3, 3, 1), (300, 255, 40, 1), (300, 257, 40, 2),   # around one merge piece
    (512, 1, 0, 1), (513, 200, 100, 3), (1024, 255, 1, 1),
    (6000, 3000, 1000, 1), (6000, 3000, 1096, 1), (9000, 4000, 2000, 2),    # around the shared-memory sort
])
def test_batches_on_a_heavy_row(hub_deg, hub_ins, hub_dels, repeats):
    g, dels, ins = heavy_batch(20000, hub_deg, hub_ins, hub_dels, 7, repeats)
    want = O.apply_batch(*g, dels, ins)
    with L.Context(max_n=20000, max_nnz=len(g[1]) + 4 * len(ins[0]) + 2 * len(dels[0])) as ctx:
        got = ctx.apply_batch(L.Graph.from_numpy(*g), L.Edges.from_numpy(dels), L.Edges.from_numpy(ins))
        for a, b in zip((got.off, got.idx, got.w), want):
            assert np.array_equal(a.cpu().numpy(), b)
        # refused as before: a deletion listed twice, one of a wrong weight
        if hub_dels >= 2:
            twice = tuple(np.concatenate([x, x[:1]]) for x in dels)
            wrong = (dels[0], dels[1], dels[2] + 1)
            for bad in (twice, wrong):
                with pytest.raises(L.LeidenError) as e:
                    ctx.apply_batch(L.Graph.from_numpy(*g), L.Edges.from_numpy(bad), L.Edges.from_numpy(ins))
                assert e.value.code == -1
