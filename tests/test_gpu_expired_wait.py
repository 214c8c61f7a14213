"""A grid barrier of the resident pass whose wait runs out: with a limit of one
poll, in a build of its own, the first barrier of a pass on many blocks gives
up, every block leaves the kernel, the call answers LEIDEN_ETIMEOUT, and the
context goes on working (a small level runs on one cluster, whose hardware
barrier has no limit)."""
from __future__ import annotations

import os
import shutil

import numpy as np
import pytest

import oracle as O
from paper_2405_11658_gb300 import build as B
from paper_2405_11658_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2405_11658_gb300 as L  # noqa: E402


def test_an_expired_wait_is_reported_and_the_context_goes_on(tmp_path, monkeypatch):
    B.build()
    for src in B.SOURCES:   # only the resident pass's objects differ
        obj = src.replace(".cu", ".o")
        if not src.startswith("team_") and os.path.exists(os.path.join(B.BUILD, obj)):
            shutil.copy2(os.path.join(B.BUILD, obj), tmp_path / obj)
    out = B.build(extra_flags=["-DLK_TEAM_SPIN_LIMIT=1"], out=str(tmp_path / "libleiden_wait.so"), build_dir=str(tmp_path))
    monkeypatch.setattr(L, "LIB_PATH", out)
    monkeypatch.setattr(L, "_lib", None)
    small, big = S.planted_partition(2000, 8, 0.03, 0.002, 1), S.rmat(15, 16, seed=3)
    ref = O.static(*small)
    Gs, Gb = L.Graph.from_numpy(*small), L.Graph.from_numpy(*big)
    ctx = L.Context(max_n=Gb.n, max_nnz=Gb.nnz)
    with ctx:
        for _ in range(2):
            with pytest.raises(L.LeidenError) as e:
                ctx.static(Gb)
            assert e.value.code == -4 and "wait expired" in e.value.detail
            memb, q = ctx.static(Gs)
            assert np.array_equal(memb.cpu().numpy(), ref.membership) and q == ref.q
    torch.cuda.synchronize()   # no error left behind
