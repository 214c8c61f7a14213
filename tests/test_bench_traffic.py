"""The stored DRAM-traffic figure of the decide phase: every source that phase is
compiled from invalidates it, and a capture without decide kernels records
nothing."""
from __future__ import annotations

import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2405_11658_gb300", "csrc")


def closure(name, seen):
    """A source of csrc/ and the files there it includes."""
    if name in seen or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'#include "([^"]+)"', f.read()):
            closure(inc, seen)
    return seen


def test_every_source_of_the_decide_phase_counts():
    want = set()
    for name in ("move.cu", "hub.cu", "team_n32.cu", "team_n64.cu", "team_w32.cu", "team_w64.cu"):
        closure(name, want)
    assert {"team.cuh", "team.h", "team_launch.cuh"} <= want
    assert want <= {os.path.basename(f) for f in bench.DECIDE_SOURCES}


def test_a_capture_without_decide_kernels_is_refused(monkeypatch, tmp_path):
    hdr = '"ID","Kernel Name","Metric Name","Metric Unit","Metric Value"'
    cap = tmp_path / "cap.csv"
    cap.write_text(hdr + '\n"0","void lk::team_pass_k<int, long>(TeamArgs<T1>, int)","dram__bytes_read.sum","Gbyte","1.0"\n')
    prof = tmp_path / "prof.log"
    prof.write_text('{"workload": "w", "move0_kernel_launches": 2, "move0_bytes": 1.0, "move0_scanned_entries": 1}\n')
    out = tmp_path / "traffic.json"
    monkeypatch.setitem(bench.TRAFFIC_FILES, "cl", str(out))

    class A:
        record_traffic, profile_json, workload = str(cap), str(prof), "cl"
    assert bench.record_traffic(A) != 0
    assert not out.exists()
