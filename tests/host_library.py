"""The library's own objects linked with tests/fake_cudart.cpp: its host paths
without a GPU.  Kernels do nothing there, so only what the host decides --
which launches it makes, of what shape, and what it does when one is refused
-- can be looked at."""
from __future__ import annotations

import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp_dir):
    import paper_2405_11658_gb300 as L
    from paper_2405_11658_gb300 import build as B
    B.build()
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    out = os.path.join(str(tmp_dir), "libleiden_host.so")
    cuda = os.path.dirname(os.path.dirname(B.nvcc()))
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out, "-lpthread"], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = ctypes.c_char_p
    return L, lib
