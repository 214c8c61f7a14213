"""What the host side launches, and what it does when a launch is refused, on a
runtime without a device (tests/fake_cudart.cpp): kernels do nothing there, so
a run ends early with an error; the log of its launches is what is checked."""
from __future__ import annotations

import ctypes as C
import re

import numpy as np
import pytest

from tests import host_library
from tests.batch_shapes import SHAPES


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    L, lib = host_library.load(tmp_path_factory.mktemp("host"))
    return Host(L, lib)


class Host:
    def __init__(self, L, lib):
        self.L, self.lib = L, lib

    def reset(self, device=0, sms=152):
        self.lib.fake_reset()
        self.lib.fake_set_device(device)
        self.lib.fake_set_sms(sms)

    def log(self):
        """The launches so far: (device, kernel, grid, block, cluster, cooperative, refused)."""
        out = []
        for ln in self.lib.fake_log().decode().splitlines():
            m = re.match(r"(\d+) (\S+) grid (\d+) block (\d+) smem \d+ cluster (\d+)( coop)? (ok|refused)", ln)
            out.append((int(m[1]), m[2], int(m[3]), int(m[4]), int(m[5]), bool(m[6]), m[7] == "refused"))
        return out

    def csr(self, n, nnz):
        """A graph by its sizes alone: nothing reads its entries."""
        self.off = np.zeros(n + 1, np.int64)
        self.dummy = np.zeros(4, np.int32)
        return self.L._Csr(n, nnz, self.off.ctypes.data, self.dummy.ctypes.data, self.dummy.ctypes.data)

    def opts(self):
        o = self.L._Opts()
        self.lib.leiden_opts_default(C.byref(o))
        return o

    def static(self, n, nnz, tiers=None):
        ctx = C.c_void_p()
        assert self.lib.leiden_ctx_create(C.byref(ctx), None, C.c_int64(n), C.c_int64(nnz)) == 0
        out = np.zeros(max(n, 1), np.int32)
        g, o = self.csr(n, nnz), self.opts()
        rc = self.lib.leiden_static(ctx, C.byref(g), C.byref(o), C.c_void_p(out.ctypes.data), None)
        self.lib.leiden_ctx_destroy(ctx)
        return rc

    def batch(self, sizes, subsets=8):
        """sizes: (n, nnz) of each graph."""
        b = C.c_void_p()
        assert self.lib.leiden_batch_create(C.byref(b), None, len(sizes), C.c_int64(sum(s[0] for s in sizes)),
                                            C.c_int64(sum(s[1] for s in sizes)), 0, 0) == 0
        items = (self.L._BatchItem * len(sizes))()
        res = (self.L._BatchResult * len(sizes))()
        keep = []
        for it, (n, nnz) in zip(items, sizes):
            it.g = self.csr(n, nnz)
            out = np.zeros(n, np.int32)
            keep.append((self.off, self.dummy, out))
            it.out = out.ctypes.data
        o = self.opts()
        o.det_subsets = subsets
        rc = self.lib.leiden_batch_run(b, len(sizes), items, C.byref(o), res)
        self.lib.leiden_batch_destroy(b)
        return rc


def test_a_second_device_gets_its_own_attributes(host):
    # the first device's calls must not stand in for the second's: a kernel
    # whose shared-memory limit or cluster attribute is unset there is refused
    for device in (0, 1):
        host.reset(device)
        host.static(2000, 18000)       # one cluster of 16 blocks
        host.static(20000, 4000000)    # a cooperative grid
        host.batch([(20000, 400000)] * 4)   # clusters of 16
        log = host.log()
        assert {d for d, *_ in log} == {device}
        team = [x for x in log if "team_pass_k" in x[1]]
        assert [(x[4], x[5]) for x in team] == [(16, False), (1, True)], team
        assert [x[4] for x in log if "small_leiden_k" in x[1]] == [16]
        assert not [x for x in log if x[6]]
        rows = [x for x in log if "rows_k" in x[1] and "check" not in x[1]][-1]
        assert rows[2] == 152 * ((2048 // rows[3]) >> device)   # its own occupancy


@pytest.mark.parametrize("n,nnz,coop,cluster", [(2000, 18000, 0, 1), (20000, 4000000, 1, 0)])
def test_a_refused_resident_launch_runs_the_multi_kernel_path(host, n, nnz, coop, cluster):
    host.reset()
    host.lib.fake_refuse(coop, cluster)
    host.static(n, nnz)
    kernels = [x[1] for x in host.log()]
    team = [k for k, name in enumerate(kernels) if "team_pass_k" in name]
    assert team and host.log()[team[0]][6]
    # the class lists of the multi-kernel path are its first launch
    assert any("bucket_count_k" in name for name in kernels[team[0] + 1:])
    assert host.lib.fake_pending_error() == 0


@pytest.mark.parametrize("most", [16, 8, 4, 2, 1])
def test_batch_clusters_fit_the_device(host, most):
    host.reset()
    host.lib.fake_set_max_cluster(most)
    assert host.batch([(20000, 400000)] * 4) == 0
    small = [x for x in host.log() if "small_leiden_k" in x[1]]
    assert [x[4] for x in small] == [most] and not small[0][6]
    assert host.lib.fake_pending_error() == 0


@pytest.mark.parametrize("name", list(SHAPES))
def test_batch_shapes(host, name):
    sizes, cluster, threads, _ = SHAPES[name]
    host.reset()
    assert host.batch([(s // 10, s - s // 10) for s in sizes]) == 0
    assert [(x[4], x[3]) for x in host.log() if "small_leiden_k" in x[1]] == [(cluster, threads)]


@pytest.mark.parametrize("share,subsets,threads", [(27648, 1, 512), (27649, 1, 1024), (49152, 8, 512), (49153, 8, 1024),
                                                   (122880, 32, 512), (122881, 32, 1024)])
def test_batch_threads_by_the_share_of_a_block(host, share, subsets, threads):
    host.reset()
    host.lib.fake_set_max_cluster(1)
    assert host.batch([(100, share - 100), (100, 900)], subsets) == 0
    assert [x[3] for x in host.log() if "small_leiden_k" in x[1]] == [threads]


def admit(host, srv, n, nnz):
    """Admits a graph of these sizes and waits for its Static run."""
    off = np.zeros(n + 1, np.int64)
    off[n] = nnz
    idx = np.zeros(max(nnz, 1), np.int32)
    gid, rid = C.c_int32(), C.c_int64()
    assert host.lib.leiden_server_admit(srv, C.c_int64(n), C.c_int64(nnz), C.c_void_p(off.ctypes.data),
                                        C.c_void_p(idx.ctypes.data), C.c_void_p(idx.ctypes.data), C.byref(gid),
                                        C.byref(rid)) == 0
    info = host.L._RequestInfo()
    assert host.lib.leiden_server_wait(srv, rid, C.c_double(-1.0), C.byref(info)) == 0
    return gid


def test_the_server_leaves_sms_to_the_small_workers(host):
    # a large graph's pass takes 32 SMs less while a small graph is resident
    host.reset()
    cfg = host.L._ServerConfig()
    host.lib.leiden_server_config_default(C.byref(cfg))
    n, nnz = 20000, 4000000
    cfg.small_max_n, cfg.small_max_nnz, cfg.large_max_n, cfg.large_max_nnz = 1000, 10000, n, 2 * nnz
    srv = C.c_void_p()
    assert host.lib.leiden_server_create(C.byref(srv), C.byref(cfg)) == 0

    def large():
        first = len(host.log())
        admit(host, srv, n, nnz)
        return [x[2] for x in host.log()[first:] if "team_pass_k" in x[1]]

    assert large() == [152]
    small = admit(host, srv, 100, 1000)
    assert large() == [152 - 32]
    assert host.lib.leiden_server_evict(srv, small) == 0
    assert large() == [152]
    host.lib.leiden_server_destroy(srv)


def test_the_csr_pass_follows_the_sms_of_the_device(host):
    # one wave on a device (or a context's share) of 8 SMs, not on 152
    host.reset(sms=8)
    n, nnz = 20000, 4000000
    host.static(n, nnz)
    g = host.csr(n, nnz)
    lab, q = np.zeros(n, np.int32), C.c_double()
    assert host.lib.leiden_modularity_noalloc(C.byref(g), C.c_void_p(lab.ctypes.data), C.c_double(1.0), None,
                                              C.byref(q)) == 0
    rows = [x for x in host.log() if "rows_k" in x[1] and "check" not in x[1]]
    assert len(rows) == 2 and all(x[2] == 8 * (2048 // x[3]) for x in rows), rows
