// small.h -- device-visible descriptors of the persistent many-graph kernel
// (small.cuh) and the workspace layout of one graph, shared by the kernel and
// its host driver (batch.cu).
#pragma once

#include <stdint.h>

#include <cuda_runtime.h>

#include "leiden.h"
#include "team.h"

namespace lk {

struct SmallHeader {
  int32_t count;     // jobs in this run
  int32_t wide;      // jobs [0, wide) are run by whole clusters
  uint32_t next;     // queue head of the clusters (0 at launch)
  uint32_t next1;    // queue head of the single blocks (wide at launch)
  int64_t pad[6];
};

struct SmallJob {
  int64_t n, nnz;
  const int64_t *off;
  const int32_t *idx;
  const int32_t *w;
  int32_t mode;      // LEIDEN_STATIC, LEIDEN_ND, LEIDEN_DS or LEIDEN_DF
  int32_t pad0;
  const int32_t *prior;
  int64_t nd, ni;
  const int32_t *ds, *dd, *dw, *is, *id, *iw;
  int32_t *out;
  char *ws;          // this job's workspace slice
  int64_t result;    // index of the caller's item (results are written there)
};

struct SmallOpts {
  int64_t p, q;
  double tol, tol_drop;
  int32_t max_iters, max_passes, log2S, refine_all_first_pass;
};

struct SmallResult {
  int32_t status, passes;
  int64_t affected0, changed0;
  int64_t inside, two_m;
  uint64_t sq_lo, sq_hi;
  int32_t iters[LEIDEN_STATS_PASSES];
  int64_t nv[LEIDEN_STATS_PASSES];
  int64_t nnz[LEIDEN_STATS_PASSES];
  int64_t moves[LEIDEN_STATS_PASSES];
  int64_t refine_moves[LEIDEN_STATS_PASSES];
};

// Byte offsets of one graph's arrays inside its workspace slice (every array
// 256-byte aligned).  n vertices and nnz CSR entries of the input graph bound
// every level (aggregation never grows a graph).
struct SmallLayout {
  int64_t Ctop, Cp, CB, rep, vl, pi, pc, idxA, idxB;
  int64_t Kp, Sp, S2, cnt, cur, K2, offA, offB, wA, wB;
  int64_t ch, ch2, proc, stamp, flag;
  int64_t table;     // aggregation keys and sums; before that the hubs' tables
  int64_t slots;     // aggregation slots (keys, then as many sums)
  int64_t piece_i, piece_k;
  // graphs with more than TEAM_MAX_CAND vertices only (0 elements otherwise)
  int64_t tkeys, hub_i, hub_s, hub_done, part_c, part_kid, part_sc;
  int64_t tcap;      // hub table slots
  int64_t total;
};

__host__ __device__ inline SmallLayout small_layout(int64_t n, int64_t nnz) {
  SmallLayout L{};
  const int64_t nv = n > 0 ? n : 1;
  const int64_t ne = nnz > 0 ? nnz : 1;
  int64_t at = 0;
  auto put = [&](int64_t bytes) {
    const int64_t o = at;
    at += (bytes + 255) & ~(int64_t)255;
    return o;
  };
  L.Ctop = put(nv * 4); L.Cp = put(nv * 4); L.CB = put(nv * 4); L.rep = put(nv * 4); L.vl = put(nv * 4);
  L.pi = put(nv * 4); L.pc = put(nv * 4);
  L.idxA = put(ne * 4); L.idxB = put(ne * 4);
  L.Kp = put(nv * 8); L.Sp = put(nv * 8); L.S2 = put(nv * 8);
  L.cnt = put(nv * 8); L.cur = put(nv * 8); L.K2 = put(nv * 8);
  L.offA = put((nv + 1) * 8); L.offB = put((nv + 1) * 8);
  L.wA = put(ne * 8); L.wB = put(ne * 8);
  L.ch = put(nv); L.ch2 = put(nv); L.proc = put(nv); L.stamp = put(nv); L.flag = put(nv);
  L.slots = ne + ne / 2 + 64;
  L.table = put(L.slots * 16);
  // a mover's row of more than 1024 entries in pieces of 1024
  L.piece_i = put((ne / 512 + 16) * 4); L.piece_k = put((ne / 512 + 16) * 4);
  // hubs: a class's tables hold twice its hubs' entries, each table rounded up
  // to 4096 slots, so the table's 3 nnz words are enough for all of them
  const bool hubs = n > 8192;
  L.tcap = hubs ? 2 * L.slots : 0;
  const int64_t nh = hubs ? ne / 8192 + 16 : 0, np = hubs ? L.tcap / 4096 + 16 : 0;
  L.tkeys = put(L.tcap * 4);
  L.hub_i = put(nh * 4); L.hub_s = put(nh * 4); L.hub_done = put(nh * 4);
  L.part_c = put(np * 4); L.part_kid = put(np * 8); L.part_sc = put(np * 16);
  L.total = at;
  return L;
}

// Upper bound of small_layout(n, nnz).total that is affine in n and nnz, so
// a workspace for sum(n) vertices and sum(nnz) entries over g graphs holds
// every batch within those totals.
__host__ __device__ inline int64_t small_layout_bound(int64_t n, int64_t nnz, int64_t graphs) {
  // per vertex: 7 x 4 + 8 x 8 + 5 bytes; per entry 2 x (4 + 8), 1.5 x 16 for
  // the table, 3 x 4 for the hubs' keys and below 1 for the pieces and hub
  // items; per graph 32 arrays of alignment slack and the fixed extras
  return n * 97 + nnz * 61 + graphs * (34 * 256 + 8192);
}

// Control words of one block (of a cluster: those of its first block).
struct SmallCtl {
  TeamCtl t;
  u64 err;                  // input checks and device consistency flags
  u64 two_m, kmax, inside;
  u64 sq[2];
  u64 affected;
  int32_t job;
};

// The kernel with THREADS (512 or 1024) threads a block.
// Blocks of the largest cluster (1, 2, 4, 8 or 16) that can be resident on the
// current device.
template <int THREADS>
int small_max_cluster();
// Enqueues the kernel: `blocks` blocks in clusters of `cluster`; jobs before
// hdr->wide are run by whole clusters, the others by single blocks.
template <int THREADS>
int launch_small(SmallHeader *hdr, const SmallJob *jobs, const SmallOpts &o, SmallResult *results, SmallCtl *ctl,
                 int blocks, int cluster, cudaStream_t s);
template <> int small_max_cluster<512>();
template <> int small_max_cluster<1024>();
template <> int launch_small<512>(SmallHeader *, const SmallJob *, const SmallOpts &, SmallResult *, SmallCtl *, int,
                                  int, cudaStream_t);
template <> int launch_small<1024>(SmallHeader *, const SmallJob *, const SmallOpts &, SmallResult *, SmallCtl *, int,
                                   int, cudaStream_t);

}  // namespace lk
