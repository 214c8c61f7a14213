// small.cuh -- many small graphs in one persistent launch (leiden_batch_run).
// Compiled for two block sizes (small_512.cu, small_1024.cu).
//
// Each team of blocks (team.cuh) runs the whole of Alg. leiden for one graph
// at a time -- marking (Alg. naive / delta / frontier), every pass, the
// dendrogram lookup, canonical labels and the terms of Eq. 1 -- then takes the
// next graph from a device-side queue.  A team is a thread-block cluster for
// the graphs at the head of the queue (the largest) and a single block for
// the others; teams never wait for one another.
//
// The passes are those of leiden_static / leiden_update (team_pass), so each
// graph ends with the same membership and statistics as those calls give it.
//
// What bounds it: one graph's chain of sub-sweeps, each two barriers and the
// dependent loads of one vertex; a cluster shortens the work between the
// barriers, and with fewer graphs than SMs the others would be idle anyway.
// On the smallest graphs it is the code itself: 1024 threads leave 64 registers
// each, and the spilled words of a block (270 KB) do not fit the L1 that the
// tables leave, so every reload waits for L2 (L1 hit rate 34%).  512 threads
// hold everything in 128 registers; with more of a graph to a block, 1024's
// gathers in flight count for more (batch.cu has the rule).  ms with one 512-thread block per graph, tables cleared per
// vertex and 128-bit scores throughout / 1024 threads here / 512 threads here:
// 64 graphs of 1e3..1e4 vertices, half of them updates 47.8 / 14.2 / 12.7; 8
// graphs of up to 300 vertices 3.2 / 4.7 / 2.7; 88 of up to 1000 8.3 / 8.0 /
// 5.9; 60 R-MAT of scale 14 176 / 69 / 81.
#include <limits.h>

#include "common.cuh"
#include "internal.h"
#include "small.h"
#include "team.cuh"

namespace lk {
inline namespace LK_TEAM_SPACE {

namespace {

typedef TeamShared<i128> WideShared;
static_assert(sizeof(TeamShared<int64_t>) <= sizeof(WideShared), "one shared block for both score widths");

// What the block's current job reads again and again: one copy per block in
// shared memory, read anew at every use (Held).  As by-value arguments, or as
// plain shared words that the compiler keeps in registers, they spilled
// thousands of bytes in a thread of a 1024-thread block.
struct SmallArrays {
  static constexpr bool MANY_HUBS = true;
  Held<int32_t *> C, CB, rep, vlist;
  Held<int64_t *> K, Sig, Sig2;
  Held<uint8_t *> ch, ch2, processed, stamp, exists;
  Held<int32_t *> prop_i, prop_c;
  Held<u64 *> err;
  Held<int32_t *> tkeys;
  Held<u64 *> tvals;
  Held<int64_t> tcap;
  Held<int32_t *> hub_i, hub_s, hub_done, part_c;
  Held<i128 *> part_sc;
  Held<int64_t *> part_kid;
  Held<int32_t *> piece_i, piece_k;
  Held<u64 *> hkey, hval;
  Held<int64_t *> cnt, cur, K2, off2;
  Held<int32_t *> idx2;
  Held<int64_t *> w2;
};
struct SmallConst {
  Held<int64_t> A, p;
  Held<double> den;
  Held<int64_t> two_m;
  Held<int> log2S, dynamic, timing;
  Held<const uint8_t *> in_range;
};
template <typename WT>
struct SmallLevel {
  Held<int64_t> n, nnz;
  Held<const int64_t *> off;
  Held<const int32_t *> idx;
  Held<const WT *> w;
  __device__ void set(int64_t n_, int64_t nnz_, const int64_t *off_, const int32_t *idx_, const WT *w_) {
    n = n_; nnz = nnz_; off = off_; idx = idx_; w = w_;
  }
};
// Workspace of one graph, carved from its slice of the batch arena.
struct WS {
  int32_t *Ctop, *idx[2];
  int64_t *off[2], *w[2];
  int64_t slots;
};
struct SmallState {
  SmallArrays a;
  SmallConst ct;
  SmallLevel<int64_t> g;
  WS w;
  // the pass at hand: its number, level buffer (-1: the input), sizes, largest
  // K', tolerance and score width
  int lp, cur, narrow;
  int64_t nv, nnz, kmax;
  double tau;
};

// Carves the slice (one thread of the block).
__device__ __forceinline__ void carve_ws(char *base, int64_t n, int64_t nnz, u64 *err, WS &w, SmallArrays &a) {
  const SmallLayout L = small_layout(n, nnz);
  w.Ctop = (int32_t *)(base + L.Ctop);
  w.idx[0] = (int32_t *)(base + L.idxA);
  w.idx[1] = (int32_t *)(base + L.idxB);
  w.off[0] = (int64_t *)(base + L.offA);
  w.off[1] = (int64_t *)(base + L.offB);
  w.w[0] = (int64_t *)(base + L.wA);
  w.w[1] = (int64_t *)(base + L.wB);
  w.slots = L.slots;
  a.C = (int32_t *)(base + L.Cp);
  a.CB = (int32_t *)(base + L.CB);
  a.rep = (int32_t *)(base + L.rep);
  a.vlist = (int32_t *)(base + L.vl);
  a.K = (int64_t *)(base + L.Kp);
  a.Sig = (int64_t *)(base + L.Sp);
  a.Sig2 = (int64_t *)(base + L.S2);
  a.ch = (uint8_t *)(base + L.ch);
  a.ch2 = (uint8_t *)(base + L.ch2);
  a.processed = (uint8_t *)(base + L.proc);
  a.stamp = (uint8_t *)(base + L.stamp);
  a.exists = (uint8_t *)(base + L.flag);
  a.prop_i = (int32_t *)(base + L.pi);
  a.prop_c = (int32_t *)(base + L.pc);
  a.err = err;
  a.tkeys = (int32_t *)(base + L.tkeys);
  a.tvals = (u64 *)(base + L.table);
  a.tcap = L.tcap;
  a.hub_i = (int32_t *)(base + L.hub_i);
  a.hub_s = (int32_t *)(base + L.hub_s);
  a.hub_done = (int32_t *)(base + L.hub_done);
  a.part_c = (int32_t *)(base + L.part_c);
  a.part_sc = (i128 *)(base + L.part_sc);
  a.part_kid = (int64_t *)(base + L.part_kid);
  a.piece_i = (int32_t *)(base + L.piece_i);
  a.piece_k = (int32_t *)(base + L.piece_k);
  a.hkey = (u64 *)(base + L.table);
  a.hval = a.hkey + L.slots;
  a.cnt = (int64_t *)(base + L.cnt);
  a.cur = (int64_t *)(base + L.cur);
  a.K2 = (int64_t *)(base + L.K2);
}

// Checks of one job's inputs into ctl->err.
__device__ __forceinline__ void check_job(const SmallJob &j, const Team &t, u64 *err) {
  const int64_t gt = t.index(), nt = (int64_t)t.nb * TEAM_THREADS, n = j.n;
  bool bad = false;
  for (int64_t i = gt; i < n; i += nt) {
    const int64_t a = j.off[i], b = j.off[i + 1];
    if (a > b || a < 0 || b > j.nnz) bad = true;
  }
  if (gt == 0 && (j.off[0] != 0 || j.off[n] != j.nnz)) bad = true;
  for (int64_t e = gt; e < j.nnz; e += nt)
    if (j.idx[e] < 0 || j.idx[e] >= n || j.w[e] <= 0) bad = true;
  if (j.mode != LEIDEN_STATIC) {
    for (int64_t i = gt; i < n; i += nt)
      if (j.prior[i] < 0 || j.prior[i] >= n) bad = true;
    for (int64_t k = gt; k < j.nd + j.ni; k += nt) {
      const bool del = k < j.nd;
      const int64_t x = del ? k : k - j.nd;
      const int32_t u = del ? j.ds[x] : j.is[x], v = del ? j.dd[x] : j.id[x];
      const int32_t wt = del ? j.dw[x] : j.iw[x];
      if (u < 0 || u >= n || v < 0 || v >= n || u == v || wt <= 0) bad = true;
    }
  }
  if (bad) atomicOr(err, 1ull);
}

// Alg. delta: the affected vertices (a.exists, the range of the first pass;
// they start unprocessed), with a.ch2 as delta-E (vertices whose neighbours
// are affected) and a.stamp as delta-C (communities whose members are
// affected).  Deletions inside a community mark both ends and the community;
// for each source of insertions, the best community c* != its own by Eq. 2
// with K_{i->c} the inserted weight towards c and K_{i->d} = 0 (ties to the
// smallest c) marks the source and c*.  K and Sigma are those of G^t and
// C^{t-1}.  Batches of the persistent path are small: each source's insertions
// are grouped by scanning the batch.  Returns false after an expired wait.
__device__ __forceinline__ bool mark_ds(const SmallJob &j, const SmallArrays &a, const SmallConst &ct, Team &t) {
  const int64_t N = j.n, gt = t.index(), nt = (int64_t)t.nb * TEAM_THREADS;
  uint8_t *aff = a.exists, *dE = a.ch2, *dC = a.stamp;
  for (int64_t i = gt; i < N; i += nt) { aff[i] = 0; dE[i] = 0; dC[i] = 0; }
  TEAM_SYNC_OR(false);
  for (int64_t k = gt; k < j.nd; k += nt) {
    const int32_t u = j.ds[k], v = j.dd[k];
    const int32_t c = j.prior[u];
    if (c != j.prior[v]) continue;
    aff[u] = 1; dE[u] = 1;
    aff[v] = 1; dE[v] = 1;
    dC[c] = 1;
  }
  // directed insertion entries x in [0, 2 ni): (is, id) then (id, is)
  const int64_t E = 2 * j.ni;
  auto src = [&](int64_t x) { return x < j.ni ? j.is[x] : j.id[x - j.ni]; };
  auto dst = [&](int64_t x) { return x < j.ni ? j.id[x] : j.is[x - j.ni]; };
  auto wt = [&](int64_t x) { return (int64_t)(x < j.ni ? j.iw[x] : j.iw[x - j.ni]); };
  for (int64_t x = gt; x < E; x += nt) {
    const int32_t u = src(x);
    bool first = true;
    for (int64_t y = 0; y < x && first; y++) first = src(y) != u;
    if (!first) continue;
    const int32_t d = j.prior[u];
    const int64_t Ki = a.K[u];
    int32_t best = INT32_MAX;
    i128 bS = 0;
    for (int64_t y = x; y < E; y++) {
      if (src(y) != u) continue;
      const int32_t c = j.prior[dst(y)];
      if (c == d) continue;
      bool seen = false;
      for (int64_t z = x; z < y && !seen; z++) seen = src(z) == u && j.prior[dst(z)] == c;
      if (seen) continue;
      int64_t h = 0;
      for (int64_t z = y; z < E; z++)
        if (src(z) == u && j.prior[dst(z)] == c) h += wt(z);
      const i128 S = (i128)ct.A * h - (i128)ct.p * Ki * (Ki + a.Sig[c] - a.Sig[d]);
      if (best == INT32_MAX || S > bS || (S == bS && c < best)) { bS = S; best = c; }
    }
    if (best != INT32_MAX) {
      aff[u] = 1;
      dE[u] = 1;
      dC[best] = 1;
    }
  }
  TEAM_SYNC_OR(false);
  // expansion: members of delta-C communities and neighbours of delta-E vertices
  for (int64_t i = gt; i < N; i += nt) {
    if (dC[j.prior[i]]) aff[i] = 1;
    if (dE[i])
      for (int64_t e = j.off[i]; e < j.off[i + 1]; e++) aff[j.idx[e]] = 1;
  }
  TEAM_SYNC_OR(false);
  for (int64_t i = gt; i < N; i += nt) a.processed[i] = aff[i] ? 0 : 1;
  return true;
}

// Dynamic shared memory of a block: the tables (sized for 64-bit values), the
// TeamShared words, the job's state.  Every function takes its address anew,
// so that the compiler knows the accesses for shared ones.
constexpr size_t kTables = (size_t)TEAM_WARPS * TEAM_WSLOTS * (sizeof(u64) + sizeof(int32_t));
constexpr size_t kState = kTables + ((sizeof(WideShared) + 15) & ~(size_t)15);
constexpr size_t kSmem = kState + sizeof(SmallState);
extern __shared__ __align__(16) unsigned char small_dyn[];
__device__ __forceinline__ SmallState &small_state() { return *reinterpret_cast<SmallState *>(small_dyn + kState); }


// The pass at hand of state: clears the control words, points the arrays at the
// level and its output, picks the score width.
__device__ __forceinline__ void small_next(const SmallJob &j, const SmallOpts &o, const Team &t, SmallCtl *ctl) {
  SmallState &s = small_state();
  unsigned *z = reinterpret_cast<unsigned *>(&ctl->t);
  for (unsigned k = (unsigned)t.index(); k < sizeof(TeamCtl) / 4; k += (unsigned)(t.nb * TEAM_THREADS)) z[k] = 0;
  if (threadIdx.x == 0) {
    const int cur = s.cur, dst = cur < 0 ? 0 : 1 - cur;
    s.a.off2 = s.w.off[dst];
    s.a.idx2 = s.w.idx[dst];
    s.a.w2 = s.w.w[dst];
    if (cur < 0) s.g.set(j.n, j.nnz, j.off, j.idx, s.w.w[1]);
    else s.g.set(s.nv, s.nnz, s.w.off[cur], s.w.idx[cur], s.w.w[cur]);
    // 64-bit scores while every product stays below 2^62 (see narrow_scores)
    const int64_t pq = o.p > o.q ? o.p : o.q, two_m = s.ct.two_m;
    s.narrow = !LK_FORCE_WIDE_SCORES && s.kmax < ((int64_t)1 << 31) &&
               (i128)s.kmax * two_m * pq < ((i128)1 << 62);
  }
}

// Everything before the first pass of a job; false when there is none (bad
// input, or a result without passes).  The functions around the passes are not
// inlined: the passes, inlined once each into the kernel, then have its
// registers to themselves (as functions of their own they spilled twice as
// much: 64 graphs of 1e3..1e4 vertices 16.6 ms, 14.1 so).
__device__ __noinline__ bool small_setup(const SmallJob &j, const SmallOpts &o, SmallResult *res, Team t,
                                         SmallCtl *ctl) {
  const int64_t N = j.n, gt = t.index(), nt = (int64_t)t.nb * TEAM_THREADS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wg = warp * t.nb + t.rank, W = t.nb * TEAM_WARPS;
  const bool lead = t.rank == 0 && threadIdx.x == 0;
  if (lead) {
    res->status = LEIDEN_OK;
    res->passes = 0;
    res->affected0 = 0;
    res->changed0 = 0;
    ctl->err = ctl->two_m = ctl->kmax = ctl->inside = ctl->sq[0] = ctl->sq[1] = ctl->affected = 0;
  }
  TEAM_SYNC_OR(false);
  check_job(j, t, &ctl->err);
  TEAM_SYNC_OR(false);
  if (*(volatile u64 *)&ctl->err) {
    if (lead) res->status = LEIDEN_EINVAL;
    return false;
  }
  SmallState &state = small_state();
  if (threadIdx.x == 0) carve_ws(j.ws, N, j.nnz, &ctl->err, state.w, state.a);
  __syncthreads();
  const WS &w = state.w;
  const SmallArrays &a0 = state.a;
  const bool upd = j.mode != LEIDEN_STATIC;
  // K = row sums of G^t; 2m = their total
  {
    u64 tot = 0, kmax = 0;
    for (int64_t i = wg; i < N; i += W) {
      int64_t k = 0;
      for (int64_t e = j.off[i] + lane; e < j.off[i + 1]; e += 32) k += (int64_t)j.w[e];
      for (int s = 16; s; s >>= 1) k += shfl_xor_i64(k, s);
      if (lane == 0) a0.K[i] = k;
      tot += (u64)k;
      kmax = (u64)k > kmax ? (u64)k : kmax;
    }
    if (lane == 0 && tot) { atomicAdd(&ctl->two_m, tot); atomicMax(&ctl->kmax, kmax); }
  }
  // the input's weights as the passes read them (64 bits), in the level buffer
  // that the first aggregation leaves alone; the scratch tables start empty
  for (int64_t e = gt; e < j.nnz; e += nt) w.w[1][e] = (int64_t)j.w[e];
  for (int64_t s = gt; s < 2 * w.slots; s += nt) a0.hkey[s] = 0;
  for (int64_t s = gt; s < a0.tcap; s += nt) a0.tkeys[s] = LEIDEN_EMPTY_KEY;
  for (int64_t i = gt; i < N; i += nt) {
    w.Ctop[i] = (int32_t)i;
    a0.C[i] = upd ? j.prior[i] : (int32_t)i;
    a0.Sig[i] = 0;
    a0.ch[i] = upd ? (o.refine_all_first_pass ? 1 : 0) : 1;
    a0.processed[i] = (upd && j.mode == LEIDEN_DF) ? 1 : 0;
  }
  TEAM_SYNC_OR(false);
  const int64_t two_m = (int64_t)__ldcg(&ctl->two_m);
  if (two_m < 0 || two_m >= ((int64_t)1 << 40)) {
    if (lead) res->status = LEIDEN_EOVERFLOW;
    return false;
  }
  if (threadIdx.x == 0) {
    SmallConst &ct = state.ct;
    ct.p = o.p;
    ct.two_m = two_m;
    ct.A = two_m * o.q;
    ct.den = (double)two_m * (double)two_m * 0.5 * (double)o.q;
    ct.log2S = o.log2S;
    ct.dynamic = upd ? 1 : 0;
    ct.timing = 0;
    // the DS range stays in the exists flags, which a pass clears after its moves
    ct.in_range = j.mode == LEIDEN_DS ? (const uint8_t *)(uint8_t *)a0.exists : nullptr;
  }
  __syncthreads();
  for (int64_t i = gt; i < N; i += nt) {
    if (!upd) a0.Sig[i] = a0.K[i];
    else if (a0.K[i]) atomic_add_i64(&a0.Sig[a0.C[i]], a0.K[i]);
  }
  if (upd) {
    for (int64_t k = gt; k < j.nd + j.ni; k += nt) {
      const bool del = k < j.nd;
      const int64_t x = del ? k : k - j.nd;
      const int32_t u = del ? j.ds[x] : j.is[x], v = del ? j.dd[x] : j.id[x];
      const bool same = j.prior[u] == j.prior[v];
      if (same && !o.refine_all_first_pass) a0.ch[j.prior[u]] = 1;                       // changedCommunities
      if (j.mode == LEIDEN_DF && same == del) { a0.processed[u] = 0; a0.processed[v] = 0; }  // Alg. frontier
    }
    TEAM_SYNC_OR(false);
    if (j.mode == LEIDEN_DS) {
      if (!mark_ds(j, a0, state.ct, t)) return false;
      TEAM_SYNC_OR(false);
    }
    u64 k = 0;
    for (int64_t i = gt; i < N; i += nt) k += a0.processed[i] == 0;
    for (int s = 16; s; s >>= 1) k += (u64)shfl_xor_i64((int64_t)k, s);
    if (lane == 0 && k) atomicAdd(&ctl->affected, k);
    TEAM_SYNC_OR(false);
    if (lead) res->affected0 = (int64_t)__ldcg(&ctl->affected);
  } else {
    if (lead) res->affected0 = N;
    TEAM_SYNC_OR(false);
  }

  if (threadIdx.x == 0) {
    state.lp = 0;
    state.cur = -1;
    state.nv = N;
    state.nnz = j.nnz;
    state.kmax = (int64_t)__ldcg(&ctl->kmax);
    state.tau = o.tol;
  }
  __syncthreads();
  if (N == 0 && lead) {   // an empty graph: one pass over nothing
    res->passes = 1;
    res->iters[0] = 1;
    res->nv[0] = res->nnz[0] = res->moves[0] = res->refine_moves[0] = 0;
  }
  if (N > 0) small_next(j, o, t, ctl);
  t.sync();
  return N > 0;
}

// After a pass: its statistics, the dendrogram lookup and the next pass; false
// when it was the last one.
__device__ __noinline__ bool small_after(const SmallJob &j, const SmallOpts &o, SmallResult *res, Team t,
                                         SmallCtl *ctl) {
  SmallState &s = small_state();
  const bool lead = t.rank == 0 && threadIdx.x == 0;
  const volatile TeamCtl &h = ctl->t;
  const int status = h.status, lp = s.lp;
  if (lead && lp < LEIDEN_STATS_PASSES) {
    if (lp == 0) res->changed0 = (int64_t)h.changed;
    res->nnz[lp] = s.nnz;
    res->passes = lp + 1;
    res->iters[lp] = h.li;
    res->nv[lp] = s.nv;
    res->moves[lp] = h.moves;
    res->refine_moves[lp] = (int64_t)h.rmoves;
  }
  if (status != TEAM_AGGREGATED) {
    if (status != TEAM_CONVERGED && status != TEAM_NO_SHRINK && lead) atomicOr(&ctl->err, 2048ull);
    return false;
  }
  for (int64_t v = t.index(); v < j.n; v += (int64_t)t.nb * TEAM_THREADS)
    s.w.Ctop[v] = s.a.CB[s.w.Ctop[v]];
  const int64_t nv = h.nc, nnz = h.nnz2, kmax = (int64_t)h.kmax;
  t.sync();   // the control words are read before they are cleared
  if (threadIdx.x == 0) {
    s.cur = s.cur < 0 ? 0 : 1 - s.cur;
    s.nv = nv;
    s.nnz = nnz;
    s.kmax = kmax;
    s.tau /= o.tol_drop;
    s.lp = lp + 1;
    s.ct.dynamic = 0;
    s.ct.in_range = (const uint8_t *)nullptr;
  }
  __syncthreads();
  if (lp + 1 >= o.max_passes) return false;
  small_next(j, o, t, ctl);
  t.sync();
  return true;
}

// The returned membership and the terms of its modularity.
__device__ __noinline__ void small_finish(const SmallJob &j, SmallResult *res, Team t, SmallCtl *ctl) {
  WideShared &sm = *reinterpret_cast<WideShared *>(small_dyn + kTables);
  SmallState &state = small_state();
  const WS &w = state.w;
  const int64_t N = j.n, gt = t.index(), nt = (int64_t)t.nb * TEAM_THREADS, two_m = state.ct.two_m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wg = warp * t.nb + t.rank, W = t.nb * TEAM_WARPS;
  const bool lead = t.rank == 0 && threadIdx.x == 0;
  TEAM_SYNC_OR();
  // last lookup, then canonical labels: communities numbered by their
  // smallest member
  const SmallArrays &a = state.a;
  for (int64_t v = gt; v < N; v += nt) {
    w.Ctop[v] = a.C[w.Ctop[v]];
    a.exists[v] = 0;
    a.rep[v] = INT_MAX;
    a.Sig2[v] = 0;
  }
  TEAM_SYNC_OR();
  for (int64_t v = gt; v < N; v += nt) {
    const int32_t c = w.Ctop[v];
    if (__ldcg(&a.rep[c]) > (int32_t)v) atomicMin(&a.rep[c], (int32_t)v);
  }
  TEAM_SYNC_OR();
  for (int64_t c = gt; c < N; c += nt) {
    const int32_t r = __ldcg(&a.rep[c]);
    if (r != INT_MAX) a.exists[r] = 1;
  }
  TEAM_SYNC_OR();
  team_scan<i128>(
      N, t, sm, [&](int64_t c) { return (int64_t)a.exists[c]; },
      [&](int64_t c, int64_t pre) { a.CB[c] = (int32_t)pre; });
  if (t.dead) return;
  TEAM_SYNC_OR();
  for (int64_t v = gt; v < N; v += nt) j.out[v] = a.CB[a.rep[w.Ctop[v]]];
  TEAM_SYNC_OR();
  // Eq. 1 terms of the returned membership on the input graph
  {
    int64_t inside = 0;
    for (int64_t i = wg; i < N; i += W) {
      const int32_t ci = j.out[i];
      int64_t k = 0;
      for (int64_t e = j.off[i] + lane; e < j.off[i + 1]; e += 32) {
        const int64_t x = (int64_t)j.w[e];
        k += x;
        if (j.out[j.idx[e]] == ci) inside += x;
      }
      for (int s = 16; s; s >>= 1) k += shfl_xor_i64(k, s);
      if (lane == 0 && k) atomic_add_i64(&a.Sig2[ci], k);
    }
    for (int s = 16; s; s >>= 1) inside += shfl_xor_i64(inside, s);
    if (lane == 0 && inside) atomicAdd(&ctl->inside, (u64)inside);
  }
  TEAM_SYNC_OR();
  {
    i128 sq = 0;
    for (int64_t c = gt; c < N; c += nt) sq += (i128)__ldcg(&a.Sig2[c]) * __ldcg(&a.Sig2[c]);
    for (int s = 16; s; s >>= 1) sq += shfl_xor_i128(sq, s);
    if (lane == 0 && sq != 0) atomic_add_i128(ctl->sq, sq);
  }
  TEAM_SYNC_OR();
  if (lead) {
    res->inside = (int64_t)__ldcg(&ctl->inside);
    res->two_m = two_m;
    res->sq_lo = __ldcg(&ctl->sq[0]);
    res->sq_hi = __ldcg(&ctl->sq[1]);
    if (__ldcg(&ctl->err)) res->status = LEIDEN_ECUDA;
  }
}

}  // namespace

__global__ void __launch_bounds__(TEAM_THREADS, 1) small_leiden_k(SmallHeader *hdr, const SmallJob *jobs, SmallOpts o,
                                                                  SmallResult *results, SmallCtl *ctls) {
  WideShared &sm = *reinterpret_cast<WideShared *>(small_dyn + kTables);
  unsigned rank, nb;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nb));
  if (threadIdx.x == 0) sm.dead = 0;
  __syncthreads();
  Team t;
  t.gen = 0;
  t.dead_s = &sm.dead;
  t.dead = false;
  const int count = hdr->count, wide = hdr->wide;
  // the largest graphs first, a cluster each; then the others, a block each
  t.rank = (int)rank;
  t.nb = (int)nb;
  t.kind = nb > 1 ? TEAM_CLUSTER : TEAM_BLOCK;
  SmallCtl *ctl = &ctls[blockIdx.x - rank];
  bool cluster = true;
  for (;;) {
    t.ctl = &ctl->t;
    if (t.rank == 0 && threadIdx.x == 0) ctl->job = (int)atomicAdd(cluster ? &hdr->next : &hdr->next1, 1u);
    t.sync();
    const int k = *(volatile int32_t *)&ctl->job;
    t.sync();
    if (k >= (cluster ? wide : count)) {
      if (!cluster) break;
      cluster = false;
      t.rank = 0;
      t.nb = 1;
      t.kind = TEAM_BLOCK;
      ctl = &ctls[blockIdx.x];
      continue;
    }
    const SmallJob &j = jobs[k];
    SmallResult *res = &results[j.result];
    if (small_setup(j, o, res, t, ctl)) {
      SmallState &s = small_state();
      do {
        if (s.narrow)
          team_pass<true, int64_t, int64_t>(s.g, s.a, s.ct, s.lp, s.tau, o.max_iters, s.w.slots, t, small_dyn,
                                            *reinterpret_cast<TeamShared<int64_t> *>(small_dyn + kTables));
        else
          team_pass<true, int64_t, i128>(s.g, s.a, s.ct, s.lp, s.tau, o.max_iters, s.w.slots, t, small_dyn,
                                         *reinterpret_cast<TeamShared<i128> *>(small_dyn + kTables));
        t.sync();
      } while (small_after(j, o, res, t, ctl));
      small_finish(j, res, t, ctl);
    } else if (j.n == 0 && *(volatile u64 *)&ctl->err == 0) {
      small_finish(j, res, t, ctl);
    }
    t.sync();   // a job may end early, in every block alike; its words are done with
  }
}

// The launch of `blocks` blocks in clusters of `cluster`.
static void small_config(int blocks, int cluster, cudaStream_t s, cudaLaunchAttribute *attr, cudaLaunchConfig_t *cfg) {
  ensure_smem((const void *)small_leiden_k, kSmem);
  ensure_wide_clusters((const void *)small_leiden_k);
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)(blocks / cluster * cluster), 1, 1);
  cfg->blockDim = dim3(TEAM_THREADS, 1, 1);
  cfg->dynamicSmemBytes = kSmem;
  cfg->stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cluster;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

}  // namespace LK_TEAM_SPACE

template <>
int small_max_cluster<LK_TEAM_THREADS>() {
  for (int c = 16; c > 1; c >>= 1) {
    cudaLaunchAttribute attr{};
    cudaLaunchConfig_t cfg;
    small_config(c, c, nullptr, &attr, &cfg);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (const void *)small_leiden_k, &cfg) == cudaSuccess && n > 0) return c;
    (void)cudaGetLastError();
  }
  return 1;
}

template <>
int launch_small<LK_TEAM_THREADS>(SmallHeader *hdr, const SmallJob *jobs, const SmallOpts &o, SmallResult *results,
                                  SmallCtl *ctl, int blocks, int cluster, cudaStream_t s) {
  cudaLaunchAttribute attr{};
  cudaLaunchConfig_t cfg;
  small_config(blocks, cluster, s, &attr, &cfg);
  if (cudaLaunchKernelEx(&cfg, small_leiden_k, hdr, jobs, o, results, ctl) != cudaSuccess) return LEIDEN_ECUDA;
  return LEIDEN_OK;
}

}  // namespace lk
