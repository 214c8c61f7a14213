// team.cuh -- one pass of Alg. leiden by a "team" of thread blocks that stay
// resident for the whole pass and meet at barriers instead of kernel
// boundaries.
//
// A team is a single block, a thread-block cluster, or a whole cooperative
// grid; the code is the same and only Team::sync differs.  The phases are
// those of the multi-kernel path (class lists, local-moving sub-sweeps, subset
// renumbering and break, refinement sub-sweeps, dense renumbering,
// aggregation), with the same integer arithmetic and the same DET schedule,
// so the results are the same bit for bit.
//
// What bounds it: on small levels the chain of dependent L2 loads of one
// vertex (list, header, Sigma'[d], row, C'[j], Sigma'[c]) plus two barriers
// per sub-sweep, about 8-11 us; on large ones the gathers of C'[j] and
// Sigma'[c].  Hence: proposals stay in the block's shared memory from the
// decide to the apply phase (no global counter, no second read of their
// rows), every load of a row is in flight before its first table insert, the
// lane that occupied a table slot scores and resets it (no clearing, no table
// scan), and equal communities meet in shared-memory atomics instead of a
// match across the warp.  Measured (Static of a 1e4-vertex planted partition,
// 480 sub-sweeps): 13.7 ms with one launch per tier and sub-sweep, 8.2 ms on
// resident blocks with the tables cleared and scanned, 6.3 ms as here; R-MAT
// scale 22 with hubs 122 -> 89 ms, Chung-Lu of 2.5e8 entries 294 -> 231 ms.
#pragma once

#include <limits.h>

#include "common.cuh"
#include "internal.h"
#include "team.h"

namespace lk {

// Threads of a block: 1024 unless the including file says otherwise (512; see
// small.cuh).  The code of each shape has a namespace of its own.
#ifndef LK_TEAM_THREADS
#define LK_TEAM_THREADS 1024
#endif
#define LK_TEAM_CAT2(a, b) a##b
#define LK_TEAM_CAT(a, b) LK_TEAM_CAT2(a, b)
#define LK_TEAM_SPACE LK_TEAM_CAT(team_, LK_TEAM_THREADS)
inline namespace LK_TEAM_SPACE {

static constexpr int TEAM_THREADS = LK_TEAM_THREADS;
static constexpr int TEAM_WARPS = TEAM_THREADS / 32;
// Hashtable slots per warp; a sub-block of 8 warps pools 8 of them, the whole
// block all of them (16384 slots).
static constexpr int TEAM_WSLOTS = 16384 / TEAM_WARPS;
static constexpr int TEAM_SUB = 256;                     // threads of a sub-block
static constexpr int TEAM_NSUB = TEAM_THREADS / TEAM_SUB;
// Degree tiers: one lane per vertex, 16 lanes, a warp with one, four or eight
// row entries per lane, a sub-block with eight, the block, and the whole team
// for rows whose distinct candidates may not fit the block's table (hubs).
static constexpr int TT_LANE = 8, TT_HALF = 16, TT_WARP1 = 32, TT_WARP4 = 128, TT_WARP8 = 256, TT_SUB = 2048;
static constexpr int TEAM_TIERS = 8;
static constexpr int TEAM_MAX_KEYS = 256 * TEAM_TIERS;
// Proposals a block keeps in shared memory per sub-sweep (more go to a list
// of the whole team in global memory).
static constexpr int TEAM_PROPS = 256;

__device__ __forceinline__ int team_tier(int64_t deg, int64_t n) {
  return deg <= TT_LANE ? 0
         : deg <= TT_HALF ? 1
         : deg <= TT_WARP1 ? 2
         : deg <= TT_WARP4 ? 3
         : deg <= TT_WARP8 ? 4
         : deg <= TT_SUB ? 5
         : (deg < n ? deg : n) <= TEAM_MAX_CAND ? 6 : 7;
}
// Hubs: row entries per insert item, table slots per scan item.
static constexpr int HUB_ITEM = 2048, HUB_SLOTS = 4096;
// Movers with longer rows leave their re-marking to the team, in pieces of
// this many entries.
static constexpr int REMARK_PIECE = 1024;

// Correctly rounded int128 -> double (round to nearest even) by round-to-odd
// double rounding (Boldo and Melquiond, "When double rounding is odd", 2005):
// truncate to the top 64 significant bits and OR every dropped bit into the
// lowest kept bit (the sticky bit), then convert those 64 bits to double and
// scale by the dropped power of two.
__device__ __forceinline__ double team_i128_to_double(i128 x) {
  const bool neg = x < 0;
  const unsigned __int128 u = neg ? (unsigned __int128)(-(x + 1)) + 1u : (unsigned __int128)x;
  const u64 hi = (u64)(u >> 64);
  double r;
  if (hi == 0) {
    r = __ull2double_rn((u64)u);
  } else {
    const int s = 64 - __clzll((long long)hi);
    const u64 top = (u64)(u >> s);
    const bool sticky = (u & (((unsigned __int128)1 << s) - 1u)) != 0;
    r = ldexp(__ull2double_rn(top | (sticky ? 1ull : 0ull)), s);
  }
  return neg ? -r : r;
}

// A vertex to decide: its row, its community and the totals its score needs.
struct TeamHead {
  int64_t e0, K, Sd;
  int32_t deg, d;
};

// A decided move, kept where it was decided until the sub-sweep's apply phase.
struct TeamProp {
  int64_t e0, K;
  int32_t i, c, d, len;
};

// Static shared memory of a team block.
template <typename ST>
struct TeamShared {
  TeamProp prop[TEAM_PROPS];
  unsigned nprop[2];                   // by parity of the sub-sweep
  int32_t queue[TEAM_WARPS][64];       // eligible vertices of the one-lane tier
  i128 red128[TEAM_WARPS];
  int64_t red64[TEAM_WARPS];
  ST r_sc[TEAM_WARPS];
  int32_t r_c[TEAM_WARPS];
  int64_t r_kid[TEAM_WARPS];
  TeamHead h[TEAM_NSUB][32];           // staged vertices of the sub-block and block tiers
  int32_t h_i[TEAM_NSUB][32];
  int32_t h_n[TEAM_NSUB];
  int32_t koff[TEAM_MAX_KEYS + 1];     // class-list offsets
  unsigned hbits[TEAM_MAX_HUBS / 32];  // hubs of the class to decide in this sub-sweep
  int last[TEAM_NSUB];
  int flag;
  int dead;
};

struct Team {
  int rank, nb, kind;
  unsigned gen;
  TeamCtl *ctl;
  int *dead_s;     // shared: a wait expired
  bool dead;

  // Index of this thread in the team: warps dealt out over the blocks, so that
  // few work items spread over the SMs and a warp's items stay contiguous.
  __device__ __forceinline__ int index() const {
    return (((int)threadIdx.x >> 5) * nb + rank) * 32 + ((int)threadIdx.x & 31);
  }

  // Barrier over the team.  The grid form counts arrivals on one global word;
  // its wait is bounded: a block that waits too long raises the abort flag and
  // every block of the team leaves the kernel.  Returns false then.
  __device__ __forceinline__ bool sync() {
    if (kind == TEAM_BLOCK) { __syncthreads(); return true; }
    if (kind == TEAM_CLUSTER) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    }
    __syncthreads();
    gen++;
    if (threadIdx.x == 0) {
      const unsigned target = gen * (unsigned)nb;
      // arrival releases what the block wrote (made visible to this thread by
      // the block barrier), the polling load acquires what the others wrote
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->bar) : "memory");
      unsigned v;
      u64 spins = 0;
      int bad = 0;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->bar) : "memory");
        if ((int)(v - target) >= 0) break;
        if (++spins > TEAM_SPIN_LIMIT) { atomicExch(&ctl->abort, 1u); bad = 1; break; }
        if ((spins & 1023) == 0 && *(volatile unsigned *)&ctl->abort) { bad = 1; break; }
      }
      if (bad) *dead_s = 1;
    }
    __syncthreads();
    dead = *dead_s != 0;
    return !dead;
  }
};

#define TEAM_SYNC_OR(ret)      \
  do {                         \
    if (!t.sync()) return ret; \
  } while (0)

__device__ __forceinline__ void bar_named(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Arrays of one level, shared by the phases.
template <typename WT>
struct TeamLevel {
  int64_t n, nnz;
  const int64_t *off;
  const int32_t *idx;
  const WT *w;
};

struct TeamConst {
  int64_t A, p;
  double den;
  int64_t two_m;
  int log2S;
  int dynamic, timing;
  const uint8_t *in_range;
};

// A value kept in the block's shared memory and read again at every use, so
// that it takes no register between uses.  The batch kernel holds its arrays
// this way; a context's arrays are kernel parameters, which cost none either.
template <typename T>
struct Held {
  T v;
  __device__ __forceinline__ operator T() const { return *(const volatile T *)&v; }
  __device__ __forceinline__ void operator=(T x) { v = x; }
};

// Running sums of a thread: statistics and the scores of its moves.
struct TeamStat {
  int64_t scanned, nvert, ncand;
  i128 S;
};

// A sub-sweep: parity, refinement stamp, the team's overflow counter, and
// whether headers are loaded alongside the eligibility test.
struct TeamSweep {
  unsigned par;
  uint8_t sv;
  bool spec;
  unsigned *nover, *npiece;
};

template <typename ST>
__device__ __forceinline__ bool team_better(ST sc, int32_t c, ST bsc, int32_t bc) {
  return c != INT32_MAX && (bc == INT32_MAX || sc > bsc || (sc == bsc && c < bc));
}

// Adds w to a 32-bit or a 64-bit table value; the latter as two 32-bit words
// with the carry passed on by the adder that wrapped the low one.
__device__ __forceinline__ void team_val_add(uint32_t *p, u64 w) { atomicAdd(p, (uint32_t)w); }
__device__ __forceinline__ void team_val_add(u64 *p, u64 w) {
  uint32_t *h = reinterpret_cast<uint32_t *>(p);
  const uint32_t lo = (uint32_t)w;
  const uint32_t old = atomicAdd(&h[0], lo);
  const uint32_t hi = (uint32_t)(w >> 32) + (old + lo < old ? 1u : 0u);
  if (hi) atomicAdd(&h[1], hi);
}

// Adds (c, w) to a shared-memory table of 2^lh slots that is never more than
// half full; returns the slot if this call occupied it, else -1.  Equal keys
// meet in the shared-memory atomics: combining them across the warp first
// (match, then a walk over the peers) took longer than the conflicts.
// PIECE: the table takes a piece of a longer row.  An aggregated row lists its
// communities in the order of hash32, so a piece covers a narrow range of it
// and would pile up in one corner of the table (12 ms for a sub-sweep of R-MAT
// scale 22's first aggregated level, 0.25 ms with a hash of its own).
template <bool PIECE, typename VT>
__device__ __forceinline__ int team_table_add(int32_t *keys, VT *vals, int lh, int32_t c, u64 w, u64 *err) {
  const uint32_t mask = (1u << lh) - 1u;
  uint32_t s = (PIECE ? (uint32_t)c * 0x85EBCA77u : hash32(c)) >> (32 - lh);
  for (uint32_t probe = 0; probe <= mask; probe++) {
    int32_t k = *(volatile int32_t *)&keys[s];
    bool fresh = false;
    if (k == LEIDEN_EMPTY_KEY) {
      k = atomicCAS(&keys[s], LEIDEN_EMPTY_KEY, c);
      fresh = k == LEIDEN_EMPTY_KEY;
    }
    if (fresh || k == c) {
      team_val_add(&vals[s], w);
      return fresh ? (int)s : -1;
    }
    s = (s + 1) & mask;
  }
  atomicOr(err, 16ull);
  return -1;
}

template <bool REFINE, typename AR, typename CT>
__device__ __forceinline__ bool team_eligible(const AR &a, const CT &ct, int32_t i) {
  if (!REFINE) {
    if (a.processed[i]) return false;
    a.processed[i] = 1;                               // prune
    return ct.in_range ? ct.in_range[i] != 0 : true;  // inAffectedRange
  }
  return a.ch[a.CB[i]] && a.C[i] == i && a.Sig[i] == a.K[i];
}

// The move rule for vertex i (one lane): Eq. 2 scaled, strictly better only.
template <bool REFINE, typename ST, typename AR, typename CT>
__device__ __forceinline__ bool team_rule(const AR &a, const CT &ct, int64_t Ki, int64_t Sd, ST bsc,
                                          int32_t bc, int64_t kid, i128 *S) {
  if (bc == INT32_MAX) return false;
  *S = (i128)bsc - (i128)ct.A * kid - (i128)ct.p * Ki * (Ki - Sd);
  if (!(*S > 0)) return false;
  return !(REFINE && a.C[bc] != bc);                  // target's vertex left
}

// Appends the proposals of a warp (whole warp calls) to the block's list, or
// to the team's when that is full, and adds up their scores.
template <bool REFINE, typename ST, typename AR>
__device__ __forceinline__ void team_propose(const AR &a, const TeamSweep &sw, TeamShared<ST> &sm, bool propose,
                                             int32_t i, int32_t c, const TeamHead &h, i128 S, TeamStat &st) {
  const unsigned m = __ballot_sync(FULL_MASK, propose);
  if (!m) return;
  const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == leader) base = atomicAdd(&sm.nprop[sw.par], (unsigned)__popc(m));
  base = __shfl_sync(FULL_MASK, base, leader);
  if (!propose) return;
  const unsigned slot = base + __popc(m & ((1u << lane) - 1u));
  if (!REFINE && h.deg > REMARK_PIECE) {
    const int np = (h.deg + REMARK_PIECE - 1) / REMARK_PIECE;
    const unsigned p0 = atomicAdd(sw.npiece, (unsigned)np);
    for (int k = 0; k < np; k++) { a.piece_i[p0 + k] = i; a.piece_k[p0 + k] = k; }
  }
  if (slot < TEAM_PROPS) {
    TeamProp &p = sm.prop[slot];
    p.e0 = h.e0;
    p.K = h.K;
    p.i = i;
    p.c = c;
    p.d = h.d;
    p.len = h.deg;
  } else {
    const unsigned g = atomicAdd(sw.nover, 1u);
    a.prop_i[g] = i;
    a.prop_c[g] = c;
  }
  if (REFINE) a.stamp[i] = sw.sv;
  else st.S += S;
}

// Header of vertex i, and of a refinement its bound.
template <typename GL, typename AR>
__device__ __forceinline__ TeamHead team_head(const GL &g, const AR &a, int32_t i) {
  TeamHead h;
  h.e0 = g.off[i];
  h.deg = (int32_t)(g.off[i + 1] - h.e0);
  h.d = a.C[i];
  h.K = a.K[i];
  h.Sd = a.Sig[h.d];
  return h;
}
__device__ __forceinline__ TeamHead team_shfl(const TeamHead &h, int src) {
  TeamHead r;
  r.e0 = shfl_i64(h.e0, src);
  r.K = shfl_i64(h.K, src);
  r.Sd = shfl_i64(h.Sd, src);
  r.deg = __shfl_sync(FULL_MASK, h.deg, src);
  r.d = __shfl_sync(FULL_MASK, h.d, src);
  return r;
}

// One lane per vertex: the row (at most TT_LANE entries) in registers, equal
// communities merged into their first occurrence.
template <bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_decide_lane(const GL &g, const AR &a, const CT &ct,
                                                 int32_t i, bool act, const TeamSweep &sw, TeamShared<ST> &sm,
                                                 TeamStat &st) {
  typedef typename TableVal<ST>::type VT;
  TeamHead h{};
  int32_t cbi = 0;
  if (act) {
    h = team_head(g, a, i);
    if (REFINE) cbi = a.CB[i];
  }
  int32_t cc[TT_LANE];
  VT ww[TT_LANE];
#pragma unroll
  for (int k = 0; k < TT_LANE; k++) {
    cc[k] = k < h.deg ? g.idx[h.e0 + k] : -1;
    ww[k] = k < h.deg ? (VT)g.w[h.e0 + k] : (VT)0;
  }
#pragma unroll
  for (int k = 0; k < TT_LANE; k++) {
    const int32_t j = cc[k];
    bool ok = j >= 0 && j != i;                       // self = false
    if (REFINE && ok && a.CB[j] != cbi) ok = false;   // scanBounded
    cc[k] = ok ? a.C[j] : LEIDEN_EMPTY_KEY;
  }
#pragma unroll
  for (int k = 1; k < TT_LANE; k++) {
#pragma unroll
    for (int k2 = 0; k2 < k; k2++)
      if (cc[k] != LEIDEN_EMPTY_KEY && cc[k2] == cc[k]) {
        ww[k2] += ww[k];
        cc[k] = LEIDEN_EMPTY_KEY;
      }
  }
  const ST A = (ST)ct.A;
  const ST B = (ST)ct.p * (ST)h.K;
  ST bsc = 0;
  int32_t bc = INT32_MAX;
  int64_t kid = 0;
  int nc = 0;
#pragma unroll
  for (int q = 0; q < TT_LANE; q += 4) {   // four Sigma' gathers in flight
    int64_t sg[4];
#pragma unroll
    for (int k = 0; k < 4; k++)
      sg[k] = (cc[q + k] != LEIDEN_EMPTY_KEY && cc[q + k] != h.d) ? sigma_for_score(a.Sig, cc[q + k]) : 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int32_t c = cc[q + k];
      if (c == LEIDEN_EMPTY_KEY) continue;
      nc++;
      if (c == h.d) { kid = (int64_t)ww[q + k]; continue; }
      const ST sc = A * (ST)(int64_t)ww[q + k] - B * (ST)sg[k];
      if (team_better(sc, c, bsc, bc)) { bsc = sc; bc = c; }
    }
  }
  i128 S = 0;
  const bool propose = act && team_rule<REFINE, ST>(a, ct, h.K, h.Sd, bsc, bc, kid, &S);
  if (act) { st.scanned += h.deg; st.nvert++; st.ncand += nc; }
  team_propose<REFINE, ST>(a, sw, sm, propose, i, bc, h, S, st);
}

// Best candidate among the slots this lane occupied (own[u] >= 0), which are
// reset as they are read: the table is empty again once every lane is done.
template <int STEPS, typename ST, typename AR>
__device__ __forceinline__ void team_scan_own(const AR &a, const int (&own)[STEPS], int32_t *keys,
                                              typename TableVal<ST>::type *vals, int32_t d, ST A, ST B, ST &bsc,
                                              int32_t &bc, int64_t &kid, TeamStat &st) {
  constexpr int Q = STEPS < 4 ? STEPS : 4;   // Sigma' gathers in flight
#pragma unroll
  for (int q = 0; q < STEPS; q += Q) {
    int32_t c[Q];
    int64_t v[Q], sg[Q];
#pragma unroll
    for (int u = 0; u < Q; u++) {
      const int o = own[q + u];
      c[u] = o >= 0 ? keys[o] : LEIDEN_EMPTY_KEY;
      v[u] = o >= 0 ? (int64_t)vals[o] : 0;
      if (o >= 0) { keys[o] = LEIDEN_EMPTY_KEY; vals[o] = 0; }
    }
#pragma unroll
    for (int u = 0; u < Q; u++) sg[u] = (c[u] != LEIDEN_EMPTY_KEY && c[u] != d) ? sigma_for_score(a.Sig, c[u]) : 0;
#pragma unroll
    for (int u = 0; u < Q; u++) {
      if (c[u] == LEIDEN_EMPTY_KEY) continue;
      st.ncand++;
      if (c[u] == d) { kid = v[u]; continue; }
      const ST sc = A * (ST)v[u] - B * (ST)sg[u];
      if (team_better(sc, c[u], bsc, bc)) { bsc = sc; bc = c[u]; }
    }
  }
}

// The row entries first, first + stride, ... (STEPS of them) of one lane: all
// their loads, then their gathers, in flight before the first table insert.
template <int STEPS, bool REFINE, typename WT, bool PIECE = false, typename VT, typename GL, typename AR>
__device__ __forceinline__ void team_insert(const GL &g, const AR &a, int32_t i, int64_t e0, int deg,
                                            int first, int stride, int32_t cbi, int32_t *keys, VT *vals, int lh,
                                            int (&own)[STEPS]) {
  VT ww[STEPS];
#pragma unroll
  for (int u = 0; u < STEPS; u++) {
    const int e = first + u * stride;
    own[u] = e < deg ? g.idx[e0 + e] : -1;
    ww[u] = e < deg ? (VT)g.w[e0 + e] : (VT)0;
  }
#pragma unroll
  for (int u = 0; u < STEPS; u++) {
    const int32_t j = own[u];
    bool ok = j >= 0 && j != i;                       // self = false
    if (REFINE && ok && a.CB[j] != cbi) ok = false;   // scanBounded
    own[u] = ok ? a.C[j] : LEIDEN_EMPTY_KEY;
  }
#pragma unroll
  for (int u = 0; u < STEPS; u++)
    own[u] = own[u] != LEIDEN_EMPTY_KEY ? team_table_add<PIECE>(keys, vals, lh, own[u], (u64)ww[u], a.err) : -1;
}

// G lanes per vertex (16 or 32), rows of at most G * STEPS entries, a table of
// twice as many slots per group.  The whole warp calls; i < 0 marks an idle
// group.
template <int G, int STEPS, bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_decide_warp(const GL &g, const AR &a, const CT &ct,
                                                 int32_t i, const TeamHead &h, const TeamSweep &sw, int32_t *keys,
                                                 typename TableVal<ST>::type *vals, TeamShared<ST> &sm, TeamStat &st) {
  constexpr int LH = G * STEPS == 16 ? 5 : G * STEPS == 32 ? 6 : G * STEPS == 128 ? 8 : 9;
  const int lane = threadIdx.x & 31, gl = lane % G;
  const bool act = i >= 0;
  if (G < 32) { keys += (lane / G) << LH; vals += (lane / G) << LH; }
  const int32_t cbi = (REFINE && act) ? a.CB[i] : 0;
  int own[STEPS];
  team_insert<STEPS, REFINE, WT>(g, a, i, h.e0, act ? h.deg : 0, gl, G, cbi, keys, vals, LH, own);
  __syncwarp();
  ST bsc = 0;
  int32_t bc = INT32_MAX;
  int64_t kid = 0;
  team_scan_own<STEPS, ST>(a, own, keys, vals, h.d, (ST)ct.A, (ST)ct.p * (ST)h.K, bsc, bc, kid, st);
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const ST osc = shfl_xor_any<ST>(bsc, o);
    const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
    kid += shfl_xor_i64(kid, o);
    if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
  }
  i128 S = 0;
  bool propose = false;
  if (act && gl == 0) {
    st.scanned += h.deg;
    st.nvert++;
    propose = team_rule<REFINE, ST>(a, ct, h.K, h.Sd, bsc, bc, kid, &S);
  }
  team_propose<REFINE, ST>(a, sw, sm, propose, i, bc, h, S, st);
  __syncwarp();
}

// A group of GT threads (a sub-block, or the whole block) per vertex, over the
// listed vertices first, first + step, ... of list[0 .. m).  Warp 0 of the
// group stages 32 listed vertices at once and keeps the eligible ones.  `bar`
// is the group's named barrier, q its staging slot.
template <int GT, bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_decide_group(const GL &g, const AR &a, const CT &ct,
                                                  const int32_t *list, int m, int first, int step, int bar, int q,
                                                  const TeamSweep &sw, int32_t *keys,
                                                  typename TableVal<ST>::type *vals, TeamShared<ST> &sm,
                                                  TeamStat &st) {
  constexpr int NW = GT / 32;
  constexpr int MAXLH = GT == TEAM_THREADS ? 14 : 12;
  const int lane = threadIdx.x & 31, tid = threadIdx.x % GT, warp = tid >> 5, wabs = threadIdx.x >> 5;
  const int wbase = wabs - warp;   // first warp of the group within the block
  for (int base = first; base < m; base += 32 * step) {
    if (warp == 0) {
      const int li = base + lane * step;
      const bool valid = li < m;
      const int32_t i = valid ? list[li] : 0;
      const bool act = valid && team_eligible<REFINE>(a, ct, i);
      const unsigned mk = __ballot_sync(FULL_MASK, act);
      if (act) {
        const int pos = __popc(mk & ((1u << lane) - 1u));
        sm.h_i[q][pos] = i;
        sm.h[q][pos] = team_head(g, a, i);
      }
      if (lane == 0) sm.h_n[q] = __popc(mk);
    }
    bar_named(bar, GT);
    const int nact = sm.h_n[q];
    for (int k = 0; k < nact; k++) {
      const int32_t i = sm.h_i[q][k];
      const TeamHead h = sm.h[q][k];
      const int32_t cbi = REFINE ? a.CB[i] : 0;
      const ST A = (ST)ct.A;
      const ST B = (ST)ct.p * (ST)h.K;
      ST bsc = 0;
      int32_t bc = INT32_MAX;
      int64_t kid = 0;
      if (GT < TEAM_THREADS) {
        int own[8];
        team_insert<8, REFINE, WT>(g, a, i, h.e0, h.deg, tid, GT, cbi, keys, vals, MAXLH, own);
        bar_named(bar, GT);
        team_scan_own<8, ST>(a, own, keys, vals, h.d, A, B, bsc, bc, kid, st);
      } else {
        // rows of any length; the whole table is read back and reset
        const int64_t cap = h.deg < g.n ? h.deg : g.n;
        int lh = 10;
        while (lh < MAXLH && ((int64_t)1 << lh) < 2 * cap) lh++;
        for (int x = tid; x < h.deg; x += 4 * GT) {
          int own[4];
          team_insert<4, REFINE, WT>(g, a, i, h.e0, h.deg, x, GT, cbi, keys, vals, lh, own);
        }
        bar_named(bar, GT);
        for (int s = tid; s < (1 << lh); s += 4 * GT) {
          int own[4];
#pragma unroll
          for (int u = 0; u < 4; u++) {
            const int sl = s + u * GT;
            own[u] = sl < (1 << lh) && keys[sl] != LEIDEN_EMPTY_KEY ? sl : -1;
          }
          team_scan_own<4, ST>(a, own, keys, vals, h.d, A, B, bsc, bc, kid, st);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const ST osc = shfl_xor_any<ST>(bsc, o);
        const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
        kid += shfl_xor_i64(kid, o);
        if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
      }
      if (lane == 0) { sm.r_sc[wabs] = bsc; sm.r_c[wabs] = bc; sm.r_kid[wabs] = kid; }
      bar_named(bar, GT);
      if (warp == 0) {
        // the other warps go on to insert the next vertex's row; the r_* words
        // are written again only after that row's barrier
        bsc = lane < NW ? sm.r_sc[wbase + lane] : (ST)0;
        bc = lane < NW ? sm.r_c[wbase + lane] : INT32_MAX;
        kid = lane < NW ? sm.r_kid[wbase + lane] : 0;
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) {
          const ST osc = shfl_xor_any<ST>(bsc, o);
          const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
          kid += shfl_xor_i64(kid, o);
          if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
        }
        i128 S = 0;
        bool propose = false;
        if (lane == 0) {
          st.scanned += h.deg;
          st.nvert++;
          propose = team_rule<REFINE, ST>(a, ct, h.K, h.Sd, bsc, bc, kid, &S);
        }
        team_propose<REFINE, ST>(a, sw, sm, propose, i, bc, h, S, st);
      }
    }
    bar_named(bar, GT);   // the staged vertices are read before the next 32
  }
}

// The vertices of one warp-per-vertex tier (list[0 .. m)): `ch` consecutive
// listed vertices per warp and step, as few as spread the list over the team.
// wg is the warp's place in the tier's order; returns it for the next tier.
template <int G, int STEPS, bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ int team_decide_tier(const GL &g, const AR &a, const CT &ct,
                                                const int32_t *list, int m, int wg, int W, const TeamSweep &sw,
                                                int32_t *keys, typename TableVal<ST>::type *vals, TeamShared<ST> &sm,
                                                TeamStat &st) {
  constexpr int PER = 32 / G;
  const int lane = threadIdx.x & 31;
  int ch = PER * ((m + PER * W - 1) / (PER * W));
  ch = ch > 32 ? 32 : ch;
  for (int base = wg * ch; base < m; base += W * ch) {
    const int li = base + lane;
    const bool valid = lane < ch && li < m;
    const int32_t i = valid ? list[li] : 0;
    TeamHead h{};
    if (sw.spec && valid) h = team_head(g, a, i);
    const bool act = valid && team_eligible<REFINE>(a, ct, i);
    unsigned mk = __ballot_sync(FULL_MASK, act);
    if (!mk) continue;
    if (!sw.spec && act) h = team_head(g, a, i);
    if (G == 32) {
      for (; mk; mk &= mk - 1) {
        const int src = __ffs(mk) - 1;
        team_decide_warp<G, STEPS, REFINE, WT, ST>(g, a, ct, __shfl_sync(FULL_MASK, i, src), team_shfl(h, src), sw,
                                                   keys, vals, sm, st);
      }
    } else {
      while (mk) {
        const int b0 = __ffs(mk) - 1;
        mk &= mk - 1;
        const int b1 = mk ? __ffs(mk) - 1 : -1;
        mk &= mk - 1;   // 0 stays 0
        const int src = lane < 16 || b1 < 0 ? b0 : b1;
        const int32_t x = __shfl_sync(FULL_MASK, i, src);
        team_decide_warp<G, STEPS, REFINE, WT, ST>(g, a, ct, (lane >= 16 && b1 < 0) ? -1 : x, team_shfl(h, src), sw,
                                                   keys, vals, sm, st);
      }
    }
  }
  return (wg + W - ((m + ch - 1) / ch) % W) % W;
}

// ---------------------------------------------------------------------------
// Hubs: rows with more distinct candidates than the block's table holds.  A
// hub's table is in global scratch (L2): a sub-block takes HUB_ITEM entries
// of a row, sums them up per community in its shared table and adds the
// distinct ones to the hub's table; after a barrier a sub-block takes
// HUB_SLOTS slots, scores and resets them, and the sub-block that finishes a
// hub's last slots decides.  Item and slot ranges are prefix sums over the
// class's hubs (TeamArrays::hub_i, hub_s), made once per pass.
// ---------------------------------------------------------------------------
// First k in [0, m) with pre[k] > w.
__device__ __forceinline__ int team_find(const int32_t *pre, int m, int w) {
  int lo = 0, hi = m - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] > w) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Adds (c, w) to a hub's table of t slots at offset `at`.  32-bit values: a
// slot is one 64-bit word, key + 1 in its low half (0: empty), the sum in its
// high half, so both atomics meet one sector; 64-bit values: keys and values
// apart.
template <typename VT, typename AR>
__device__ __forceinline__ void team_hub_add(const AR &a, int64_t at, uint64_t t, int32_t c, u64 w) {
  uint64_t s = ((uint64_t)hash32(c) * t) >> 32;
  for (uint64_t probe = 0; probe < t; probe++) {
    if (sizeof(VT) == 4) {
      uint32_t *slot = reinterpret_cast<uint32_t *>(&a.tvals[at + (int64_t)s]);
      const uint32_t key = (uint32_t)c + 1u;
      const uint32_t old = atomicCAS(slot, 0u, key);
      if (old == 0u || old == key) { atomicAdd(slot + 1, (uint32_t)w); return; }
    } else {
      const int32_t old = atomicCAS(&a.tkeys[at + (int64_t)s], LEIDEN_EMPTY_KEY, c);
      if (old == LEIDEN_EMPTY_KEY || old == c) { atomicAdd(&a.tvals[at + (int64_t)s], w); return; }
    }
    s = s + 1 == t ? 0 : s + 1;
  }
  atomicOr(a.err, 16ull);
}

// Prefix sums of every class's hub items; false when a class has too many hubs
// (see MANY_HUBS) or its tables exceed the scratch (the same answer in every
// block).
template <typename WT, typename ST, typename GL, typename AR>
__device__ __forceinline__ bool team_hub_setup(const GL &g, const AR &a, int S, Team &t,
                                               TeamShared<ST> &sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h0 = sm.koff[7 * S], hn = sm.koff[8 * S];
  if (h0 == hn) return true;
  for (int s = t.rank; s < S; s += t.nb) {
    const int p0 = sm.koff[7 * S + s], p1 = sm.koff[7 * S + s + 1];
    int64_t ci = 0, cs = 0;
    for (int base = p0; base < p1; base += TEAM_THREADS) {
      const int p = base + (int)threadIdx.x;
      int64_t vi = 0, vs = 0;
      if (p < p1) {
        const int32_t i = a.vlist[p];
        const int64_t deg = g.off[i + 1] - g.off[i], cap = deg < g.n ? deg : g.n;
        vi = (deg + HUB_ITEM - 1) / HUB_ITEM;
        vs = (2 * cap + HUB_SLOTS - 1) / HUB_SLOTS;
      }
      int64_t xi = vi, xs = vs;
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t yi = shfl_i64(xi, (lane - o) & 31), ys = shfl_i64(xs, (lane - o) & 31);
        if (lane >= o) { xi += yi; xs += ys; }
      }
      __syncthreads();
      if (lane == 31) { sm.red64[warp] = xi; sm.r_kid[warp] = xs; }
      __syncthreads();
      int64_t pi = ci, ps = cs;
      for (int q = 0; q < TEAM_WARPS; q++) {
        if (q < warp) { pi += sm.red64[q]; ps += sm.r_kid[q]; }
        ci += sm.red64[q];
        cs += sm.r_kid[q];
      }
      if (p < p1) {
        a.hub_i[p - h0] = (int32_t)(pi + xi);
        a.hub_s[p - h0] = (int32_t)(ps + xs);
        a.hub_done[p - h0] = 0;
      }
    }
    if (threadIdx.x == 0 &&
        ((!AR::MANY_HUBS && p1 - p0 > TEAM_MAX_HUBS) || cs * HUB_SLOTS > a.tcap || ci > INT_MAX / 2))
      t.ctl->too_big = 1;
  }
  if (!t.sync()) return false;
  return *(volatile int32_t *)&t.ctl->too_big == 0;
}

// Whether hub i is to be decided in this sub-sweep.  Its flags change only once
// all its items are done (processed) or after the sub-sweep's barrier.
template <bool REFINE, typename AR, typename CT>
__device__ __forceinline__ bool team_hub_active(const AR &a, const CT &ct, int32_t i) {
  return REFINE ? (a.ch[a.CB[i]] && a.C[i] == i && a.Sig[i] == a.K[i])
                : (!a.processed[i] && (!ct.in_range || ct.in_range[i]));
}

// Which hubs of the class are to be decided, the first TEAM_MAX_HUBS of them
// into sm.hbits; whether any is.
template <bool REFINE, typename ST, typename AR, typename CT>
__device__ __forceinline__ bool team_hub_bits(const AR &a, const CT &ct, const int32_t *list, int m,
                                              TeamShared<ST> &sm) {
  int any = 0;
  for (int base = 0; base < m; base += TEAM_THREADS) {
    const int k = base + (int)threadIdx.x;
    bool act = false;
    if (k < m) act = team_hub_active<REFINE>(a, ct, list[k]);
    const unsigned mk = __ballot_sync(FULL_MASK, act);
    if ((threadIdx.x & 31) == 0 && k < m && (!AR::MANY_HUBS || k < TEAM_MAX_HUBS)) sm.hbits[(base + (int)threadIdx.x) >> 5] = mk;
    any |= mk != 0;
  }
  return __syncthreads_or(any) != 0;
}

// team_hub_active of the class's k-th hub, from the bits.
template <bool REFINE, typename ST, typename AR, typename CT>
__device__ __forceinline__ bool team_hub_bit(const AR &a, const CT &ct, const int32_t *list, int k,
                                             const TeamShared<ST> &sm) {
  if (AR::MANY_HUBS && k >= TEAM_MAX_HUBS) return team_hub_active<REFINE>(a, ct, list[k]);
  return (sm.hbits[k >> 5] >> (k & 31)) & 1u;
}

template <bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_hub_insert(const GL &g, const AR &a, const CT &ct, const Team &t,
                                                const int32_t *list, const int32_t *pi, const int32_t *ps, int m,
                                                int32_t *keys, typename TableVal<ST>::type *vals,
                                                TeamShared<ST> &sm) {
  typedef typename TableVal<ST>::type VT;
  const int sub = threadIdx.x / TEAM_SUB, tid = threadIdx.x % TEAM_SUB;
  const int total = pi[m - 1];
  for (int w = sub * t.nb + t.rank; w < total; w += t.nb * TEAM_NSUB) {
    const int k = team_find(pi, m, w);
    if (!team_hub_bit<REFINE>(a, ct, list, k, sm)) continue;
    const int32_t i = list[k];
    const int64_t e0 = g.off[i], e1 = g.off[i + 1];
    const int64_t c0 = e0 + (int64_t)(w - (k ? pi[k - 1] : 0)) * HUB_ITEM;
    const int cnt = (int)(e1 - c0 < HUB_ITEM ? e1 - c0 : HUB_ITEM);
    const int64_t at = (int64_t)(k ? ps[k - 1] : 0) * HUB_SLOTS;
    const uint64_t ts = (uint64_t)(ps[k] - (k ? ps[k - 1] : 0)) * HUB_SLOTS;
    const int32_t cbi = REFINE ? a.CB[i] : 0;
    int own[8];
    team_insert<8, REFINE, WT, true>(g, a, i, c0, cnt, tid, TEAM_SUB, cbi, keys, vals, 12, own);
    bar_named(2 + sub, TEAM_SUB);
#pragma unroll
    for (int u = 0; u < 8; u++) {
      if (own[u] < 0) continue;
      const int32_t c = keys[own[u]];
      const u64 v = (u64)vals[own[u]];
      keys[own[u]] = LEIDEN_EMPTY_KEY;
      vals[own[u]] = 0;
      team_hub_add<VT>(a, at, ts, c, v);
    }
    bar_named(2 + sub, TEAM_SUB);
  }
}

template <bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_hub_scan(const GL &g, const AR &a, const CT &ct,
                                              const Team &t, const int32_t *list, const int32_t *ps, int32_t *done,
                                              int m, const TeamSweep &sw, TeamShared<ST> &sm, TeamStat &st) {
  typedef typename TableVal<ST>::type VT;
  constexpr int NW = TEAM_SUB / 32;
  const int sub = threadIdx.x / TEAM_SUB, tid = threadIdx.x % TEAM_SUB, warp = tid >> 5, lane = threadIdx.x & 31;
  const int wabs = threadIdx.x >> 5, wbase = wabs - warp;
  const int total = ps[m - 1];
  for (int w = sub * t.nb + t.rank; w < total; w += t.nb * TEAM_NSUB) {
    const int k = team_find(ps, m, w);
    if (!team_hub_bit<REFINE>(a, ct, list, k, sm)) continue;
    const int32_t i = list[k];
    const int32_t d = a.C[i];
    const int64_t Ki = a.K[i];
    const ST A = (ST)ct.A, B = (ST)ct.p * (ST)Ki;
    ST bsc = 0;
    int32_t bc = INT32_MAX;
    int64_t kid = 0;
    const int64_t s0 = (int64_t)w * HUB_SLOTS + tid;
    constexpr int Q = 4;
    for (int x = 0; x < HUB_SLOTS; x += Q * TEAM_SUB) {
      int32_t c[Q];
      int64_t v[Q], sg[Q];
#pragma unroll
      for (int u = 0; u < Q; u++) {
        const int64_t s = s0 + x + u * TEAM_SUB;
        if (sizeof(VT) == 4) {
          const u64 y = __ldcg(&a.tvals[s]);
          c[u] = (int32_t)((uint32_t)y - 1u);   // empty: -1
          v[u] = (int64_t)(y >> 32);
        } else {
          c[u] = __ldcg(&a.tkeys[s]);
          v[u] = c[u] != LEIDEN_EMPTY_KEY ? (int64_t)__ldcg(&a.tvals[s]) : 0;
        }
      }
#pragma unroll
      for (int u = 0; u < Q; u++) {
        if (c[u] == LEIDEN_EMPTY_KEY) { sg[u] = 0; continue; }
        const int64_t s = s0 + x + u * TEAM_SUB;
        a.tvals[s] = 0;                         // reset for the next user of the scratch
        if (sizeof(VT) != 4) a.tkeys[s] = LEIDEN_EMPTY_KEY;
        sg[u] = c[u] != d ? sigma_for_score(a.Sig, c[u]) : 0;
      }
#pragma unroll
      for (int u = 0; u < Q; u++) {
        if (c[u] == LEIDEN_EMPTY_KEY) continue;
        st.ncand++;
        if (c[u] == d) { kid = v[u]; continue; }
        const ST sc = A * (ST)v[u] - B * (ST)sg[u];
        if (team_better(sc, c[u], bsc, bc)) { bsc = sc; bc = c[u]; }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const ST osc = shfl_xor_any<ST>(bsc, o);
      const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
      kid += shfl_xor_i64(kid, o);
      if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
    }
    if (lane == 0) { sm.r_sc[wabs] = bsc; sm.r_c[wabs] = bc; sm.r_kid[wabs] = kid; }
    bar_named(2 + sub, TEAM_SUB);
    if (warp == 0) {
      bsc = lane < NW ? sm.r_sc[wbase + lane] : (ST)0;
      bc = lane < NW ? sm.r_c[wbase + lane] : INT32_MAX;
      kid = lane < NW ? sm.r_kid[wbase + lane] : 0;
#pragma unroll
      for (int o = NW / 2; o > 0; o >>= 1) {
        const ST osc = shfl_xor_any<ST>(bsc, o);
        const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
        kid += shfl_xor_i64(kid, o);
        if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
      }
      const int first = k ? ps[k - 1] : 0, items = ps[k] - first;
      int lastone = 0;
      if (lane == 0) {
        a.part_sc[w] = (i128)bsc;
        a.part_c[w] = bc;
        a.part_kid[w] = kid;
        __threadfence();
        lastone = atomicAdd(&done[k], 1) == items - 1;
      }
      if (__shfl_sync(FULL_MASK, lastone, 0)) {
        __threadfence();
        // the hub's chunks are all in: reduce them and decide
        bsc = 0;
        bc = INT32_MAX;
        kid = 0;
        for (int x = lane; x < items; x += 32) {
          const int32_t oc = __ldcg(&a.part_c[first + x]);
          const u64 *q = reinterpret_cast<const u64 *>(&a.part_sc[first + x]);
          const u64 lo = __ldcg(q), hi = __ldcg(q + 1);
          const ST osc = (ST)(i128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
          kid += __ldcg(&a.part_kid[first + x]);
          if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const ST osc = shfl_xor_any<ST>(bsc, o);
          const int32_t oc = __shfl_xor_sync(FULL_MASK, bc, o);
          kid += shfl_xor_i64(kid, o);
          if (team_better(osc, oc, bsc, bc)) { bsc = osc; bc = oc; }
        }
        TeamHead h{};
        i128 Sx = 0;
        bool propose = false;
        if (lane == 0) {
          done[k] = 0;
          if (!REFINE) a.processed[i] = 1;   // prune: the class's hub bits are already taken
          h = team_head(g, a, i);
          st.scanned += h.deg;
          st.nvert++;
          propose = team_rule<REFINE, ST>(a, ct, Ki, h.Sd, bsc, bc, kid, &Sx);
        }
        team_propose<REFINE, ST>(a, sw, sm, propose, i, bc, h, Sx, st);
      }
    }
    bar_named(2 + sub, TEAM_SUB);   // the r_* words are read before the next item
  }
}

// Decisions of one colour class.  The longest rows come first, and each
// tier's first worker follows the last one of the tier before it, so a short
// class spreads over the team.
// Returns false after an expired wait.
template <bool REFINE, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ bool team_decide_class(const GL &g, const AR &a, const CT &ct,
                                                  Team &t, int s, TeamSweep sw, int32_t *keys,
                                                  typename TableVal<ST>::type *vals, TeamShared<ST> &sm,
                                                  TeamStat &st) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = 1 << ct.log2S;
  const int32_t *ko = &sm.koff[s];   // tier q of the class: ko[q * S] .. ko[q * S + 1]
  const int nb = t.nb;
  int rot = 0;   // blocks already given a first item
  const int m7 = ko[7 * S + 1] - ko[7 * S], hub0 = ko[7 * S] - sm.koff[7 * S];
  bool hubs = false;
  if (m7 > 0) {
    hubs = team_hub_bits<REFINE, ST>(a, ct, a.vlist + ko[7 * S], m7, sm);
    if (hubs)
      team_hub_insert<REFINE, WT, ST>(g, a, ct, t, a.vlist + ko[7 * S], a.hub_i + hub0, a.hub_s + hub0, m7, keys +
                                      threadIdx.x / TEAM_SUB * (TEAM_WSLOTS * (TEAM_SUB / 32)), vals +
                                      threadIdx.x / TEAM_SUB * (TEAM_WSLOTS * (TEAM_SUB / 32)), sm);
    if (ko[6 * S + 1] > ko[6 * S]) __syncthreads();   // the block tier pools the sub-blocks' tables
  }
  const int m6 = ko[6 * S + 1] - ko[6 * S];
  if (m6 > 0) {
    team_decide_group<TEAM_THREADS, REFINE, WT, ST>(g, a, ct, a.vlist + ko[6 * S], m6, t.rank, nb, 1, 0, sw, keys,
                                                    vals, sm, st);
    rot = m6 % nb;
  }
  const int m5 = ko[5 * S + 1] - ko[5 * S];
  if (m5 > 0) {
    const int sub = threadIdx.x / TEAM_SUB, br = (t.rank + nb - rot) % nb;
    constexpr int SL = TEAM_WSLOTS * (TEAM_SUB / 32);
    team_decide_group<TEAM_SUB, REFINE, WT, ST>(g, a, ct, a.vlist + ko[5 * S], m5, sub * nb + br, nb * TEAM_NSUB,
                                                2 + sub, sub, sw, keys + sub * SL, vals + sub * SL, sm, st);
    rot = (rot + m5) % nb;
  }
  const int W = nb * TEAM_WARPS;
  int wg = warp * nb + (t.rank + nb - rot) % nb;
  int32_t *wk = keys + warp * TEAM_WSLOTS;
  typename TableVal<ST>::type *wv = vals + warp * TEAM_WSLOTS;
  const int m4 = ko[4 * S + 1] - ko[4 * S], m3 = ko[3 * S + 1] - ko[3 * S], m2 = ko[2 * S + 1] - ko[2 * S],
            m1 = ko[S + 1] - ko[S], m0 = ko[1] - ko[0];
  if (m4 > 0)
    wg = team_decide_tier<32, 8, REFINE, WT, ST>(g, a, ct, a.vlist + ko[4 * S], m4, wg, W, sw, wk, wv, sm, st);
  if (m3 > 0)
    wg = team_decide_tier<32, 4, REFINE, WT, ST>(g, a, ct, a.vlist + ko[3 * S], m3, wg, W, sw, wk, wv, sm, st);
  if (m2 > 0)
    wg = team_decide_tier<32, 1, REFINE, WT, ST>(g, a, ct, a.vlist + ko[2 * S], m2, wg, W, sw, wk, wv, sm, st);
  if (m1 > 0)
    wg = team_decide_tier<16, 1, REFINE, WT, ST>(g, a, ct, a.vlist + ko[S], m1, wg, W, sw, wk, wv, sm, st);
  if (m0 > 0) {
    const int32_t *list = a.vlist + ko[0];
    int32_t *qu = sm.queue[warp];
    int qn = 0;
    for (int base = wg * 32; base < m0; base += W * 32) {
      const int li = base + lane;
      const bool valid = li < m0;
      const int32_t i = valid ? list[li] : 0;
      const bool act = valid && team_eligible<REFINE>(a, ct, i);
      const unsigned mk = __ballot_sync(FULL_MASK, act);
      if (mk == FULL_MASK) {   // the common case of a first iteration
        team_decide_lane<REFINE, WT, ST>(g, a, ct, i, true, sw, sm, st);
        continue;
      }
      // few are eligible: gathered until they fill a warp
      if (act) qu[qn + __popc(mk & ((1u << lane) - 1u))] = i;
      qn += __popc(mk);
      __syncwarp();
      if (qn >= 32) {
        qn -= 32;
        const int32_t x = qu[qn + lane];
        __syncwarp();
        team_decide_lane<REFINE, WT, ST>(g, a, ct, x, true, sw, sm, st);
      }
    }
    if (qn > 0) {
      const int32_t x = lane < qn ? qu[lane] : 0;
      team_decide_lane<REFINE, WT, ST>(g, a, ct, x, lane < qn, sw, sm, st);
    }
    __syncwarp();
  }
  if (hubs) {
    if (!t.sync()) return false;
    team_hub_scan<REFINE, WT, ST>(g, a, ct, t, a.vlist + ko[7 * S], a.hub_s + hub0, a.hub_done + hub0, m7, sw, sm, st);
  }
  return true;
}

// Vertex pruning: `nl` lanes re-mark entries l, l + nl, ... of a row, U of
// them in flight.  Most neighbours of a mover are unprocessed already:
// reading the flag first spares the random byte store.
template <int U, typename GL>
__device__ __forceinline__ void team_remark(const GL &g, uint8_t *processed, int64_t e0, int len, int l,
                                            int nl) {
  for (int x = l; x < len; x += nl * U) {
    int32_t j[U];
    uint8_t f[U];
#pragma unroll
    for (int u = 0; u < U; u++) j[u] = x + nl * u < len ? g.idx[e0 + x + nl * u] : -1;
#pragma unroll
    for (int u = 0; u < U; u++) f[u] = j[u] >= 0 ? processed[j[u]] : 0;
#pragma unroll
    for (int u = 0; u < U; u++)
      if (f[u]) processed[j[u]] = 0;
  }
}

// Commits of a local-moving sub-sweep: the block's own proposals, then the
// team's overflow list (nover entries).
template <typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_apply_moves(const GL &g, const AR &a, const CT &ct,
                                                 const Team &t, unsigned np, unsigned nover, unsigned npiece,
                                                 TeamShared<ST> &sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < np) {
    const TeamProp p = sm.prop[threadIdx.x];
    atomic_add_i64(&a.Sig[p.d], -p.K);
    atomic_add_i64(&a.Sig[p.c], p.K);
    a.C[p.i] = p.c;
    if (ct.dynamic) { a.ch[p.d] = 1; a.ch[p.c] = 1; }
  }
  // rows of up to 64 entries: eight lanes each; up to REMARK_PIECE: a warp;
  // longer ones: in pieces over the team's warps
  constexpr int SHORT = 64;
  for (unsigned m = threadIdx.x >> 3; m < np; m += TEAM_THREADS / 8)
    if (sm.prop[m].len <= SHORT) team_remark<4>(g, a.processed, sm.prop[m].e0, sm.prop[m].len, lane & 7, 8);
  for (unsigned m = warp; m < np; m += TEAM_WARPS)
    if (sm.prop[m].len > SHORT && sm.prop[m].len <= REMARK_PIECE)
      team_remark<8>(g, a.processed, sm.prop[m].e0, sm.prop[m].len, lane, 32);
  const unsigned gt = t.index(), nt = t.nb * TEAM_THREADS;
  for (unsigned m = gt >> 5; m < npiece; m += nt >> 5) {
    const int32_t i = a.piece_i[m];
    const int64_t e0 = g.off[i] + (int64_t)a.piece_k[m] * REMARK_PIECE, left = g.off[i + 1] - e0;
    team_remark<8>(g, a.processed, e0, left < REMARK_PIECE ? (int)left : REMARK_PIECE, lane, 32);
  }
  if (!nover) return;
  for (unsigned m = gt; m < nover; m += nt) {
    const int32_t i = a.prop_i[m], c = a.prop_c[m], d = a.C[i];
    const int64_t Ki = a.K[i];
    atomic_add_i64(&a.Sig[d], -Ki);
    atomic_add_i64(&a.Sig[c], Ki);
    a.C[i] = c;
    if (ct.dynamic) { a.ch[d] = 1; a.ch[c] = 1; }
  }
  for (unsigned m = gt >> 3; m < nover; m += nt >> 3) {
    const int32_t i = a.prop_i[m];
    const int64_t e0 = g.off[i];
    const int len = (int)(g.off[i + 1] - e0);
    if (len <= SHORT) team_remark<4>(g, a.processed, e0, len, lane & 7, 8);
  }
  for (unsigned m = gt >> 5; m < nover; m += nt >> 5) {
    const int32_t i = a.prop_i[m];
    const int64_t e0 = g.off[i];
    const int len = (int)(g.off[i + 1] - e0);
    if (len > SHORT && len <= REMARK_PIECE) team_remark<8>(g, a.processed, e0, len, lane, 32);
  }
}

template <typename ST>
__device__ __forceinline__ int64_t team_block_sum(int64_t v, TeamShared<ST> &sm) {
  for (int o = 16; o; o >>= 1) v += shfl_xor_i64(v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sm.red64[warp] = v;
  __syncthreads();
  int64_t r = lane < TEAM_WARPS ? sm.red64[lane] : 0;
  for (int o = 16; o; o >>= 1) r += shfl_xor_i64(r, o);
  return r;
}

// Exclusive scan over [0, n): in(k) gives element k, out(k, prefix) receives
// its exclusive prefix; returns the total.  Each block owns one contiguous
// segment; the block sums meet in ctl->part.
template <typename ST, typename FI, typename FO>
__device__ __forceinline__ int64_t team_scan(int64_t n, Team &t, TeamShared<ST> &sm, FI in, FO out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t seg = ((n + t.nb - 1) / t.nb + 3) & ~(int64_t)3;
  const int64_t b0 = seg * t.rank < n ? seg * t.rank : n, b1 = b0 + seg < n ? b0 + seg : n;
  int64_t s = 0;
  for (int64_t k = b0 + threadIdx.x; k < b1; k += TEAM_THREADS) s += in(k);
  s = team_block_sum(s, sm);
  if (threadIdx.x == 0) t.ctl->part[t.rank] = s;
  if (!t.sync()) return 0;
  int64_t before = 0, total = 0;
  for (int b = threadIdx.x; b < t.nb; b += TEAM_THREADS) {
    const int64_t x = t.ctl->part[b];
    total += x;
    if (b < t.rank) before += x;
  }
  before = team_block_sum(before, sm);
  total = team_block_sum(total, sm);
  int64_t carry = before;
  for (int64_t base = b0; base < b1; base += 4 * TEAM_THREADS) {
    int64_t v[4], x = 0;
    const int64_t k0 = base + 4 * threadIdx.x;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      v[u] = k0 + u < b1 ? in(k0 + u) : 0;
      x += v[u];
    }
    int64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = shfl_i64(incl, (lane - o) & 31);
      if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) sm.red64[warp] = incl;
    __syncthreads();
    int64_t ws = lane < TEAM_WARPS ? sm.red64[lane] : 0, wi = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = shfl_i64(wi, (lane - o) & 31);
      if (lane >= o) wi += y;
    }
    const int64_t wpre = shfl_i64(wi - ws, warp);
    const int64_t tile = shfl_i64(wi, 31);
    int64_t run = carry + wpre + incl - x;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (k0 + u < b1) out(k0 + u, run);
      run += v[u];
    }
    carry += tile;
  }
  return total;
}

// Vertex lists by (tier, colour class) in a.vlist, offsets in sm.koff (key =
// tier * S + class); vertices without entries are left out.  hist: shared
// words for the block's counts (the table area, free here).
template <typename WT, typename ST, typename GL, typename AR>
__device__ __forceinline__ bool team_lists(const GL &g, const AR &a, int log2S, Team &t,
                                           int32_t *hist, TeamShared<ST> &sm) {
  const int nk = (1 << log2S) * TEAM_TIERS;
  for (int k = threadIdx.x; k < nk; k += TEAM_THREADS) hist[k] = 0;
  __syncthreads();
  const int64_t seg = (g.n + t.nb - 1) / t.nb;
  const int64_t b0 = seg * t.rank < g.n ? seg * t.rank : g.n, b1 = b0 + seg < g.n ? b0 + seg : g.n;
  for (int64_t v = b0 + threadIdx.x; v < b1; v += TEAM_THREADS) {
    const int64_t deg = g.off[v + 1] - g.off[v];
    if (deg > 0) atomicAdd(&hist[(team_tier(deg, g.n) << log2S) + det_class((int32_t)v, log2S)], 1);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nk; k += TEAM_THREADS)
    if (hist[k]) atomicAdd(&t.ctl->ktot[k], (unsigned)hist[k]);
  TEAM_SYNC_OR(false);
  // offsets: every block scans the totals for itself
  {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t carry = 0;
    for (int base = 0; base < nk; base += TEAM_THREADS) {
      const int k = base + threadIdx.x;
      const int32_t v = k < nk ? (int32_t)__ldcg(&t.ctl->ktot[k]) : 0;
      int32_t x = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(FULL_MASK, x, o);
        if (lane >= o) x += y;
      }
      __syncthreads();
      if (lane == 31) sm.red64[warp] = x;
      __syncthreads();
      int32_t pre = carry, tile = 0;
      for (int q = 0; q < TEAM_WARPS; q++) {
        const int32_t y = (int32_t)sm.red64[q];
        if (q < warp) pre += y;
        tile += y;
      }
      if (k < nk) sm.koff[k] = pre + x - v;
      carry += tile;
    }
    if (threadIdx.x == 0) sm.koff[nk] = carry;
    __syncthreads();
    for (int k = threadIdx.x; k < nk; k += TEAM_THREADS) {
      const int h = hist[k];
      if (h) hist[k] = sm.koff[k] + (int)atomicAdd(&t.ctl->kcur[k], (unsigned)h);
    }
    __syncthreads();
  }
  for (int64_t v = b0 + threadIdx.x; v < b1; v += TEAM_THREADS) {
    const int64_t deg = g.off[v + 1] - g.off[v];
    if (deg > 0)
      a.vlist[atomicAdd(&hist[(team_tier(deg, g.n) << log2S) + det_class((int32_t)v, log2S)], 1)] = (int32_t)v;
  }
  return t.sync();
}

// Alg. leidenlm; returns l_i (0 after an expired wait).
template <typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ int team_local_move(const GL &g, const AR &a, const CT &ct,
                                               double tau, int max_iters, Team &t, int32_t *keys,
                                               typename TableVal<ST>::type *vals, TeamShared<ST> &sm, TeamStat &st) {
  const int S = 1 << ct.log2S;
  TeamCtl *ctl = t.ctl;
  int li = 0;
  TeamSweep sw{0, 0, true, nullptr, nullptr};
  int64_t moves = 0;
  while (li < max_iters) {
    st.S = 0;
    u64 *sums = ctl->sums[li & 1];
    for (int s = 0; s < S; s++, sw.par ^= 1) {
      u64 t0 = 0;
      if (ct.timing && t.rank == 0 && threadIdx.x == 0) asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
      sw.nover = &ctl->nover[sw.par];
      sw.npiece = &ctl->npiece[sw.par];
      // headers alongside the eligibility test while most listed vertices are
      // eligible or the class is too short to fill the team anyway
      sw.spec = (li == 0 && !ct.dynamic) || sm.koff[TEAM_TIERS * S] <= t.nb * TEAM_THREADS;
      if (!team_decide_class<false, WT, ST>(g, a, ct, t, s, sw, keys, vals, sm, st)) return 0;
      if (s == S - 1) {
        // the iteration's sum of scores, one addition per block
        i128 acc = st.S;
        for (int o = 16; o; o >>= 1) acc += shfl_xor_i128(acc, o);
        if ((threadIdx.x & 31) == 0) sm.red128[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x < 32) {
          acc = threadIdx.x < TEAM_WARPS ? sm.red128[threadIdx.x] : 0;
          for (int o = 16; o; o >>= 1) acc += shfl_xor_i128(acc, o);
          if (threadIdx.x == 0 && acc != 0) atomic_add_i128(sums, acc);
        }
      }
      TEAM_SYNC_OR(0);
      if (t0) {
        u64 t1;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
        ctl->decide_ns += t1 - t0;
        ctl->subsweeps++;
      }
      const unsigned nover = __ldcg(sw.nover), npiece = __ldcg(sw.npiece);
      unsigned np = sm.nprop[sw.par];
      np = np < TEAM_PROPS ? np : TEAM_PROPS;
      if (threadIdx.x == 0) {
        // the other parity's counters were read before the previous barrier
        sm.nprop[sw.par ^ 1] = 0;
        moves += np;
        if (t.rank == 0) {
          ctl->nover[sw.par ^ 1] = 0;
          ctl->npiece[sw.par ^ 1] = 0;
          moves += nover;
          if (s == 0) { ctl->sums[(li & 1) ^ 1][0] = 0; ctl->sums[(li & 1) ^ 1][1] = 0; }
        }
      }
      if (np | nover | npiece) team_apply_moves<WT, ST>(g, a, ct, t, np, nover, npiece, sm);
      TEAM_SYNC_OR(0);
    }
    li++;
    if (threadIdx.x == 0) {
      const u64 lo = __ldcg(&sums[0]), hi = __ldcg(&sums[1]);
      const i128 tot = (i128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
      sm.flag = (ct.two_m == 0 || team_i128_to_double(tot) / ct.den <= tau) ? 1 : 0;
    }
    __syncthreads();
    const int stop = sm.flag;
    __syncthreads();
    if (stop) break;
  }
  if (threadIdx.x == 0) {
    sm.nprop[0] = sm.nprop[1] = 0;
    if (moves) atomicAdd((u64 *)&ctl->moves, (u64)moves);
    if (t.rank == 0) { ctl->li = li; ctl->nover[0] = ctl->nover[1] = 0; }
  }
  return li;
}

// Alg. leidenre: one sweep, one sub-sweep per colour class.  stamp is zero.
template <typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ bool team_refine(const GL &g, const AR &a, const CT &ct, Team &t,
                                            int32_t *keys, typename TableVal<ST>::type *vals, TeamShared<ST> &sm) {
  const int S = 1 << ct.log2S;
  TeamCtl *ctl = t.ctl;
  const int gt = t.index(), nt = t.nb * TEAM_THREADS;
  TeamStat st{};
  TeamSweep sw{0, 0, true, nullptr, nullptr};
  int64_t moved = 0;
  for (int s = 0; s < S; s++, sw.par ^= 1) {
    // stamps 1..255 name the sub-sweep a vertex proposed in; a stamp only
    // matters inside its own sub-sweep, so the array is cleared on wrap
    sw.sv = (uint8_t)(s % 255 + 1);
    if (s > 0 && sw.sv == 1) {
      for (int64_t i = gt; i < g.n; i += nt) a.stamp[i] = 0;
      TEAM_SYNC_OR(false);
    }
    sw.nover = &ctl->nover[sw.par];
    sw.spec = !ct.dynamic;   // every vertex starts isolated in a changed bound, but for an update's first pass
    if (!team_decide_class<true, WT, ST>(g, a, ct, t, s, sw, keys, vals, sm, st)) return false;
    TEAM_SYNC_OR(false);
    const unsigned nover = __ldcg(sw.nover);
    unsigned np = sm.nprop[sw.par];
    np = np < TEAM_PROPS ? np : TEAM_PROPS;
    if (threadIdx.x == 0) {
      sm.nprop[sw.par ^ 1] = 0;
      if (t.rank == 0) ctl->nover[sw.par ^ 1] = 0;
    }
    auto commit = [&](int32_t i, int32_t c, int64_t Ki) {
      if (a.stamp[c] == sw.sv) return;   // the target proposed to leave in this sub-sweep
      atomic_add_i64(&a.Sig[i], -Ki);    // C'[i] = i: Sigma'[i] drops to 0
      atomic_add_i64(&a.Sig[c], Ki);
      a.C[i] = c;
      moved++;
    };
    if (threadIdx.x < np) commit(sm.prop[threadIdx.x].i, sm.prop[threadIdx.x].c, sm.prop[threadIdx.x].K);
    for (unsigned m = gt; m < nover; m += nt) {
      const int32_t i = a.prop_i[m];
      commit(i, a.prop_c[m], a.K[i]);
    }
    TEAM_SYNC_OR(false);
  }
  for (int o = 16; o; o >>= 1) moved += shfl_xor_i64(moved, o);
  if ((threadIdx.x & 31) == 0 && moved) atomicAdd(&ctl->rmoves, (u64)moved);
  return true;
}

// Insert of one ((c, d), w) into the aggregation's global table of H slots:
// key c * 2^32 + d, plus one.  The first insert of a pair counts it
// as an entry of c's row.
template <typename AR>
__device__ __forceinline__ void team_agg_add(const AR &a, u64 H, int32_t c, int32_t d, u64 w) {
  const u64 key = (((u64)(uint32_t)c << 32) | (uint32_t)d) + 1ull;
  u64 s = __umul64hi(key * 0x9E3779B97F4A7C15ull, H);
  for (u64 probe = 0; probe < H; probe++) {
    u64 k = *(volatile u64 *)&a.hkey[s];
    if (k == 0) {
      k = atomicCAS(&a.hkey[s], 0ull, key);
      if (k == 0) atomicAdd((u64 *)&a.cnt[c], 1ull);
    }
    if (k == 0 || k == key) { atomicAdd(&a.hval[s], w); return; }
    s = s + 1 == H ? 0 : s + 1;
  }
  atomicOr(a.err, 16ull);
}

// Alg. leidenag over the whole team: every CSR entry (i, j, w) adds w to the
// pair (C'[i], C'[j]) of one global table, so a giant community spreads over
// the team as evenly as small ones; the pairs then go to their rows.
// Writes off2, idx2, w2, K'' = row sums, and the level state of the next
// pass.  cnt and K2 are zero on entry; the table is empty on entry and exit.
template <typename WT, typename ST, typename GL, typename AR>
__device__ __forceinline__ bool team_aggregate(const GL &g, const AR &a, int64_t nc, u64 H, int S, Team &t,
                                               u64 (*wscr)[32], TeamShared<ST> &sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t gt = t.index(), nt = (int64_t)t.nb * TEAM_THREADS;
  const int32_t *ko = sm.koff;
  // rows of more than TT_WARP8 entries: the block each
  for (int r = ko[5 * S] + t.rank; r < ko[8 * S]; r += t.nb) {
    const int32_t v = a.vlist[r];
    const int64_t e0 = g.off[v], e1 = g.off[v + 1];
    const int32_t c = a.C[v];
    u64 rs = 0;
    for (int64_t x = e0 + 32 * warp; x < e1; x += TEAM_THREADS) {
      const int64_t e = x + lane;
      const bool in = e < e1;
      const int32_t d = in ? a.C[g.idx[e]] : 0;
      const u64 w = in ? (u64)(int64_t)g.w[e] : 0;
      rs += w;
      u64 sum = 0;
      if (warp_combine((unsigned long long)(uint32_t)d, in, w, &sum, wscr[warp])) team_agg_add(a, H, c, d, sum);
    }
    for (int o = 16; o; o >>= 1) rs += (u64)shfl_xor_i64((int64_t)rs, o);
    if (lane == 0 && rs) atomicAdd((u64 *)&a.K2[c], rs);
  }
  // rows of 17 .. TT_WARP8 entries: a warp each
  const int wg = warp * t.nb + t.rank, W = t.nb * TEAM_WARPS;
  for (int r = ko[2 * S] + wg; r < ko[5 * S]; r += W) {
    const int32_t v = a.vlist[r];
    const int64_t e0 = g.off[v];
    const int deg = (int)(g.off[v + 1] - e0);
    const int32_t c = a.C[v];
    u64 rs = 0;
    for (int x = 0; x < deg; x += 32) {
      const bool in = x + lane < deg;
      const int32_t d = in ? a.C[g.idx[e0 + x + lane]] : 0;
      const u64 w = in ? (u64)(int64_t)g.w[e0 + x + lane] : 0;
      rs += w;
      u64 sum = 0;
      if (warp_combine((unsigned long long)(uint32_t)d, in, w, &sum, wscr[warp])) team_agg_add(a, H, c, d, sum);
    }
    for (int o = 16; o; o >>= 1) rs += (u64)shfl_xor_i64((int64_t)rs, o);
    if (lane == 0 && rs) atomicAdd((u64 *)&a.K2[c], rs);
  }
  // shorter rows: eight lanes each
  const int gl = lane & 7;
  for (int rb = ko[0] + 4 * wg; rb < ko[2 * S]; rb += 4 * W) {   // uniform per warp
    const int r = rb + (lane >> 3);
    int64_t e0 = 0;
    int deg = 0;
    int32_t c = 0;
    if (r < ko[2 * S]) {
      const int32_t v = a.vlist[r];
      e0 = g.off[v];
      deg = (int)(g.off[v + 1] - e0);
      c = a.C[v];
    }
    const int span = __reduce_max_sync(FULL_MASK, deg);
    u64 rs = 0;
    for (int x = 0; x < span; x += 8) {
      const bool in = x + gl < deg;
      const int32_t d = in ? a.C[g.idx[e0 + x + gl]] : 0;
      const u64 w = in ? (u64)(int64_t)g.w[e0 + x + gl] : 0;
      rs += w;
      u64 sum = 0;
      const unsigned long long key = ((unsigned long long)(uint32_t)c << 32) | (uint32_t)d;
      if (warp_combine(key, in, w, &sum, wscr[warp])) team_agg_add(a, H, c, d, sum);
    }
#pragma unroll
    for (int o = 4; o; o >>= 1) rs += (u64)shfl_xor_i64((int64_t)rs, o);
    if (gl == 0 && rs) atomicAdd((u64 *)&a.K2[c], rs);
  }
  TEAM_SYNC_OR(false);
  u64 mdeg = 0, mk = 0;
  const int64_t nnz2 = team_scan<ST>(
      nc, t, sm, [&](int64_t c) { return __ldcg(&a.cnt[c]); },
      [&](int64_t c, int64_t pre) {
        a.off2[c] = pre;
        a.cur[c] = pre;
        const u64 x = (u64)__ldcg(&a.cnt[c]), k = (u64)__ldcg(&a.K2[c]);
        if (x > mdeg) mdeg = x;
        if (k > mk) mk = k;
      });
  if (t.dead) return false;
  if (t.rank == 0 && threadIdx.x == 0) a.off2[nc] = nnz2;
  for (int o = 16; o; o >>= 1) {
    const u64 y = __shfl_xor_sync(FULL_MASK, mdeg, o), z = __shfl_xor_sync(FULL_MASK, mk, o);
    if (y > mdeg) mdeg = y;
    if (z > mk) mk = z;
  }
  if (lane == 0) {
    if (mdeg) atomicMax(&t.ctl->maxdeg, mdeg);
    if (mk) atomicMax(&t.ctl->kmax, mk);
  }
  TEAM_SYNC_OR(false);
  // the pairs to their rows, the table empty again
  for (int64_t s = gt; s < (int64_t)H; s += nt) {
    const u64 k = __ldcg(&a.hkey[s]);
    if (!k) continue;
    const u64 v = __ldcg(&a.hval[s]);
    a.hkey[s] = 0;
    a.hval[s] = 0;
    const int64_t pos = (int64_t)atomicAdd((u64 *)&a.cur[(k - 1) >> 32], 1ull);
    a.idx2[pos] = (int32_t)(uint32_t)(k - 1);
    a.w2[pos] = (int64_t)v;
  }
  if (t.rank == 0 && threadIdx.x == 0) t.ctl->nnz2 = nnz2;
  return true;
}

// One whole pass.  See TeamArgs for what it reads and leaves behind.  SHARED:
// the array table is one copy in the block's shared memory (else each thread
// has its own).
template <bool SHARED, typename WT, typename ST, typename GL, typename AR, typename CT>
__device__ __forceinline__ void team_pass(const GL &g, AR &a, const CT &ct, int lp, double tau,
                                          int max_iters, int64_t agg_slots, Team &t, unsigned char *dyn,
                                          TeamShared<ST> &sm) {
  typedef typename TableVal<ST>::type VT;
  VT *vals = reinterpret_cast<VT *>(dyn);
  int32_t *keys = reinterpret_cast<int32_t *>(vals + TEAM_WARPS * TEAM_WSLOTS);
  TeamCtl *ctl = t.ctl;
  const int gt = t.index(), nt = t.nb * TEAM_THREADS;
  const int64_t n = g.n;
  TeamStat st{};
  auto stamp_time = [&](int k) {
    if (t.rank == 0 && threadIdx.x == 0) {
      u64 x;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(x));
      ctl->stamp[k] = x;
    }
  };
  stamp_time(0);
  if (!team_lists<WT, ST>(g, a, ct.log2S, t, reinterpret_cast<int32_t *>(dyn), sm)) return;
  // the shared-memory tables: empty whenever no vertex uses them
  for (int k = threadIdx.x; k < TEAM_WARPS * TEAM_WSLOTS; k += TEAM_THREADS) { keys[k] = LEIDEN_EMPTY_KEY; vals[k] = 0; }
  if (threadIdx.x < 2) sm.nprop[threadIdx.x] = 0;
  __syncthreads();
  if (!team_hub_setup<WT, ST>(g, a, 1 << ct.log2S, t, sm)) {
    if (!t.dead && t.rank == 0 && threadIdx.x == 0) ctl->status = TEAM_TOO_BIG;
    return;
  }
  const int li = team_local_move<WT, ST>(g, a, ct, tau, max_iters, t, keys, vals, sm, st);
  if (t.dead) return;
  for (int o = 16; o; o >>= 1) {
    st.scanned += shfl_xor_i64(st.scanned, o);
    st.nvert += shfl_xor_i64(st.nvert, o);
    st.ncand += shfl_xor_i64(st.ncand, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (st.scanned) atomicAdd(&ctl->scanned_e, (u64)st.scanned);
    if (st.nvert) atomicAdd(&ctl->scanned_v, (u64)st.nvert);
    if (st.ncand) atomicAdd(&ctl->cand, (u64)st.ncand);
  }
  stamp_time(1);
  // Alg. leidensr (representative = smallest member), the bounds, the break
  int64_t changed = 0;
  for (int64_t c = gt; c < n; c += nt) {
    a.rep[c] = INT_MAX;
    a.Sig2[c] = 0;
    a.ch2[c] = 0;
    a.stamp[c] = 0;
    a.exists[c] = 0;
    changed += a.ch[c] != 0;
  }
  for (int o = 16; o; o >>= 1) changed += shfl_xor_i64(changed, o);
  if ((threadIdx.x & 31) == 0 && changed) atomicAdd(&ctl->changed, (u64)changed);
  TEAM_SYNC_OR();
  for (int64_t i = gt; i < n; i += nt) {
    const int32_t c = a.C[i];
    if (__ldcg(&a.rep[c]) > (int32_t)i) atomicMin(&a.rep[c], (int32_t)i);
  }
  TEAM_SYNC_OR();
  for (int64_t c = gt; c < n; c += nt) {
    const int32_t r = __ldcg(&a.rep[c]);
    if (r == INT_MAX) continue;
    a.Sig2[r] = a.Sig[c];
    a.ch2[r] = a.ch[c];
  }
  TEAM_SYNC_OR();
  if (!SHARED || threadIdx.x == 0) {
    { int64_t *x = a.Sig; a.Sig = a.Sig2; a.Sig2 = x; }
    { uint8_t *x = a.ch; a.ch = a.ch2; a.ch2 = x; }
  }
  if (SHARED) __syncthreads();
  for (int64_t i = gt; i < n; i += nt) {
    const int32_t c = a.rep[a.C[i]];
    a.CB[i] = c;
    if (a.ch[c]) {
      a.C[i] = (int32_t)i;
      a.Sig[i] = a.K[i];   // only vertex i reads or writes its own total here
    } else {
      a.C[i] = c;
    }
  }
  TEAM_SYNC_OR();
  if (!team_refine<WT, ST>(g, a, ct, t, keys, vals, sm)) return;
  stamp_time(2);
  if (lp > 0 && li <= 1) {   // globally converged
    if (t.rank == 0 && threadIdx.x == 0) ctl->status = TEAM_CONVERGED;
    return;
  }
  // dense renumbering in increasing order of the old ID
  for (int64_t i = gt; i < n; i += nt) {
    const int32_t c = a.C[i];
    if (!a.exists[c]) a.exists[c] = 1;
  }
  TEAM_SYNC_OR();
  const int64_t nc = team_scan<ST>(
      n, t, sm, [&](int64_t c) { return (int64_t)a.exists[c]; },
      [&](int64_t c, int64_t pre) { a.rep[c] = (int32_t)pre; });
  if (t.dead) return;
  if (t.rank == 0 && threadIdx.x == 0) ctl->nc = nc;
  const bool agg = agg_slots > 0 && nc != n;
  TEAM_SYNC_OR();
  for (int64_t i = gt; i < n; i += nt) {
    const int32_t c = a.rep[a.C[i]];
    a.C[i] = c;
    a.CB[i] = c;   // kept for the dendrogram lookup
    if (agg && i < nc) { a.cnt[i] = 0; a.K2[i] = 0; }
  }
  if (!agg) {
    stamp_time(3);
    if (t.rank == 0 && threadIdx.x == 0) ctl->status = nc == n ? TEAM_NO_SHRINK : TEAM_RENUMBERED;
    return;
  }
  TEAM_SYNC_OR();
  if (!team_aggregate<WT, ST>(g, a, nc, (u64)agg_slots, 1 << ct.log2S, t, reinterpret_cast<u64(*)[32]>(dyn), sm)) return;
  // the next level: K' = Sigma' = row sums, C' = identity, everything
  // unprocessed, every community changed (C, K, Sig were read last before
  // the barriers of the aggregation)
  for (int64_t c = gt; c < nc; c += nt) {
    const int64_t k = __ldcg(&a.K2[c]);
    a.K[c] = k;
    a.Sig[c] = k;
    a.C[c] = (int32_t)c;
    a.processed[c] = 0;
    a.ch[c] = 1;
  }
  stamp_time(3);
  if (t.rank == 0 && threadIdx.x == 0) ctl->status = TEAM_AGGREGATED;
}

}  // namespace LK_TEAM_SPACE
}  // namespace lk
