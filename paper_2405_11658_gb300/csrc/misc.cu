// misc.cu -- the small phases of Alg. leiden and the dynamic front-ends:
// weighted degrees, subset renumbering (Alg. leidensr), breakChangedCommunities,
// dense renumbering, dendrogram lookup, canonical labels, modularity terms
// (Eq. 1), updateWeights (Alg. update), changedCommunities and DF marking
// (Alg. frontier).
#include <limits.h>

#include "common.cuh"
#include "internal.h"

namespace lk {

static inline unsigned grid_for(int64_t n, int threads, int64_t cap = 1 << 20) {
  int64_t b = (n + threads - 1) / threads;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (unsigned)b;
}

#define GRID_STRIDE(i, n) \
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// ---------------------------------------------------------------------------
// One pass over a CSR that checks it and sums its rows (K_i, self-loop
// included once, and 2m) or takes the terms of Eq. 1.
//
// Bound by the stream of idx and w (8 bytes an entry) and, for Eq. 1, by the
// gathers of C[j] from L2.  A warp takes `ch` consecutive items of the merged
// sequence of entries and row ends (entry e of row i is item e + i), found by
// a 32-way search of the row offsets, so heavy rows, runs of empty rows and
// ordinary ones all split evenly: with the rows dealt out instead, the block
// with R-MAT scale 22's first rows took 4.8 ms, the whole pass takes 1.0
// ms here (3.4 ms with a warp and an atomic per row).  G lanes share a short
// row (2 where rows have up to 8 entries on average, else 8), four entries per
// lane in flight; longer pieces take the whole warp.  32 rows' totals meet
// per community before they reach Sigma: neighbouring vertices often share
// one, and an atomic per vertex queued on a few addresses.
//
// The offsets and labels are checked by check_graph_rows_k; this kernel tests
// every index before it uses it all the same -- the row bounds against
// [0, nnz], the labels and column IDs against [0, n) -- so a malformed input
// can never make it read or write outside the arrays: an offending row or
// entry is skipped and sets 512 in *err, as does a weight that is not
// positive.  K and Sigma are zero on entry.
// ---------------------------------------------------------------------------
static constexpr int ROWS_THREADS = 256, ROWS_WARPS = ROWS_THREADS / 32;
template <int G, bool MOD>
__global__ void __launch_bounds__(ROWS_THREADS) rows_k(GraphView<int32_t> g, int64_t nnz, const int32_t *C, int64_t *K,
                                                       int64_t *Sig, u64 *acc, u64 *err, int64_t ch) {
  __shared__ int64_t sbuf[32];
  __shared__ u64 wscr[ROWS_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t inside = 0, total = 0;
  bool bad = false;
  // entries first, first + step, ... < e1 of a row of community ci
  auto part = [&](int64_t first, int64_t e1, int64_t step, int32_t ci) -> int64_t {
    int64_t k = 0;
    for (int64_t e = first; e < e1; e += 4 * step) {
      int32_t j[4], w[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const bool in = e + u * step < e1;
        j[u] = in ? g.idx[e + u * step] : 0;
        w[u] = in ? g.w[e + u * step] : 0;
        if (in && (j[u] < 0 || (int64_t)j[u] >= g.n || w[u] <= 0)) { bad = true; w[u] = 0; j[u] = 0; }
      }
      if (MOD) {
        int32_t cj[4];
#pragma unroll
        for (int u = 0; u < 4; u++) cj[u] = w[u] ? C[j[u]] : -1;
#pragma unroll
        for (int u = 0; u < 4; u++)
          if (cj[u] == ci) inside += w[u];
      }
#pragma unroll
      for (int u = 0; u < 4; u++) k += w[u];
    }
    return k;
  };
  const int64_t items = g.n + nnz;
  for (int64_t d0 = ((int64_t)warp * gridDim.x + blockIdx.x) * ch; d0 < items;
       d0 += (int64_t)ROWS_WARPS * gridDim.x * ch) {   // uniform per warp
    const int64_t d1 = d0 + ch < items ? d0 + ch : items;
    // last row r with off[r] + r <= d0
    int64_t r0 = 0, len = g.n;
    while (len > 1) {
      const int64_t step = (len + 31) / 32, r = r0 + lane * step;
      const unsigned m = __ballot_sync(FULL_MASK, lane * step < len && g.off[r] + r <= d0);
      const int k = m ? 31 - __clz(m) : 0;
      len = len - k * step < step ? len - k * step : step;
      r0 += k * step;
    }
    int64_t windows = ch / 32 + 2;   // rows of the piece at most, 32 at a time
    for (int64_t rb = r0; rb < g.n && windows > 0; rb += 32, windows--) {
      const int64_t i = rb + lane;
      int64_t e0 = 0, e1 = 0;
      int32_t ci = -1;
      bool mine = false, whole = false;
      if (i < g.n) {
        const int64_t a = g.off[i], b = g.off[i + 1];
        mine = a + i < d1;
        if (mine) {
          if (MOD) ci = C[i];
          if (a < 0 || b < a || b > nnz || (MOD && (ci < 0 || (int64_t)ci >= g.n))) {
            bad = true;
            ci = -1;
          } else {
            e0 = a + i >= d0 ? a : d0 - i;
            e1 = b + i <= d1 ? b : d1 - i;
            if (e1 < e0) e1 = e0;
            whole = e0 == a && e1 == b;
          }
        }
      }
      if (!__any_sync(FULL_MASK, mine)) break;
      const int64_t n_i = e1 - e0;
      int64_t Ki = 0;
      // short pieces, 32 / G at a time
#pragma unroll 1
      for (int it = 0; it < G; it++) {
        const int src = it * (32 / G) + lane / G;
        const int64_t a = shfl_i64(e0, src), b = shfl_i64(e1, src);
        const int32_t c = __shfl_sync(FULL_MASK, ci, src);
        int64_t k = b - a <= 16 * G ? part(a + lane % G, b, G, c) : 0;
#pragma unroll
        for (int o = G / 2; o; o >>= 1) k += shfl_xor_i64(k, o);
        // row it * (32 / G) + q was summed by the lanes from q * G on
        const int64_t v = shfl_i64(k, (lane % (32 / G)) * G);
        if (lane / (32 / G) == it) Ki = v;
      }
      for (unsigned m = __ballot_sync(FULL_MASK, n_i > 16 * G); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        int64_t k = part(shfl_i64(e0, src) + lane, shfl_i64(e1, src), 32, __shfl_sync(FULL_MASK, ci, src));
        for (int o = 16; o; o >>= 1) k += shfl_xor_i64(k, o);
        if (lane == src) Ki = k;
      }
      total += Ki;
      if (MOD) {
        u64 sum = 0;
        if (warp_combine((unsigned long long)(uint32_t)ci, ci >= 0 && Ki != 0, (u64)Ki, &sum, wscr[warp]))
          atomicAdd((u64 *)&Sig[ci], sum);
      } else if (Ki != 0) {
        if (whole) K[i] = Ki;
        else atomic_add_i64(&K[i], Ki);   // a row shared with the neighbouring pieces
      }
    }
  }
  if (bad) atomicOr(err, 512ull);
  if (MOD) {
    inside = block_sum_i64(inside, sbuf);
    if (threadIdx.x == 0 && inside) atomicAdd(&acc[0], (u64)inside);
  }
  total = block_sum_i64(total, sbuf);
  if (threadIdx.x == 0 && total) atomicAdd(&acc[3], (u64)total);
}

// Row offsets: off[0] = 0, off[n] = nnz, non-decreasing; labels (if any) in
// [0, n).  Sets *err on violation.
__global__ void check_graph_rows_k(int64_t n, int64_t nnz, const int64_t *off, const int32_t *C, u64 *err) {
  bool bad = blockIdx.x == 0 && threadIdx.x == 0 && (off[0] != 0 || off[n] != nnz);
  GRID_STRIDE(i, n) {
    const int64_t a = off[i], b = off[i + 1];
    if (a > b || a < 0 || b > nnz) bad = true;
    if (C && (C[i] < 0 || (int64_t)C[i] >= n)) bad = true;
  }
  if (bad) atomicOr(err, 128ull);
}

template <bool MOD>
static void launch_rows(GraphView<int32_t> g, int64_t nnz, const int32_t *C, int64_t *K, int64_t *Sig, u64 *acc,
                        u64 *err, int sms, cudaStream_t s) {
  LK_COUNTED check_graph_rows_k<<<grid_for(g.n > 0 ? g.n : 1, 256, sms * 32), 256, 0, s>>>(g.n, nnz, g.off, C, err);
  if (g.n <= 0) return;
  auto k2 = rows_k<2, MOD>;
  auto k8 = rows_k<8, MOD>;
  const bool two = nnz <= 8 * g.n;
  const int64_t cap = resident_blocks(two ? (const void *)k2 : (const void *)k8, ROWS_THREADS, 0, sms);
  // pieces of 256 .. 2048 items, small ones where the graph is too short to
  // give every resident warp one of the longer
  int64_t ch = (g.n + nnz) / (cap * ROWS_WARPS);
  ch = ch < 256 ? 256 : ch > 2048 ? 2048 : ch;
  int64_t blocks = ((g.n + nnz + ch - 1) / ch + ROWS_WARPS - 1) / ROWS_WARPS;
  if (blocks > cap) blocks = cap;
  if (two) LK_COUNTED k2<<<(unsigned)blocks, ROWS_THREADS, 0, s>>>(g, nnz, C, K, Sig, acc, err, ch);
  else LK_COUNTED k8<<<(unsigned)blocks, ROWS_THREADS, 0, s>>>(g, nnz, C, K, Sig, acc, err, ch);
}

void launch_row_sums(GraphView<int32_t> g, int64_t nnz, int64_t *K, u64 *acc, u64 *err, int sms, cudaStream_t s) {
  cudaMemsetAsync(acc, 0, 4 * sizeof(u64), s);
  if (g.n > 0) cudaMemsetAsync(K, 0, (size_t)g.n * sizeof(int64_t), s);
  launch_rows<false>(g, nnz, nullptr, K, nullptr, acc, err, sms, s);
}

__global__ void iota_k(int32_t *a, int64_t n) { GRID_STRIDE(i, n) a[i] = (int32_t)i; }
void launch_iota(int32_t *a, int64_t n, cudaStream_t s) {
  if (n > 0) LK_COUNTED iota_k<<<grid_for(n, 256), 256, 0, s>>>(a, n);
}
__global__ void fill_u8_k(uint8_t *a, uint8_t v, int64_t n) { GRID_STRIDE(i, n) a[i] = v; }
void launch_fill_u8(uint8_t *a, uint8_t v, int64_t n, cudaStream_t s) {
  if (n > 0) cudaMemsetAsync(a, v, (size_t)n, s);
}
void launch_copy_i64(int64_t *dst, const int64_t *src, int64_t n, cudaStream_t s) {
  if (n > 0) cudaMemcpyAsync(dst, src, (size_t)n * sizeof(int64_t), cudaMemcpyDeviceToDevice, s);
}
__global__ void invert_u8_k(uint8_t *d, const uint8_t *a, int64_t n) { GRID_STRIDE(i, n) d[i] = a[i] ? 0 : 1; }
// After an ASYNC refinement: the totals of communities whose own vertex left
// hold the departure marker; those communities are empty.
__global__ void clear_left_k(int64_t *Sig, int64_t n) { GRID_STRIDE(i, n) if (Sig[i] < 0) Sig[i] = 0; }
void launch_clear_left(int64_t *Sig, int64_t n, cudaStream_t s) {
  if (n > 0) LK_COUNTED clear_left_k<<<grid_for(n, 256), 256, 0, s>>>(Sig, n);
}
void launch_invert_u8(uint8_t *dst, const uint8_t *src, int64_t n, cudaStream_t s) {
  if (n > 0) LK_COUNTED invert_u8_k<<<grid_for(n, 256), 256, 0, s>>>(dst, src, n);
}

// ---------------------------------------------------------------------------
// Alg. leidensr: relabel each community by a member vertex (the smallest).
// ---------------------------------------------------------------------------
__global__ void sr_init_k(int64_t n, int32_t *rep, int64_t *Sig2, uint8_t *ch2) {
  GRID_STRIDE(c, n) { rep[c] = INT_MAX; Sig2[c] = 0; ch2[c] = 0; }
}
// The minima only fall: a member that reads a representative already below
// its own ID cannot lower it, and skips the atomic (a large community's
// members would otherwise queue on one address).
__global__ void sr_min_k(int64_t n, const int32_t *C, int32_t *rep) {
  GRID_STRIDE(i, n) {
    const int32_t c = C[i];
    if (rep[c] > (int32_t)i) atomicMin(&rep[c], (int32_t)i);
  }
}
__global__ void sr_move_k(int64_t n, const int32_t *rep, const int64_t *Sig, int64_t *Sig2,
                          const uint8_t *ch, uint8_t *ch2) {
  GRID_STRIDE(c, n) {
    const int32_t r = rep[c];
    if (r == INT_MAX) continue;
    Sig2[r] = Sig[c];
    ch2[r] = ch[c];
  }
}
__global__ void sr_relabel_k(int64_t n, int32_t *C, const int32_t *rep) {
  GRID_STRIDE(i, n) C[i] = rep[C[i]];
}
void launch_subset_renumber(int64_t n, int32_t *C, const int64_t *Sig, int64_t *Sig2,
                            const uint8_t *ch, uint8_t *ch2, int32_t *rep, cudaStream_t s) {
  if (n <= 0) return;
  const unsigned g = grid_for(n, 256);
  LK_COUNTED sr_init_k<<<g, 256, 0, s>>>(n, rep, Sig2, ch2);
  LK_COUNTED sr_min_k<<<g, 256, 0, s>>>(n, C, rep);
  LK_COUNTED sr_move_k<<<g, 256, 0, s>>>(n, rep, Sig, Sig2, ch, ch2);
  LK_COUNTED sr_relabel_k<<<g, 256, 0, s>>>(n, C, rep);
}

// breakChangedCommunities: every vertex of a changed community becomes its
// own community.  Thread i reads only C'[i] and the flags, writes C'[i] and
// Sigma'[i]; no other thread reads Sigma' here.
__global__ void break_k(int64_t n, int32_t *C, const int64_t *K, int64_t *Sig, const uint8_t *ch) {
  GRID_STRIDE(i, n) {
    if (!ch[C[i]]) continue;
    C[i] = (int32_t)i;
    Sig[i] = K[i];
  }
}
void launch_break(int64_t n, int32_t *C, const int64_t *K, int64_t *Sig, const uint8_t *ch,
                  cudaStream_t s) {
  if (n > 0) LK_COUNTED break_k<<<grid_for(n, 256), 256, 0, s>>>(n, C, K, Sig, ch);
}

// Dense renumbering in increasing order of the old ID (flag + exclusive scan).
__global__ void flag_k(int64_t n, const int32_t *C, uint8_t *ex) {
  GRID_STRIDE(i, n) {
    const int32_t c = C[i];
    if (!ex[c]) ex[c] = 1;   // most members find the flag set already: spare the store
  }
}
__global__ void relabel_scan_k(int64_t n, int32_t *C, const int64_t *scanned) {
  GRID_STRIDE(i, n) C[i] = (int32_t)scanned[C[i]];
}
__global__ void store_total_k(const int64_t *scanned, int64_t n, u64 *dst) { *dst = (u64)scanned[n]; }
void launch_renumber(int64_t n, int32_t *C, uint8_t *exists, int64_t *scanned, int64_t *tmp,
                     u64 *ctr, cudaStream_t s) {
  cudaMemsetAsync(exists, 0, (size_t)(n > 0 ? n : 1), s);
  if (n > 0) LK_COUNTED flag_k<<<grid_for(n, 256), 256, 0, s>>>(n, C, exists);
  exclusive_scan<uint8_t>(exists, scanned, n, tmp, s);
  if (n > 0) LK_COUNTED relabel_scan_k<<<grid_for(n, 256), 256, 0, s>>>(n, C, scanned);
  LK_COUNTED store_total_k<<<1, 1, 0, s>>>(scanned, n, &ctr[CTR_NCOMM]);
}

// Dendrogram lookup C[v] <- C'[C[v]].
__global__ void lookup_k(int64_t n, int32_t *Ctop, const int32_t *Cp) {
  GRID_STRIDE(v, n) Ctop[v] = Cp[Ctop[v]];
}
void launch_lookup(int64_t n, int32_t *Ctop, const int32_t *Cp, cudaStream_t s) {
  if (n > 0) LK_COUNTED lookup_k<<<grid_for(n, 256), 256, 0, s>>>(n, Ctop, Cp);
}

// Canonical labels: communities numbered by their smallest member vertex.
__global__ void canon_init_k(int64_t n, int32_t *minv, uint8_t *flag) {
  GRID_STRIDE(i, n) { minv[i] = INT_MAX; flag[i] = 0; }
}
__global__ void canon_min_k(int64_t n, const int32_t *C, int32_t *minv) {
  GRID_STRIDE(v, n) {
    const int32_t c = C[v];
    if (minv[c] > (int32_t)v) atomicMin(&minv[c], (int32_t)v);   // as in sr_min_k
  }
}
__global__ void canon_flag_k(int64_t n, const int32_t *minv, uint8_t *flag) {
  GRID_STRIDE(c, n) if (minv[c] != INT_MAX) flag[minv[c]] = 1;
}
__global__ void canon_out_k(int64_t n, const int32_t *C, const int32_t *minv, const int64_t *scanned,
                            int32_t *out) {
  GRID_STRIDE(v, n) out[v] = (int32_t)scanned[minv[C[v]]];
}
void launch_canonical(int64_t n, const int32_t *C, int32_t *out, int32_t *minv, uint8_t *flag,
                      int64_t *scanned, int64_t *tmp, cudaStream_t s) {
  if (n <= 0) return;
  const unsigned g = grid_for(n, 256);
  LK_COUNTED canon_init_k<<<g, 256, 0, s>>>(n, minv, flag);
  LK_COUNTED canon_min_k<<<g, 256, 0, s>>>(n, C, minv);
  LK_COUNTED canon_flag_k<<<g, 256, 0, s>>>(n, minv, flag);
  exclusive_scan<uint8_t>(flag, scanned, n, tmp, s);
  LK_COUNTED canon_out_k<<<g, 256, 0, s>>>(n, C, minv, scanned, out);
}

// Eq. 1 terms: acc[0] = sum of internal weight (sum_c sigma_c), acc[1..2] =
// sum_c Sigma_c^2 (i128), acc[3] = 2m.
__global__ void mod_sq_k(int64_t n, const int64_t *Sig, u64 *acc) {
  __shared__ i128 sbuf[32];
  i128 s = 0;
  GRID_STRIDE(c, n) s += (i128)Sig[c] * Sig[c];
  s = block_sum_i128(s, sbuf);
  if (threadIdx.x == 0 && s != 0) atomic_add_i128(&acc[1], s);
}
void launch_modularity_terms(GraphView<int32_t> g, int64_t nnz, const int32_t *C, int64_t *Sig_tmp, u64 *acc,
                             u64 *err, int sms, cudaStream_t s) {
  cudaMemsetAsync(acc, 0, 4 * sizeof(u64), s);
  if (g.n > 0) cudaMemsetAsync(Sig_tmp, 0, (size_t)g.n * sizeof(int64_t), s);
  launch_rows<true>(g, nnz, C, nullptr, Sig_tmp, acc, err, sms, s);
  if (g.n > 0) LK_COUNTED mod_sq_k<<<grid_for(g.n, 256, sms * 8), 256, 0, s>>>(g.n, Sig_tmp, acc);
}

// Sigma[c] = sum of K over members of c (Sigma zeroed first).
__global__ void sigma_from_k(int64_t n, const int32_t *C, const int64_t *K, int64_t *Sig) {
  GRID_STRIDE(i, n) if (K[i]) atomic_add_i64(&Sig[C[i]], K[i]);
}
void launch_sigma_from(int64_t n, const int32_t *C, const int64_t *K, int64_t *Sig, cudaStream_t s) {
  if (n <= 0) return;
  cudaMemsetAsync(Sig, 0, (size_t)n * sizeof(int64_t), s);
  LK_COUNTED sigma_from_k<<<grid_for(n, 256), 256, 0, s>>>(n, C, K, Sig);
}

// ---------------------------------------------------------------------------
// Batch handling.  Every undirected pair (u, v, w) stands for (u,v,w) and
// (v,u,w).
// ---------------------------------------------------------------------------
// Alg. update: K[i] += sign*w, Sigma[C^{t-1}[i]] += sign*w for both ends.
__global__ void update_weights_k(int64_t cnt, const int32_t *src, const int32_t *dst, const int32_t *w,
                                 int sign, const int32_t *Cprev, int64_t *K, int64_t *Sig) {
  GRID_STRIDE(k, cnt) {
    const int64_t x = sign * (int64_t)w[k];
    const int32_t u = src[k], v = dst[k];
    atomic_add_i64(&K[u], x);
    atomic_add_i64(&Sig[Cprev[u]], x);
    atomic_add_i64(&K[v], x);
    atomic_add_i64(&Sig[Cprev[v]], x);
  }
}
void launch_update_weights(int64_t count, const int32_t *src, const int32_t *dst, const int32_t *w,
                           int sign, const int32_t *Cprev, int64_t *K, int64_t *Sig, cudaStream_t s) {
  if (count > 0) LK_COUNTED update_weights_k<<<grid_for(count, 256), 256, 0, s>>>(count, src, dst, w, sign, Cprev, K, Sig);
}

// changedCommunities (reading: the flag of the shared community).
__global__ void changed_k(int64_t cnt, const int32_t *src, const int32_t *dst, const int32_t *Cprev,
                          uint8_t *changed) {
  GRID_STRIDE(k, cnt) {
    const int32_t cu = Cprev[src[k]];
    if (cu == Cprev[dst[k]]) changed[cu] = 1;
  }
}
void launch_changed_communities(int64_t count, const int32_t *src, const int32_t *dst,
                                const int32_t *Cprev, uint8_t *changed, cudaStream_t s) {
  if (count > 0) LK_COUNTED changed_k<<<grid_for(count, 256), 256, 0, s>>>(count, src, dst, Cprev, changed);
}

// Alg. frontier: deletions inside a community (same = 1) and insertions across
// communities (same = 0) mark both ends.
__global__ void mark_df_k(int64_t cnt, const int32_t *src, const int32_t *dst, const int32_t *Cprev,
                          int same, uint8_t *aff) {
  GRID_STRIDE(k, cnt) {
    const int32_t u = src[k], v = dst[k];
    if ((Cprev[u] == Cprev[v]) == (same != 0)) { aff[u] = 1; aff[v] = 1; }
  }
}
void launch_mark_df(int64_t count, const int32_t *src, const int32_t *dst, const int32_t *Cprev,
                    int same, uint8_t *affected, cudaStream_t s) {
  if (count > 0) LK_COUNTED mark_df_k<<<grid_for(count, 256), 256, 0, s>>>(count, src, dst, Cprev, same, affected);
}

// A CSR is well formed: off[0] = 0, off[n] = nnz, offsets non-decreasing,
// column IDs in [0, n), weights > 0.  Sets *err on violation.
// Four entries a load where both arrays start on 16 bytes (vec), else one.
__global__ void check_graph_entries_k(int64_t n, int64_t nnz, const int32_t *idx, const int32_t *w, int vec, u64 *err) {
  bool bad = false;
  const int64_t nv = vec ? nnz / 4 : 0;
  GRID_STRIDE(v, nv) {
    const int4 j = reinterpret_cast<const int4 *>(idx)[v], x = reinterpret_cast<const int4 *>(w)[v];
    bad |= (int64_t)(uint32_t)j.x >= n || (int64_t)(uint32_t)j.y >= n || (int64_t)(uint32_t)j.z >= n ||
           (int64_t)(uint32_t)j.w >= n || x.x <= 0 || x.y <= 0 || x.z <= 0 || x.w <= 0;
  }
  GRID_STRIDE(q, nnz - 4 * nv) bad |= (int64_t)(uint32_t)idx[4 * nv + q] >= n || w[4 * nv + q] <= 0;
  if (bad) atomicOr(err, 256ull);
}
void launch_check_graph(int64_t n, int64_t nnz, const int64_t *off, const int32_t *idx, const int32_t *w,
                        u64 *err, cudaStream_t s) {
  LK_COUNTED check_graph_rows_k<<<grid_for(n > 0 ? n : 1, 256, 152 * 32), 256, 0, s>>>(n, nnz, off, nullptr, err);
  const int vec = (((uintptr_t)idx | (uintptr_t)w) & 15) == 0;
  if (nnz > 0) LK_COUNTED check_graph_entries_k<<<grid_for(nnz, 256, 152 * 32), 256, 0, s>>>(n, nnz, idx, w, vec, err);
}

// Labels in [0, hi); sets *err on violation.
__global__ void check_range_k(const int32_t *a, int64_t n, int64_t hi, u64 *err) {
  GRID_STRIDE(i, n) if (a[i] < 0 || a[i] >= hi) atomicOr(err, 32ull);
}
void launch_check_range(const int32_t *a, int64_t n, int64_t hi, u64 *err, cudaStream_t s) {
  if (n > 0) LK_COUNTED check_range_k<<<grid_for(n, 256), 256, 0, s>>>(a, n, hi, err);
}

// IDs in [0, n), no self-loops, positive weights; sets *err on violation.
__global__ void check_ids_k(int64_t cnt, const int32_t *src, const int32_t *dst, const int32_t *w,
                            int64_t n, u64 *err) {
  GRID_STRIDE(k, cnt) {
    const int32_t u = src[k], v = dst[k];
    if (u < 0 || u >= n || v < 0 || v >= n || u == v || (w && w[k] <= 0)) atomicOr(err, 1ull);
  }
}
void launch_check_ids(int64_t count, const int32_t *src, const int32_t *dst, const int32_t *w,
                      int64_t n, u64 *err, cudaStream_t s) {
  if (count > 0) LK_COUNTED check_ids_k<<<grid_for(count, 256), 256, 0, s>>>(count, src, dst, w, n, err);
}

}  // namespace lk
