// batch.cu -- host driver of the persistent many-graph kernel
// (leiden_batch_*): workspace carving, job descriptors, and the CUDA graph
// that uploads the descriptors, runs the kernel and downloads the results in
// one launch.
#include <string.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include "internal.h"
#include "leiden.h"
#include "small.h"

using namespace lk;

struct leiden_batch {
  cudaStream_t st = nullptr;     // the caller's stream: every run is ordered on it
  cudaStream_t cap = nullptr;    // private stream the CUDA graph is captured on
  int device = 0, sms = 152, max_cluster = 1;
  int32_t max_graphs = 0;
  int64_t max_n = 0, max_nnz = 0;
  char *arena = nullptr;
  int64_t arena_bytes = 0;
  char *d_desc = nullptr;        // SmallHeader, then SmallJob[max_graphs]
  SmallResult *d_res = nullptr;
  SmallCtl *d_ctl = nullptr;     // control words of every block (d_desc's allocation)
  char *h_desc = nullptr;        // pinned staging of d_desc
  SmallResult *h_res = nullptr;  // pinned copy of d_res
  size_t desc_bytes = 0, res_bytes = 0;
  // one captured graph per shape used so far (clusters of 2^k blocks, of 512 or
  // 1024 threads), with the options baked into it
  static constexpr int SHAPES = 10;
  cudaGraph_t graph[SHAPES] = {};
  cudaGraphExec_t exec[SHAPES] = {};
  SmallOpts captured[SHAPES] = {};
};

namespace {

void release(leiden_batch *b) {
  for (int k = 0; k < leiden_batch::SHAPES; k++) {
    if (b->exec[k]) cudaGraphExecDestroy(b->exec[k]);
    if (b->graph[k]) cudaGraphDestroy(b->graph[k]);
  }
  if (b->arena) cudaFree(b->arena);
  if (b->d_desc) cudaFree(b->d_desc);      // also d_res, d_ctl
  if (b->h_desc) cudaFreeHost(b->h_desc);  // also h_res
  if (b->cap) cudaStreamDestroy(b->cap);
}

int opts_to_small(const leiden_opts *o, SmallOpts *so) {
  if (!o || o->sched != LEIDEN_DET) return LEIDEN_EINVAL;
  if (o->max_iters < 1 || o->max_passes < 1 || !(o->tol >= 0.0) || !(o->tol_drop > 0.0)) return LEIDEN_EINVAL;
  if (o->reserved[0] || o->reserved[1] || o->reserved[2]) return LEIDEN_EINVAL;
  const int S = o->det_subsets;
  if (S < 1 || S > 256 || (S & (S - 1))) return LEIDEN_EINVAL;
  int k = 0;
  while ((1 << k) < S) k++;
  const double scaled = o->gamma * 1048576.0;
  if (!(o->gamma > 0.0) || scaled > 9.0e15) return LEIDEN_EINVAL;
  int64_t p = (int64_t)scaled;
  if ((double)p != scaled) return LEIDEN_EINVAL;
  int64_t q = 1048576, a = p, bb = q;
  while (bb) { const int64_t t = a % bb; a = bb; bb = t; }
  so->p = p / a;
  so->q = q / a;
  so->tol = o->tol;
  so->tol_drop = o->tol_drop;
  so->max_iters = o->max_iters;
  so->max_passes = o->max_passes;
  so->log2S = k;
  so->refine_all_first_pass = o->refine_all_first_pass ? 1 : 0;
  return LEIDEN_OK;
}

int check_item(const leiden_batch_item &it) {
  const leiden_csr &g = it.g;
  if (g.n < 0 || g.nnz < 0 || g.n >= INT32_MAX || !g.off) return LEIDEN_EINVAL;
  if (g.nnz > 0 && (!g.idx || !g.w)) return LEIDEN_EINVAL;
  if (g.n > 0 && !it.membership_out) return LEIDEN_EINVAL;
  if (it.reserved != 0) return LEIDEN_EINVAL;
  if (it.mode == LEIDEN_STATIC) return LEIDEN_OK;
  if (it.mode != LEIDEN_ND && it.mode != LEIDEN_DS && it.mode != LEIDEN_DF) return LEIDEN_EINVAL;
  if (g.n > 0 && !it.prior) return LEIDEN_EINVAL;
  if (it.del.count < 0 || it.ins.count < 0) return LEIDEN_EINVAL;
  if (it.del.count > 0 && (!it.del.src || !it.del.dst || !it.del.w)) return LEIDEN_EINVAL;
  if (it.ins.count > 0 && (!it.ins.src || !it.ins.dst || !it.ins.w)) return LEIDEN_EINVAL;
  return LEIDEN_OK;
}

// Cluster size (2^log2) and threads of a block, and the graphs run by clusters.
struct Shape {
  int log2 = 0, threads = 512;
  int32_t wide = 0;
  int index() const { return 2 * log2 + (threads == 1024); }
};

// (Re)captures upload + kernel + download for opts `so` and a shape.
int capture(leiden_batch *b, const SmallOpts &so, const Shape &sh) {
  const int k = sh.index();
  if (b->exec[k]) { cudaGraphExecDestroy(b->exec[k]); b->exec[k] = nullptr; }
  if (b->graph[k]) { cudaGraphDestroy(b->graph[k]); b->graph[k] = nullptr; }
  if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return LEIDEN_ECUDA;
  }
  SmallHeader *hdr = reinterpret_cast<SmallHeader *>(b->d_desc);
  const SmallJob *jobs = reinterpret_cast<const SmallJob *>(b->d_desc + sizeof(SmallHeader));
  cudaMemcpyAsync(b->d_desc, b->h_desc, b->desc_bytes, cudaMemcpyHostToDevice, b->cap);
  const int rc = sh.threads == 512
                     ? launch_small<512>(hdr, jobs, so, b->d_res, b->d_ctl, b->sms, 1 << sh.log2, b->cap)
                     : launch_small<1024>(hdr, jobs, so, b->d_res, b->d_ctl, b->sms, 1 << sh.log2, b->cap);
  cudaMemcpyAsync(b->h_res, b->d_res, b->res_bytes, cudaMemcpyDeviceToHost, b->cap);
  cudaGraph_t g = nullptr;
  if (cudaStreamEndCapture(b->cap, &g) != cudaSuccess || !g || rc) {
    cudaGetLastError();
    if (g) cudaGraphDestroy(g);
    return LEIDEN_ECUDA;
  }
  if (cudaGraphInstantiate(&b->exec[k], g, 0) != cudaSuccess) {
    cudaGetLastError();
    b->exec[k] = nullptr;
    cudaGraphDestroy(g);
    return LEIDEN_ECUDA;
  }
  b->graph[k] = g;
  b->captured[k] = so;
  return LEIDEN_OK;
}

// Clusters of 2^k blocks for the largest `wide` of the graphs (sizes: their
// vertices + entries, largest first), single blocks for the others.  A cluster
// of c blocks for w graphs leaves sms - w c blocks for the other count - w, so
// w = (sms - count) / (c - 1) keeps every graph on SMs of its own; the largest
// c that still covers a third of the graphs (their sizes differ, and the
// largest ones finish last).  A graph below 6144 c is not worth the cluster's
// barriers, about 1 us each against the block's 0.05.  Clusters have at most
// `most` blocks, what the device can keep resident.  64 graphs of 1e3..1e4
// vertices (1.1e4 .. 1.1e5) get clusters of 4 for up to 29 of them; with 1024
// threads throughout, single blocks took 28.4 ms, clusters of 2 for all 19.7,
// of 4 for all 20.0, of 8 for the 20 largest 26.9, of 4 for the 20 largest 18.3.
//
// 512 threads (see small.cuh) while no block has much of a graph; with more
// colour classes S, a sub-sweep has less of it.  ms with 1024 / 512 threads by
// the largest share of a block: S = 8: 3.3e3 4.7 / 2.7, 2.7e4 to 4.9e4 14.2 /
// 12.7 (the 64 graphs), 21.0 / 20.6 and 17.3 / 17.2, 5.2e4 18.2 / 18.7, 1.1e5
// 33.5 / 36.2, 3.2e5 65.9 / 78.6; S = 1: about 3e4 7.3 / 7.0, 5.5e4 12.5 /
// 13.2; S = 32: 1.1e5 46.6 / 45.1, 2.5e5 40.8 / 41.4, 3.2e5 60.7 / 64.5;
// S = 256: 5.5e4 132 / 81.
Shape batch_shape(int count, int sms, int most, int log2S, const std::vector<int64_t> &sizes) {
  Shape sh;
  for (int k = 4; k > 0; k--) {
    const int c = 1 << k;
    if (c > most) continue;
    const int w = std::min(count, std::max(0, (sms - count) / (c - 1)));
    if (3 * w < count || sizes[0] < (int64_t)6144 * c) continue;
    sh.log2 = k;
    while (sh.wide < w && sizes[sh.wide] >= (int64_t)3072 * c) ++sh.wide;
    break;
  }
  int64_t share = sizes[0] >> sh.log2;   // sizes[0] is on a cluster if any graph is
  if (sh.wide < count) share = std::max(share, sizes[sh.wide]);
  if (share > 24576 + ((int64_t)3072 << log2S)) sh.threads = 1024;
  return sh;
}

bool same_opts(const SmallOpts &a, const SmallOpts &b) { return memcmp(&a, &b, sizeof(SmallOpts)) == 0; }

}  // namespace

extern "C" int leiden_batch_create(leiden_batch **out, void *stream, int32_t max_graphs, int64_t max_total_n,
                                   int64_t max_total_nnz, int32_t threads, int32_t blocks_per_sm) {
  if (!out || max_graphs < 1 || max_total_n < 0 || max_total_nnz < 0) return LEIDEN_EINVAL;
  // each run picks its shape (batch_shape); the two arguments are only checked
  if (threads && (threads < 128 || threads > 512 || threads % 32)) return LEIDEN_EINVAL;
  if (blocks_per_sm && (blocks_per_sm < 1 || blocks_per_sm > 4)) return LEIDEN_EINVAL;
  leiden_batch *b = new leiden_batch();
  b->st = (cudaStream_t)stream;
  b->max_graphs = max_graphs;
  b->max_n = max_total_n;
  b->max_nnz = max_total_nnz;
  int rc = LEIDEN_OK;
  if (cudaGetDevice(&b->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device) != cudaSuccess ||
      cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess) {
    rc = LEIDEN_ECUDA;
  }
  if (!rc) b->max_cluster = std::min(small_max_cluster<512>(), small_max_cluster<1024>());
  b->arena_bytes = small_layout_bound(max_total_n, max_total_nnz, max_graphs);
  b->desc_bytes = sizeof(SmallHeader) + (size_t)max_graphs * sizeof(SmallJob);
  b->res_bytes = (size_t)max_graphs * sizeof(SmallResult);
  // one device and one pinned allocation for the descriptors, the results and
  // the blocks' control words
  const size_t ctl_bytes = (size_t)b->sms * sizeof(SmallCtl);
  const size_t desc_al = (b->desc_bytes + 255) & ~(size_t)255, res_al = (b->res_bytes + 255) & ~(size_t)255;
  if (!rc && (cudaMalloc(&b->arena, (size_t)b->arena_bytes) != cudaSuccess ||
              cudaMalloc(&b->d_desc, desc_al + res_al + ctl_bytes) != cudaSuccess ||
              cudaMallocHost(&b->h_desc, desc_al + b->res_bytes) != cudaSuccess))
    rc = LEIDEN_ENOMEM;
  if (rc) {
    cudaGetLastError();
    release(b);
    delete b;
    return rc;
  }
  b->d_res = reinterpret_cast<SmallResult *>(b->d_desc + desc_al);
  b->d_ctl = reinterpret_cast<SmallCtl *>(b->d_desc + desc_al + res_al);
  b->h_res = reinterpret_cast<SmallResult *>(b->h_desc + desc_al);
  memset(b->h_desc, 0, b->desc_bytes);
  *out = b;
  return LEIDEN_OK;
}

extern "C" void leiden_batch_destroy(leiden_batch *b) {
  if (!b) return;
  cudaStreamSynchronize(b->st);
  cudaStreamSynchronize(b->cap);
  release(b);
  delete b;
}

extern "C" int leiden_batch_device_bytes(leiden_batch *b, int64_t *out) {
  if (!b || !out) return LEIDEN_EINVAL;
  *out = b->arena_bytes + (int64_t)b->desc_bytes + (int64_t)b->res_bytes + (int64_t)b->sms * (int64_t)sizeof(SmallCtl);
  return LEIDEN_OK;
}

extern "C" int leiden_batch_run(leiden_batch *b, int32_t count, const leiden_batch_item *items,
                                const leiden_opts *opts, leiden_batch_result *results) {
  if (!b || count < 0 || (count > 0 && (!items || !results))) return LEIDEN_EINVAL;
  if (count > b->max_graphs) return LEIDEN_ENOMEM;
  SmallOpts so{};
  int rc = opts_to_small(opts, &so);
  if (rc) return rc;
  int64_t sum_n = 0, sum_nnz = 0;
  for (int k = 0; k < count; k++) {
    rc = check_item(items[k]);
    if (rc) return rc;
    sum_n += items[k].g.n;
    sum_nnz += items[k].g.nnz;
  }
  if (sum_n > b->max_n || sum_nnz > b->max_nnz) return LEIDEN_ENOMEM;
  if (count == 0) return LEIDEN_OK;
  // largest graphs first, so the last graphs to start are the shortest
  std::vector<int> order(count);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return items[x].g.nnz + items[x].g.n > items[y].g.nnz + items[y].g.n;
  });
  SmallHeader *hdr = reinterpret_cast<SmallHeader *>(b->h_desc);
  SmallJob *jobs = reinterpret_cast<SmallJob *>(b->h_desc + sizeof(SmallHeader));
  memset(hdr, 0, sizeof(SmallHeader));
  hdr->count = count;
  std::vector<int64_t> sizes(count);
  for (int k = 0; k < count; k++) sizes[k] = items[order[k]].g.nnz + items[order[k]].g.n;
  const Shape sh = batch_shape(count, b->sms, b->max_cluster, so.log2S, sizes);
  const int x = sh.index();
  hdr->wide = sh.wide;
  hdr->next = 0;
  hdr->next1 = (uint32_t)hdr->wide;
  int64_t at = 0;
  for (int k = 0; k < count; k++) {
    const leiden_batch_item &it = items[order[k]];
    SmallJob &j = jobs[k];
    memset(&j, 0, sizeof(j));
    j.n = it.g.n;
    j.nnz = it.g.nnz;
    j.off = it.g.off;
    j.idx = it.g.idx;
    j.w = it.g.w;
    j.mode = it.mode;
    j.out = it.membership_out;
    j.result = order[k];
    if (it.mode != LEIDEN_STATIC) {
      j.prior = it.prior;
      j.nd = it.del.count;
      j.ni = it.ins.count;
      j.ds = it.del.src; j.dd = it.del.dst; j.dw = it.del.w;
      j.is = it.ins.src; j.id = it.ins.dst; j.iw = it.ins.w;
    }
    j.ws = b->arena + at;
    at += small_layout(it.g.n, it.g.nnz).total;
  }
  if (at > b->arena_bytes) return LEIDEN_ENOMEM;  // cannot happen within the totals; kept as a guard
  // the previous run's graph is still in flight until this stream point
  if (!b->exec[x] || !same_opts(so, b->captured[x])) {
    cudaStreamSynchronize(b->st);
    rc = capture(b, so, sh);
    if (rc) return rc;
  }
  note_launch();
  if (cudaGraphLaunch(b->exec[x], b->st) != cudaSuccess) {
    cudaGetLastError();
    return LEIDEN_ECUDA;
  }
  if (cudaStreamSynchronize(b->st) != cudaSuccess || cudaGetLastError() != cudaSuccess) return LEIDEN_ECUDA;
  for (int k = 0; k < count; k++) {
    const SmallResult &r = b->h_res[k];
    leiden_batch_result &o = results[k];
    memset(&o, 0, sizeof(o));
    o.status = r.status;
    o.passes = r.passes;
    o.affected0 = r.affected0;
    o.changed0 = r.changed0;
    const int np = std::min<int>(r.passes, LEIDEN_STATS_PASSES);
    for (int p = 0; p < np; p++) {
      o.iters[p] = r.iters[p];
      o.nv[p] = r.nv[p];
      o.nnz[p] = r.nnz[p];
      o.moves[p] = r.moves[p];
      o.refine_moves[p] = r.refine_moves[p];
    }
    if (r.status == LEIDEN_OK) {
      const i128 sq = (i128)(((unsigned __int128)r.sq_hi << 64) | (unsigned __int128)r.sq_lo);
      const i128 num = (i128)so.q * r.two_m * r.inside - (i128)so.p * sq;
      o.q = r.two_m == 0 ? 0.0 : (double)num / ((double)r.two_m * (double)r.two_m * (double)so.q);
    }
  }
  return LEIDEN_OK;
}
