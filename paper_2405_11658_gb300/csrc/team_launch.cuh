// team_launch.cuh -- the launch of a team pass (team.cuh) for a context.  Each
// weight type and score width is instantiated in a file of its own
// (team_*.cu), because one kernel takes the compiler a good twenty seconds.
#pragma once

#include <array>
#include <map>
#include <mutex>

#include "team.cuh"

namespace lk {

template <typename WT, typename ST>
__global__ void __launch_bounds__(TEAM_THREADS, 1) team_pass_k(TeamArgs<WT> args, int kind) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ TeamShared<ST> sm;
  if (threadIdx.x == 0) sm.dead = 0;
  __syncthreads();
  Team t;
  t.rank = blockIdx.x;
  t.nb = gridDim.x;
  t.kind = kind;
  t.gen = 0;
  t.ctl = args.ctl;
  t.dead_s = &sm.dead;
  t.dead = false;
  TeamConst ct;
  ct.A = args.A;
  ct.p = args.p;
  ct.den = args.den;
  ct.two_m = args.two_m;
  ct.log2S = args.log2S;
  ct.dynamic = args.dynamic;
  ct.timing = args.timing;
  ct.in_range = args.in_range;
  const TeamLevel<WT> g{args.g.n, args.nnz, args.g.off, args.g.idx, args.g.w};
  TeamArrays a = args.a;
  team_pass<false, WT, ST>(g, a, ct, args.lp, args.tau, args.max_iters, args.agg_slots, t, dyn, sm);
}

template <typename WT, typename ST>
static size_t team_smem() {
  return (size_t)TEAM_WARPS * TEAM_WSLOTS * (sizeof(typename TableVal<ST>::type) + sizeof(int32_t));
}

// Whether a cluster of nb team blocks can be resident on the current device
// (asked once per device and size).
template <typename WT, typename ST>
bool team_cluster_fits(int nb) {
  static std::mutex mu;
  static std::map<int, std::array<int, TEAM_MAX_CLUSTER + 1>> known;   // by device; 0: not asked, 1: yes, 2: no
  if (nb < 2 || nb > TEAM_MAX_CLUSTER) return false;
  const int dev = current_device();
  std::lock_guard<std::mutex> lock(mu);
  int &fits = known[dev][nb];
  if (fits) return fits == 1;
  auto k = team_pass_k<WT, ST>;
  ensure_smem((const void *)k, team_smem<WT, ST>());
  ensure_wide_clusters((const void *)k);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)nb, 1, 1);
  cfg.blockDim = dim3(TEAM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = team_smem<WT, ST>();
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)nb;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, (const void *)k, &cfg) != cudaSuccess) n = 0;
  (void)cudaGetLastError();
  fits = n > 0 ? 1 : 2;
  return n > 0;
}

template <typename WT, typename ST>
int launch_team_pass(const TeamArgs<WT> &args, int nb, int kind, cudaStream_t s) {
  auto k = team_pass_k<WT, ST>;
  const size_t smem = team_smem<WT, ST>();
  ensure_smem((const void *)k, smem);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)nb, 1, 1);
  cfg.blockDim = dim3(TEAM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  if (kind == TEAM_CLUSTER) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)nb;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
  } else {
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
  }
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k, args, kind) != cudaSuccess) {
    (void)cudaGetLastError();
    return LEIDEN_ECUDA;
  }
  note_launch();
  return LEIDEN_OK;
}

}  // namespace lk
