// team_w64.cu -- team pass of aggregated levels, 128-bit scores.
#include "team_launch.cuh"

namespace lk {
template int launch_team_pass<int64_t, i128>(const TeamArgs<int64_t> &, int, int, cudaStream_t);
template bool team_cluster_fits<int64_t, i128>(int);
}  // namespace lk
