// team_n64.cu -- team pass of aggregated levels, 64-bit scores.
#include "team_launch.cuh"

namespace lk {
template int launch_team_pass<int64_t, int64_t>(const TeamArgs<int64_t> &, int, int, cudaStream_t);
template bool team_cluster_fits<int64_t, int64_t>(int);
}  // namespace lk
