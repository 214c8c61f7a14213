// team_n32.cu -- team pass of the first level (int32 weights), 64-bit scores.
#include "team_launch.cuh"

namespace lk {
template int launch_team_pass<int32_t, int64_t>(const TeamArgs<int32_t> &, int, int, cudaStream_t);
template bool team_cluster_fits<int32_t, int64_t>(int);
}  // namespace lk
