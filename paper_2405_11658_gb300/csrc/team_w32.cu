// team_w32.cu -- team pass of the first level (int32 weights), 128-bit scores.
#include "team_launch.cuh"

namespace lk {
template int launch_team_pass<int32_t, i128>(const TeamArgs<int32_t> &, int, int, cudaStream_t);
template bool team_cluster_fits<int32_t, i128>(int);
}  // namespace lk
