// small_512.cu -- the batch kernel with 512 threads a block.
#define LK_TEAM_THREADS 512
#include "small.cuh"
