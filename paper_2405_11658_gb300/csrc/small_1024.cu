// small_1024.cu -- the batch kernel with 1024 threads a block.
#define LK_TEAM_THREADS 1024
#include "small.cuh"
