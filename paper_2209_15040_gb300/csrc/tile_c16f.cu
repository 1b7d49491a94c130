// Pipelined tile kernels instantiated for storage type __half2.
#define WSFFT_STORE __half2
#define WSFFT_TILE_NAME launch_tile_c16f
#include "tile_launch.cuh"
