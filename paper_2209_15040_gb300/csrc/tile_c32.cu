// Pipelined tile kernels instantiated for storage type float2.
#define WSFFT_STORE float2
#define WSFFT_TILE_NAME launch_tile_c32
#include "tile_launch.cuh"
