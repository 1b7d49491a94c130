// Pipelined tile kernels instantiated for storage type __nv_bfloat162.
#define WSFFT_STORE __nv_bfloat162
#define WSFFT_TILE_NAME launch_tile_c16bf
#include "tile_launch.cuh"
