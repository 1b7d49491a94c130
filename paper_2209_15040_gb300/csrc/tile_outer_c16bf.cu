// Fused tile kernels (outer axis and the rest of the middle one) instantiated for storage type __nv_bfloat162.
#define WSFFT_STORE __nv_bfloat162
#define WSFFT_OUTER_TILE_NAME launch_tile_outer_c16bf
#include "tile_fused_launch.cuh"
