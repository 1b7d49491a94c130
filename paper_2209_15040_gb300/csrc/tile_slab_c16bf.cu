// Fused tile kernels (two inner axes) instantiated for storage type __nv_bfloat162.
#define WSFFT_STORE __nv_bfloat162
#define WSFFT_SLAB_TILE_NAME launch_tile_slab_c16bf
#include "tile_fused_launch.cuh"
