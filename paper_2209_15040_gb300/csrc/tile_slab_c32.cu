// Fused tile kernels (two inner axes) instantiated for storage type float2.
#define WSFFT_STORE float2
#define WSFFT_SLAB_TILE_NAME launch_tile_slab_c32
#include "tile_fused_launch.cuh"
