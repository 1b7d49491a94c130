// Fused tile kernels (two inner axes) instantiated for storage type __half2.
#define WSFFT_STORE __half2
#define WSFFT_SLAB_TILE_NAME launch_tile_slab_c16f
#include "tile_fused_launch.cuh"
