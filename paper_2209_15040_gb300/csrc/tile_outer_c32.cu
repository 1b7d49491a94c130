// Fused tile kernels (outer axis and the rest of the middle one) instantiated for storage type float2.
#define WSFFT_STORE float2
#define WSFFT_OUTER_TILE_NAME launch_tile_outer_c32
#include "tile_fused_launch.cuh"
