// Fused tile kernels (outer axis and the rest of the middle one; contiguous axis) instantiated for storage type float2.
#define WSFFT_STORE float2
#define WSFFT_OUTER_TILE_NAME launch_tile_outer_c32
#define WSFFT_CONTIG_TILE_NAME launch_tile_contig_c32
#include "tile_fused_launch.cuh"
