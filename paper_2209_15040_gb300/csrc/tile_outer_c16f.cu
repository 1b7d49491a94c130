// Fused tile kernels (outer axis and the rest of the middle one; contiguous axis) instantiated for storage type __half2.
#define WSFFT_STORE __half2
#define WSFFT_OUTER_TILE_NAME launch_tile_outer_c16f
#define WSFFT_CONTIG_TILE_NAME launch_tile_contig_c16f
#include "tile_fused_launch.cuh"
