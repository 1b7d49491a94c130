// Fused tile kernels (outer axis and the rest of the middle one; contiguous axis) instantiated for storage type __nv_bfloat162.
#define WSFFT_STORE __nv_bfloat162
#define WSFFT_OUTER_TILE_NAME launch_tile_outer_c16bf
#define WSFFT_CONTIG_TILE_NAME launch_tile_contig_c16bf
#include "tile_fused_launch.cuh"
