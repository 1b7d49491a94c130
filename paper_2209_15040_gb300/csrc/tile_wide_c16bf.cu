// Fused tile kernels (long last axis and a digit of a strided one) instantiated for storage type __nv_bfloat162.
#define WSFFT_STORE __nv_bfloat162
#define WSFFT_WIDE_TILE_NAME launch_tile_wide_c16bf
#include "tile_fused_launch.cuh"
