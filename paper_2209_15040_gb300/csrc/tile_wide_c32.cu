// Fused tile kernels (long last axis and a digit of a strided one) instantiated for storage type float2.
#define WSFFT_STORE float2
#define WSFFT_WIDE_TILE_NAME launch_tile_wide_c32
#include "tile_fused_launch.cuh"
