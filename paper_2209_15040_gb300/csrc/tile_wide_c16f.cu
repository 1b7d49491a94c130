// Fused tile kernels (long last axis and a digit of a strided one) instantiated for storage type __half2.
#define WSFFT_STORE __half2
#define WSFFT_WIDE_TILE_NAME launch_tile_wide_c16f
#include "tile_fused_launch.cuh"
