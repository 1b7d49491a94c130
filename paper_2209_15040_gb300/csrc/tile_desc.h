// Host-visible interface of the pipelined tile kernels (tile.cuh).
#pragma once

#include <cuda_runtime.h>

#include "pass_desc.h"

namespace wsfft {

// Supersteps of the tile kernels.
enum {
    TILE_STRIDED = 0,       // strided axis
    TILE_STRIDED_TWID = 1,  // strided axis, four-step twiddle on the store
    TILE_TRANS = 2,         // contiguous axis, transposed store
    TILE_STRIDED_RAG = 3    // strided axis, instances of a ragged batch
};

// Values per thread of the twiddle table a tile kernel's axis of length N
// uses: the radix of its first stage.
inline int tile_table_E(int N) { return N <= 64 ? 8 : N <= 256 || N >= 2048 ? 16 : 32; }

// Launch one superstep on the pipelined tile kernels.  tb: log2 of the
// elements per tile.  Returns cudaErrorInvalidValue
// for a shape that is not instantiated or does not divide into whole tiles.
cudaError_t launch_tile_c32(int mode, int N, int tb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_c16f(int mode, int N, int tb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_c16bf(int mode, int N, int tb, const void *in, void *out, const TileArgs &a, cudaStream_t st);

// Fused tile kernels (tile_fused.cuh), tiles of 2^13 elements.
constexpr int FUSED_TILE_BITS = 13;
// Up to this many elements 32 x 32 slabs run in tiles of 2^11 (complex64), others
// one launch per axis (Plan::build_fused).
constexpr int64_t FUSED_SMALL_ELEMS = (int64_t)1 << 17;
constexpr int FUSED_SMALL_BITS = 11;

// The two inner axes of slabs (2^zb points contiguous, 2^yb rows): whole
// slabs where zb + yb < 13, in place or not; for zb + yb = 13 the 2^yb rows of
// each residue class of larger slabs (log_y0 of TileArgs; out of place unless
// it is 0).  cudaErrorInvalidValue for sizes that are not built.
cudaError_t launch_tile_slab_c32(int zb, int yb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_slab_c16f(int zb, int yb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_slab_c16bf(int zb, int yb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
// Contiguous pencils of N = 32, 64 or 128 points, any number of them, in place or not.
cudaError_t launch_tile_contig_c32(int N, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_contig_c16f(int N, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_contig_c16bf(int N, const void *in, void *out, const TileArgs &a, cudaStream_t st);
// A last axis of 2^zb = 512..4096 points and a digit of 2^rb points of a
// strided axis; out of place.
cudaError_t launch_tile_wide_c32(int zb, int rb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_wide_c16f(int zb, int rb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_wide_c16bf(int zb, int rb, const void *in, void *out, const TileArgs &a, cudaStream_t st);
// The outer axis (2^xb points) and the 2^y0b residue classes.
cudaError_t launch_tile_outer_c32(int xb, int y0b, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_outer_c16f(int xb, int y0b, const void *in, void *out, const TileArgs &a, cudaStream_t st);
cudaError_t launch_tile_outer_c16bf(int xb, int y0b, const void *in, void *out, const TileArgs &a, cudaStream_t st);

// The same for tiles of several instances of a ragged batch (complex64):
// a.refs[tile] for `a.tiles` tiles.
cudaError_t launch_ragged_slab_c32(int zb, int yb, const TileArgs &a, cudaStream_t st);
cudaError_t launch_ragged_outer_c32(int xb, int y0b, const TileArgs &a, cudaStream_t st);
cudaError_t launch_ragged_strided_c32(int N, const TileArgs &a, cudaStream_t st);

}  // namespace wsfft
