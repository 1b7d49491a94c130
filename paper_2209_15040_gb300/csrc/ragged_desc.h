// Host-visible interface of the ragged-batch kernel (ragged.cuh).
#pragma once

#include <cuda_runtime.h>

namespace wsfft {

struct RagArgs;

// One instance of a ragged batch (device table; pointers filled per execute).
struct RagInst {
    const void *in;
    void *out;
    int n[3];          // axis lengths, n[2] contiguous
    int log_n2, log_n12;
    int tiles[3];      // queue: tiles of the z, y, x supersteps
    float scale[3];    // queue: store scale of the z, y, x supersteps
    int log_y0;        // grouped: residue classes of the middle axis (tile_fused.cuh)
    float first, last; // grouped: store scale of the first and the last trip
};

// Grouped launches: the tile of an instance that a launch's tile is.
struct alignas(8) RagRef {
    int inst, tile;
};

// grid_per_sm != NULL: only report how many blocks fit on one SM.
cudaError_t launch_ragged_c32(const RagArgs &a, int *grid_per_sm, int grid, cudaStream_t st);
cudaError_t launch_ragged_c16f(const RagArgs &a, int *grid_per_sm, int grid, cudaStream_t st);
cudaError_t launch_ragged_c16bf(const RagArgs &a, int *grid_per_sm, int grid, cudaStream_t st);

}  // namespace wsfft
