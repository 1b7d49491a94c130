// Instantiation and launch of the pipelined tile kernels for one storage type.
// Included once per storage type by tile_c32.cu, tile_c16f.cu, tile_c16bf.cu
// (with WSFFT_STORE and WSFFT_TILE_NAME defined).
#pragma once

#include <algorithm>

#include "launch_util.h"
#include "tile.cuh"
#include "tile_desc.h"

namespace wsfft {
namespace {

// Persistent launch: as many blocks as are resident at once, each taking
// every grid-size-th tile.  Whole tiles of adjacent pencils only.
template <int TB, int NB>
cudaError_t launch_tile_strided(const void *in, void *out, PassArgs a, cudaStream_t st) {
    using S = WSFFT_STORE;
    using G = TileStrided<TB, NB>;
    using SM = TileSmem<G, S>;
    auto kern = tile_strided_kernel<G, S>;
    const cudaError_t attr = set_smem_attr(reinterpret_cast<const void *>(kern), SM::BYTES);
    if (attr != cudaSuccess) return attr;
    if (a.npencils <= 0) return cudaSuccess;
    if (a.npencils % G::W != 0 || a.inner % G::W != 0) return cudaErrorInvalidValue;
    a.tiles = a.npencils / G::W;
    const int sms = device_sms();
    if (sms <= 0) return cudaErrorInvalidDevice;
    const unsigned grid = (unsigned)std::min<int64_t>(a.tiles, (int64_t)sms * SM::CTAS);
    return launch_pdl(pdl_bytes((a.npencils << NB) * (int64_t)sizeof(S)), kern, grid, 1u << (TB - 6), SM::BYTES, st,
                      (const S *)in, (S *)out, a);
}

}  // namespace

cudaError_t WSFFT_TILE_NAME(int N, int tb, const void *in, void *out, const PassArgs &a, cudaStream_t st) {
    if (N == 1024 && tb == 14) return launch_tile_strided<14, 10>(in, out, a, st);
    if constexpr (sizeof(WSFFT_STORE) == 4) {
        if (N == 512 && tb == 14) return launch_tile_strided<14, 9>(in, out, a, st);
        if (N == 512 && tb == 13) return launch_tile_strided<13, 9>(in, out, a, st);
        if (N == 256 && tb == 14) return launch_tile_strided<14, 8>(in, out, a, st);
        if (N == 256 && tb == 13) return launch_tile_strided<13, 8>(in, out, a, st);
        if (N == 128 && tb == 13) return launch_tile_strided<13, 7>(in, out, a, st);
        if (N == 64 && tb == 13) return launch_tile_strided<13, 6>(in, out, a, st);
        if (N == 32 && tb == 13) return launch_tile_strided<13, 5>(in, out, a, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace wsfft
