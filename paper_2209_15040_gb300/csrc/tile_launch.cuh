// Instantiation and launch of the pipelined tile kernels for one storage type.
// Included once per storage type by tile_c32.cu, tile_c16f.cu, tile_c16bf.cu
// (with WSFFT_STORE and WSFFT_TILE_NAME defined).
#pragma once

#include <algorithm>
#include <type_traits>

#include "launch_util.h"
#include "tile.cuh"
#include "tile_desc.h"

namespace wsfft {
namespace {

// Persistent launch: as many blocks as are resident at once, each taking
// every grid-size-th tile.  Whole tiles of adjacent pencils only.
template <int TB, int NB, int MODE>
cudaError_t launch_tile_axis(const void *in, void *out, TileArgs a, cudaStream_t st) {
    using S = WSFFT_STORE;
    using G = std::conditional_t<MODE == TILE_TRANS, TileTrans<TB, NB, (int)sizeof(S)>, TileStrided<TB, NB>>;
    using SM = TileSmem<G, S, MODE>;
    auto kern = tile_axis_kernel<G, S, MODE>;
    const cudaError_t attr = set_smem_attr(reinterpret_cast<const void *>(kern), SM::BYTES);
    if (attr != cudaSuccess) return attr;
    if (a.npencils <= 0) return cudaSuccess;
    if (a.npencils % G::W != 0 || (MODE == TILE_TRANS ? a.trans_rows : a.inner) % G::W != 0)
        return cudaErrorInvalidValue;
    a.tiles = a.npencils / G::W;
    const int sms = device_sms();
    if (sms <= 0) return cudaErrorInvalidDevice;
    const unsigned grid = (unsigned)std::min<int64_t>(a.tiles, (int64_t)sms * SM::CTAS);
    return launch_pdl(pdl_bytes((a.npencils << NB) * (int64_t)sizeof(S)), kern, grid, 1u << (TB - 6), SM::BYTES, st,
                      (const S *)in, (S *)out, a);
}

}  // namespace

cudaError_t WSFFT_TILE_NAME(int mode, int N, int tb, const void *in, void *out, const TileArgs &a, cudaStream_t st) {
    constexpr bool half = sizeof(WSFFT_STORE) == 4;
#define WSFFT_TILE(m, n, b, nb) \
    if (mode == m && N == n && tb == b) return launch_tile_axis<b, nb, m>(in, out, a, st);
    WSFFT_TILE(TILE_STRIDED, 1024, 14, 10)
    WSFFT_TILE(TILE_STRIDED, 2048, 14, 11)
    WSFFT_TILE(TILE_STRIDED_TWID, 512, 13, 9)
    WSFFT_TILE(TILE_STRIDED_TWID, 256, 13, 8)
    if constexpr (!half) {
        WSFFT_TILE(TILE_STRIDED, 1024, 13, 10)
        WSFFT_TILE(TILE_STRIDED_TWID, 1024, 13, 10)
        WSFFT_TILE(TILE_TRANS, 1024, 14, 10)
    } else {
        WSFFT_TILE(TILE_STRIDED_TWID, 1024, 14, 10)
        WSFFT_TILE(TILE_TRANS, 1024, 13, 10)
        WSFFT_TILE(TILE_STRIDED, 4096, 14, 12)
        WSFFT_TILE(TILE_STRIDED, 512, 14, 9)
        WSFFT_TILE(TILE_STRIDED, 512, 13, 9)
        WSFFT_TILE(TILE_STRIDED, 256, 14, 8)
        WSFFT_TILE(TILE_STRIDED, 256, 13, 8)
        WSFFT_TILE(TILE_STRIDED, 128, 13, 7)
        WSFFT_TILE(TILE_STRIDED, 64, 13, 6)
        WSFFT_TILE(TILE_STRIDED, 32, 13, 5)
        WSFFT_TILE(TILE_STRIDED_TWID, 128, 13, 7)
        WSFFT_TILE(TILE_STRIDED_TWID, 64, 13, 6)
        WSFFT_TILE(TILE_TRANS, 512, 13, 9)
        WSFFT_TILE(TILE_TRANS, 256, 13, 8)
        WSFFT_TILE(TILE_TRANS, 128, 13, 7)
        WSFFT_TILE(TILE_TRANS, 64, 13, 6)
    }
#undef WSFFT_TILE
    return cudaErrorInvalidValue;
}

}  // namespace wsfft
