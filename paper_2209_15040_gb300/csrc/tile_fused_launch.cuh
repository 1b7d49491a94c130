// Instantiation and launch of the fused tile kernels for one storage type.
// Included by tile_slab_*.cu and tile_outer_*.cu (with WSFFT_STORE and
// WSFFT_SLAB_TILE_NAME or WSFFT_OUTER_TILE_NAME defined).
#pragma once

#include <algorithm>

#include "launch_util.h"
#include "tile_desc.h"
#include "tile_fused.cuh"

namespace wsfft {
namespace {

template <class G, class K>
cudaError_t launch_fused(K kern, const void *in, void *out, const TileArgs &a, cudaStream_t st) {
    using S = WSFFT_STORE;
    using SM = TileFusedSmem<G, S>;
    const cudaError_t attr = set_smem_attr(reinterpret_cast<const void *>(kern), SM::BYTES);
    if (attr != cudaSuccess) return attr;
    if (a.tiles <= 0) return cudaSuccess;
    const int sms = device_sms();
    if (sms <= 0) return cudaErrorInvalidDevice;
    const unsigned grid = (unsigned)std::min<int64_t>(a.tiles, (int64_t)sms * SM::CTAS);
    return launch_pdl(pdl_bytes(a.elems * (int64_t)sizeof(S)), kern, grid, 1u << (G::TB - 6), SM::BYTES, st,
                      (const S *)in, (S *)out, a);
}

}  // namespace

#ifdef WSFFT_SLAB_TILE_NAME
cudaError_t WSFFT_SLAB_TILE_NAME(int zb, int yb, const void *in, void *out, const TileArgs &arg, cudaStream_t st) {
    using S = WSFFT_STORE;
    TileArgs a = arg;
    // Few tiles (complex64 slabs of 2^10): a quarter of a tile's elements per
    // block, one warp each; loads, exchanges and stores take a quarter of the
    // time of one block of four.  Four 32^3: 5.7 us back to back and 5.6 captured
    // against 6.6 and 6.7 with tiles of 2^13.
    if constexpr (sizeof(S) == 8)
        if (a.elems <= FUSED_SMALL_ELEMS && zb == 5 && yb == 5) {
            using G = TileSlab<FUSED_SMALL_BITS, 5, 5>;
            a.tiles = (a.elems + (1 << FUSED_SMALL_BITS) - 1) >> FUSED_SMALL_BITS;
            return launch_fused<G>(tile_slab_kernel<G, S, true>, in, out, a, st);
        }
    a.tiles = (a.elems + (1 << FUSED_TILE_BITS) - 1) >> FUSED_TILE_BITS;
#define WSFFT_SLAB(z, y)                                                                          \
    if (zb == z && yb == y)                                                                       \
        return launch_fused<TileSlab<FUSED_TILE_BITS, z, y>>(                                     \
            tile_slab_kernel<TileSlab<FUSED_TILE_BITS, z, y>, S, (z + y < FUSED_TILE_BITS)>, in, out, a, st);
    WSFFT_SLAB(5, 5)
    WSFFT_SLAB(5, 6)
    WSFFT_SLAB(5, 7)
    WSFFT_SLAB(5, 8)
    WSFFT_SLAB(6, 5)
    WSFFT_SLAB(6, 6)
    WSFFT_SLAB(6, 7)
    WSFFT_SLAB(7, 5)
    WSFFT_SLAB(7, 6)
    WSFFT_SLAB(8, 5)
#undef WSFFT_SLAB
    return cudaErrorInvalidValue;
}
#endif

#ifdef WSFFT_CONTIG_TILE_NAME
cudaError_t WSFFT_CONTIG_TILE_NAME(int N, const void *in, void *out, const TileArgs &arg, cudaStream_t st) {
    using S = WSFFT_STORE;
    TileArgs a = arg;
    a.elems = a.npencils * N;
    a.tiles = (a.elems + (1 << FUSED_TILE_BITS) - 1) >> FUSED_TILE_BITS;
#define WSFFT_CONTIG(n, b)                                                                                          \
    if (N == n)                                                                                                     \
        return launch_fused<TileContig<FUSED_TILE_BITS, b>>(tile_slab_kernel<TileContig<FUSED_TILE_BITS, b>, S, true>, in, \
                                                            out, a, st);
    WSFFT_CONTIG(32, 5)
    WSFFT_CONTIG(64, 6)
    WSFFT_CONTIG(128, 7)
#undef WSFFT_CONTIG
    return cudaErrorInvalidValue;
}
#endif

#ifdef WSFFT_WIDE_TILE_NAME
cudaError_t WSFFT_WIDE_TILE_NAME(int zb, int rb, const void *in, void *out, const TileArgs &arg, cudaStream_t st) {
    using S = WSFFT_STORE;
    TileArgs a = arg;
    a.tiles = a.elems >> (zb + rb);
#define WSFFT_WIDE(b, z) \
    if (zb == z && rb == b - z) return launch_fused<TileWide<b, z>>(tile_wide_kernel<TileWide<b, z>, S>, in, out, a, st);
    WSFFT_WIDE(13, 9)
    WSFFT_WIDE(13, 10)
    WSFFT_WIDE(13, 11)
    WSFFT_WIDE(13, 12)
    WSFFT_WIDE(14, 12)
#undef WSFFT_WIDE
    return cudaErrorInvalidValue;
}
#endif

#ifdef WSFFT_OUTER_TILE_NAME
cudaError_t WSFFT_OUTER_TILE_NAME(int xb, int y0b, const void *in, void *out, const TileArgs &arg, cudaStream_t st) {
    using S = WSFFT_STORE;
    TileArgs a = arg;
    a.tiles = a.elems >> FUSED_TILE_BITS;
#define WSFFT_OUTER(x, y)                                                                                            \
    if (xb == x && y0b == y)                                                                                         \
        return launch_fused<TileOuter<FUSED_TILE_BITS, x, y>>(tile_outer_kernel<TileOuter<FUSED_TILE_BITS, x, y>, S>, \
                                                              in, out, a, st);
    WSFFT_OUTER(5, 1)
    WSFFT_OUTER(6, 1)
    WSFFT_OUTER(7, 1)
    WSFFT_OUTER(8, 1)
    WSFFT_OUTER(5, 2)
    WSFFT_OUTER(6, 2)
    WSFFT_OUTER(7, 2)
    WSFFT_OUTER(5, 3)
    WSFFT_OUTER(6, 3)
    WSFFT_OUTER(5, 4)
#undef WSFFT_OUTER
    return cudaErrorInvalidValue;
}
#endif

}  // namespace wsfft
