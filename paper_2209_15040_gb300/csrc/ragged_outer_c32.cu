// Last trips of a ragged batch in groups (tile_fused.cuh, tile.cuh): one
// launch per tile shape over all instances that have it, complex64.
#include <algorithm>

#include "launch_util.h"
#include "tile_desc.h"
#include "tile_fused.cuh"

namespace wsfft {
namespace {

template <class SM, class K>
cudaError_t launch_grouped(K kern, unsigned threads, const TileArgs &a, cudaStream_t st) {
    const cudaError_t attr = set_smem_attr(reinterpret_cast<const void *>(kern), SM::BYTES);
    if (attr != cudaSuccess) return attr;
    if (a.tiles <= 0) return cudaSuccess;
    const int sms = device_sms();
    if (sms <= 0) return cudaErrorInvalidDevice;
    const unsigned grid = (unsigned)std::min<int64_t>(a.tiles, (int64_t)sms * SM::CTAS);
    return launch_pdl(true, kern, grid, threads, SM::BYTES, st, (const float2 *)nullptr, (float2 *)nullptr, a);
}

}  // namespace

cudaError_t launch_ragged_outer_c32(int xb, int y0b, const TileArgs &a, cudaStream_t st) {
#define WSFFT_OUTER(x, y)                                                                                   \
    if (xb == x && y0b == y) {                                                                              \
        using G = TileOuter<FUSED_TILE_BITS, x, y>;                                                         \
        return launch_grouped<TileFusedSmem<G, float2>>(tile_outer_kernel<G, float2, true>, 1u << (G::TB - 6), a, st); \
    }
    WSFFT_OUTER(5, 1)
    WSFFT_OUTER(6, 1)
    WSFFT_OUTER(7, 1)
    WSFFT_OUTER(8, 1)
    WSFFT_OUTER(5, 2)
    WSFFT_OUTER(6, 2)
    WSFFT_OUTER(7, 2)
    WSFFT_OUTER(5, 3)
    WSFFT_OUTER(6, 3)
#undef WSFFT_OUTER
    return cudaErrorInvalidValue;
}

cudaError_t launch_ragged_strided_c32(int N, const TileArgs &a, cudaStream_t st) {
#define WSFFT_STRIDED(n, b)                                                                                   \
    if (N == n) {                                                                                             \
        using G = TileStrided<FUSED_TILE_BITS, b>;                                                            \
        return launch_grouped<TileSmem<G, float2, TILE_STRIDED_RAG>>(tile_axis_kernel<G, float2, TILE_STRIDED_RAG>, \
                                                                     1u << (G::TB - 6), a, st);               \
    }
    WSFFT_STRIDED(32, 5)
    WSFFT_STRIDED(64, 6)
    WSFFT_STRIDED(128, 7)
    WSFFT_STRIDED(256, 8)
#undef WSFFT_STRIDED
    return cudaErrorInvalidValue;
}

}  // namespace wsfft
