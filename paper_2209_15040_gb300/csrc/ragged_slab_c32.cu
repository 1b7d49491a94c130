// First trips of a ragged batch in groups (tile_fused.cuh): one launch per
// tile shape over all instances that have it, complex64.
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

cudaError_t launch_ragged_slab_c32(int zb, int yb, const TileArgs &a, cudaStream_t st) {
#define WSFFT_SLAB(z, y)                                                                     \
    if (zb == z && yb == y) {                                                                \
        using G = TileSlab<FUSED_TILE_BITS, z, y>;                                           \
        return launch_grouped<TileFusedSmem<G, float2>>(                                     \
            tile_slab_kernel<G, float2, (z + y < FUSED_TILE_BITS), true>, 1u << (G::TB - 6), a, st); \
    }
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

}  // namespace wsfft
