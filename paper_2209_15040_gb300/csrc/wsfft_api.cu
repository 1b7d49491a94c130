// C ABI of the library (include/wsfft.h): plan construction, twiddle tables,
// pass schedule and launch sequencing.
//
// Schedule (Section 1: one superstep per axis, in any order; Section 4.2:
// the 3D sequence z, then the other axes):
//   rank 2/3: superstep along the contiguous axis (in -> out), then one
//             superstep per remaining axis, last axis first (out -> out,
//             each kernel reading and writing the same tile).  Where the
//             inner axes fit (fused_tile_rule) device executes fuse them:
//             two axes per trip (Plan::fused).
//   rank 1, n <= 4096: one contiguous superstep.
//   rank 1, n > 4096: the long axis is split as a 2D problem n = n1*n2
//             (Section 8 proposes decomposing large 1D transforms as a
//             higher-dimensional FFT): a strided superstep of length n2 with
//             the inter-step twiddles w_n^(j1*k2) applied on store (in ->
//             workspace), then a contiguous superstep of length n1 whose
//             store transposes into natural order (workspace -> out).
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <complex>
#include <cstdlib>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "../../include/wsfft.h"
#include "fft_core.cuh"
#include "host_roots.h"
#include "pass_desc.h"
#include "pass_kernels.cuh"
#include "engine.cuh"
#include "engine_desc.h"
#include "plan_internal.h"
#include "ragged.cuh"
#include "ragged_desc.h"
#include "slab_cluster.cuh"
#include "slab_desc.h"
#include "tile_desc.h"

namespace wsfft {

namespace {

// cos and sin of (pi/4) at/n, 0 <= at <= n
OctantRoot octant_root(int64_t at, int64_t n) {
    const long double phi = 0.78539816339744830961566084581987572L * (long double)at / (long double)n;
    const long double c = cosl(phi), s = sinl(phi);
    return OctantRoot{(float)c, (float)s, (double)c, (double)s};
}

// cos and -sin of an angle in octant o, from those of its distance to the
// octant's axis (odd octants are measured from their upper end)
template <class T>
std::pair<T, T> unfold(int o, T c, T s) {
    switch (o) {
        case 0: return {c, -s};
        case 1: return {s, -c};
        case 2: return {-s, -c};
        case 3: return {-c, -s};
        case 4: return {-c, s};
        case 5: return {-s, c};
        case 6: return {s, c};
        default: return {c, s};
    }
}

// the octant of 2*pi*m/n and the root of the distance to its axis
OctantRoot fold(int64_t m, int64_t n, RootMemo *memo, int &octant) {
    const int log_n = __builtin_ctzll((unsigned long long)n);
    m &= n - 1;
    octant = (int)((8 * m) >> log_n);
    const int64_t rho = (8 * m) & (n - 1);  // position inside the octant, [0, n)
    const int64_t at = (octant & 1) == 0 ? rho : n - rho;
    if (!memo) return octant_root(at, n);
    // at/n is the same float for every n: the factors between them are powers of two
    if (log_n <= RootMemo::LOG_ORDER) {
        const int64_t i = (at << (RootMemo::LOG_ORDER - log_n)) >> 3;
        if (!memo->known[i]) {
            memo->near[i] = octant_root(at, n);
            memo->known[i] = true;
        }
        return memo->near[i];
    }
    const auto found = memo->far.try_emplace(at << (32 - log_n));
    if (found.second) found.first->second = octant_root(at, n);
    return found.first->second;
}

}  // namespace

float2 host_root(int64_t m, int64_t n, RootMemo *memo) {
    auto root = [&]() {
        int o;
        const OctantRoot r = fold(m, n, memo, o);
        const auto cs = unfold(o, r.cf, r.sf);
        return make_float2(cs.first, cs.second);
    };
    if (!memo || n > (1 << RootMemo::LOG_ORDER)) return root();
    const int shift = RootMemo::LOG_ORDER - __builtin_ctzll((unsigned long long)n);
    const size_t i = ((uint64_t)m << shift) & ((1u << RootMemo::LOG_ORDER) - 1);
    if (!memo->on_circle[i]) {
        memo->circle[i] = root();
        memo->on_circle[i] = true;
    }
    return memo->circle[i];
}

std::complex<double> host_root_d(int64_t m, int64_t n, RootMemo *memo) {
    int o;
    const OctantRoot r = fold(m, n, memo, o);
    const auto cs = unfold(o, r.cd, r.sd);
    return {cs.first, cs.second};
}

int fill_stage_table(float2 *dst, int cap, int N, int E, RootMemo *memo) {
    const int size = sched_tw_size(N, E);
    if (size + 1 > cap) return -1;
    const int ns = sched_nstages(N, E);
    for (int s = 1; s < ns; ++s) {
        const int R = sched_radix(N, E, s), Ns = sched_ns_before(N, E, s);
        const int off = sched_tw_offset(N, E, s);
        for (int r = 1; r < R; ++r)
            for (int k = 0; k < Ns; ++k) dst[off + (r - 1) * Ns + k] = host_root((int64_t)r * k, (int64_t)Ns * R, memo);
    }
    dst[size] = make_float2(0.f, 0.f);
    return size + 1;
}

}  // namespace wsfft

using namespace wsfft;

namespace {

bool is_pow2(int64_t n) { return n > 0 && (n & (n - 1)) == 0; }

int ilog2(int64_t n) {
    int l = 0;
    while (((int64_t)1 << l) < n) ++l;
    return l;
}

int64_t elem_bytes(int dtype) { return dtype == WSFFT_C32 ? 8 : 4; }

std::vector<float2> stage_table(int N, int E, RootMemo *memo) {
    std::vector<float2> t((size_t)sched_tw_size(N, E) + 1);
    fill_stage_table(t.data(), (int)t.size(), N, E, memo);
    return t;
}

// Table of the tensor-core contiguous superstep at N = 512 (layout in
// tc_contig.cuh): the DFT-16 matrix B[n = 2*k1 + part][k = n1] = (Re, Im)
// w16^(n1*k1) as 16-bit high parts and 16-bit remainders in the K-major
// core-matrix byte order, then the inter-stage twiddles w512^(k1*n2).
std::vector<float2> tc_table_host(int dtype) {
    std::vector<float2> t(TC_TABLE_FLOAT2);
    uint16_t *hi = reinterpret_cast<uint16_t *>(t.data());
    uint16_t *lo = hi + 512;
    for (int n = 0; n < 32; ++n)
        for (int k = 0; k < 16; ++k) {
            const int k1 = n / 2, part = n % 2, n1 = k;
            const float2 w = host_root((int64_t)n1 * k1, 16);
            const float v = part ? w.y : w.x;
            uint16_t h, l;
            if (dtype == WSFFT_C16BF) {
                const __nv_bfloat16 hb = __float2bfloat16_rn(v);
                h = __bfloat16_as_ushort(hb);
                l = __bfloat16_as_ushort(__float2bfloat16_rn(v - __bfloat162float(hb)));
            } else {
                const __half hh = __float2half_rn(v);
                h = __half_as_ushort(hh);
                l = __half_as_ushort(__float2half_rn(v - __half2float(hh)));
            }
            const int off = (n / 8) * 256 + (k / 8) * 128 + (n % 8) * 16 + (k % 8) * 2;  // bytes
            hi[off / 2] = h;
            lo[off / 2] = l;
        }
    for (int n2 = 0; n2 < 32; ++n2)
        for (int k1 = 0; k1 < 16; ++k1) t[TC_TABLE_TW + n2 * 16 + k1] = host_root((int64_t)k1 * n2, 512);
    return t;
}

float axis_scale(int64_t n, int dir, int norm) {
    if (norm == WSFFT_NORM_PAPER) return dir == WSFFT_INVERSE ? (float)(1.0 / (double)n) : 1.f;
    if (norm == WSFFT_NORM_ORTHO) return (float)(1.0 / std::sqrt((double)n));
    if (norm == WSFFT_NORM_FORWARD) return dir == WSFFT_FORWARD ? (float)(1.0 / (double)n) : 1.f;
    return 1.f;
}

cudaError_t launch_engine(int dtype, int n, const EngArgs &a, int grid, cudaStream_t st) {
    switch (dtype) {
        case WSFFT_C32: return launch_engine_c32(n, a, grid, st);
        case WSFFT_C16F: return launch_engine_c16f(n, a, grid, st);
        default: return launch_engine_c16bf(n, a, grid, st);
    }
}

cudaError_t launch_persist(int dtype, int n, const EngArgs &a, int s_mode, int *per_sm, int grid,
                           cudaStream_t st) {
    switch (dtype) {
        case WSFFT_C32: return launch_persist_c32(n, a, s_mode, per_sm, grid, st);
        case WSFFT_C16F: return launch_persist_c16f(n, a, s_mode, per_sm, grid, st);
        default: return launch_persist_c16bf(n, a, s_mode, per_sm, grid, st);
    }
}

cudaError_t launch_wpp(int dtype, int n, const EngArgs &a, int *per_sm, int grid, cudaStream_t st) {
    switch (dtype) {
        case WSFFT_C32: return launch_wpp_c32(n, a, per_sm, grid, st);
        case WSFFT_C16F: return launch_wpp_c16f(n, a, per_sm, grid, st);
        default: return launch_wpp_c16bf(n, a, per_sm, grid, st);
    }
}

cudaError_t launch_wps(int dtype, int n, const WpStridedArgs &b, cudaStream_t st) {
    switch (dtype) {
        case WSFFT_C32: return launch_wps_c32(n, b, st);
        case WSFFT_C16F: return launch_wps_c16f(n, b, st);
        default: return launch_wps_c16bf(n, b, st);
    }
}

cudaError_t launch_slab(int dtype, int n, const void *in, void *out, int64_t nslabs, const SlabArgs &a, bool pdl,
                        cudaStream_t st, int *max_clusters) {
    switch (dtype) {
        case WSFFT_C32: return launch_slab_c32(n, in, out, nslabs, a, pdl, st, max_clusters);
        case WSFFT_C16F: return launch_slab_c16f(n, in, out, nslabs, a, pdl, st, max_clusters);
        default: return launch_slab_c16bf(n, in, out, nslabs, a, pdl, st, max_clusters);
    }
}

cudaError_t launch_tile(int dtype, int mode, int N, int tb, const void *in, void *out, const TileArgs &a,
                        cudaStream_t st) {
    switch (dtype) {
        case WSFFT_C32: return launch_tile_c32(mode, N, tb, in, out, a, st);
        case WSFFT_C16F: return launch_tile_c16f(mode, N, tb, in, out, a, st);
        default: return launch_tile_c16bf(mode, N, tb, in, out, a, st);
    }
}

cudaError_t launch_fused(int dtype, const PassSpec &p, const void *in, void *out, const TileArgs &a,
                         cudaStream_t st) {
    using Fn = cudaError_t (*)(int, int, const void *, void *, const TileArgs &, cudaStream_t);
    static constexpr Fn slab[3] = {launch_tile_slab_c32, launch_tile_slab_c16f, launch_tile_slab_c16bf};
    static constexpr Fn outer[3] = {launch_tile_outer_c32, launch_tile_outer_c16f, launch_tile_outer_c16bf};
    static constexpr Fn wide[3] = {launch_tile_wide_c32, launch_tile_wide_c16f, launch_tile_wide_c16bf};
    if (p.kind == PASS_TILE_OUTER) return outer[dtype](p.xb, p.y0b, in, out, a, st);
    return (p.kind == PASS_TILE_SLAB ? slab : wide)[dtype](p.zb, p.yb, in, out, a, st);
}

cudaError_t launch(int dtype, const PassSpec &p, const void *in, void *out, const TileArgs &a,
                   cudaStream_t st) {
    if (p.kind == PASS_TILE_SLAB || p.kind == PASS_TILE_OUTER || p.kind == PASS_TILE_WIDE)
        return launch_fused(dtype, p, in, out, a, st);
    if (p.tile >= PIPE_TILE) {
        // the kernels' stage tables are those of one radix per axis length
        if (p.E != tile_table_E(p.N)) return cudaErrorInvalidValue;
        if (p.kind == PASS_CONTIG && !p.variant) {
            if (p.tile != PIPE_TILE + FUSED_TILE_BITS) return cudaErrorInvalidValue;
            switch (dtype) {
                case WSFFT_C32: return launch_tile_contig_c32(p.N, in, out, a, st);
                case WSFFT_C16F: return launch_tile_contig_c16f(p.N, in, out, a, st);
                default: return launch_tile_contig_c16bf(p.N, in, out, a, st);
            }
        }
        const int mode = p.kind != PASS_STRIDED ? TILE_TRANS : p.variant ? TILE_STRIDED_TWID : TILE_STRIDED;
        return launch_tile(dtype, mode, p.N, p.tile - PIPE_TILE, in, out, a, st);
    }
    switch (dtype) {
        case WSFFT_C32: return launch_pass_c32(p.kind, p.N, p.E, p.tile, p.variant, in, out, a, st);
        case WSFFT_C16F: return launch_pass_c16f(p.kind, p.N, p.E, p.tile, p.variant, in, out, a, st);
        default: return launch_pass_c16bf(p.kind, p.N, p.E, p.tile, p.variant, in, out, a, st);
    }
}

int cuda_status(cudaError_t e) { return e == cudaSuccess ? WSFFT_SUCCESS : WSFFT_ERR_CUDA; }

// a pass-shape override the schedule builder may apply: a power-of-two count
// of values per thread within the pencil (the builder makes twiddle tables for
// it) and a non-negative tile code; whether a kernel of that shape exists is
// checked separately (Plan::overrides_launchable)
bool override_usable(int E, int tile, int N) {
    return E >= 1 && E <= 32 && E <= N && (E & (E - 1)) == 0 && tile >= 0;
}

// log2 of the elements per tile with which a strided superstep of length N at
// element stride `inner`, over `total` elements, runs on the pipelined tile
// kernels; 0: the one-tile-per-block kernels are faster, or the pencils do
// not fill whole tiles.  Measured per superstep, against those kernels:
//   2048 points, three stages, 64-byte rows (complex64): 508-587 us against
//     566-603, 16-bit 383-431 against 466-481.
//   4096 points: only in 16-bit storage, from 2^25 elements up and at strides of
//     32 to 1024 elements (in place 582-592 us against 595-611, out of place 600-627
//     against 608-639; 2^25 152-155 against 153-156).  Smaller arrays, and strides
//     of 4 to 16 elements, whose general kernels read whole runs, were slower
//     on the tiles (2^23 at a stride of 8: 40.8 us against 33.0, of 256: 42.4 against
//     40.4; 2^26 at 8: 267 against 237), wide strides no faster (2^26 at 2^14: 337 against
//     330); complex64 732 against 696.
//   complex64, 1024 points (shorter axes are at the copy rate without them):
//     tiles of 2^13 elements up to a stride of 2^16 elements from 2^22
//     elements up (2^22 12.4 us against 14.4, 2^24 48-50 against 53-57, 2^25
//     89-92 against 99-108; at a stride of 8, where the general kernel reads whole
//     runs, 2^22 11.1 against 12.4 but 2^25 93.7 against 82.9); for large arrays or
//     wider strides their 64-byte rows cost too much (2^27: 349-372 us, and 540 at a stride of 2^17) and
//     tiles of 2^14 (128-byte rows) take over (2^27 351-388 us against 373-467).
//   16-bit storage: from 2^22 elements up (2^27 170-174 us against 224-273
//     at 32..128 points, 185-206 against 235-251 at 256, 200-212 against
//     255-271 at 512, 234-237 against 330-338 at 1024; within 0.5 us of each
//     other below).  Tiles of 2^13 elements (three blocks per SM) are the
//     faster ones until their rows (64 bytes at 512 points, 128 at 256, 256 at
//     128) lie 2^19 to 2^22 bytes apart: 512 points 206 us at a stride of
//     2^16 elements and 282 at 2^18, where tiles of 2^14 take 210 and 212.
int pipe_tile_bits(int dtype, int64_t N, int64_t inner, int64_t total) {
    int tb = 0;
    if (N == 2048) tb = total >= ((int64_t)1 << 22) ? 14 : 0;
    if (N == 4096 && dtype != WSFFT_C32)
        tb = total >= ((int64_t)1 << 25) && inner >= 32 && inner <= 1024 ? 14 : 0;
    if (dtype == WSFFT_C32) {
        if (N == 1024 && inner <= ((int64_t)1 << 16) && total < ((int64_t)1 << 27))
            tb = total >= ((int64_t)1 << 22) && (inner >= 16 || total < ((int64_t)1 << 25)) ? 13 : 0;
        else if (N == 1024 && total >= ((int64_t)1 << 25))
            tb = 14;
    } else if (total >= ((int64_t)1 << 22)) {
        if (N == 32 || N == 64 || N == 128) tb = inner <= ((int64_t)1 << 18) ? 13 : 0;
        if (N == 256 || N == 512) tb = inner < ((int64_t)1 << 17) ? 13 : 14;
        if (N == 1024) tb = 14;
    }
    return tb && inner % (((int64_t)1 << tb) / N) == 0 ? tb : 0;
}

// Whether a contiguous superstep of N points runs on the tile kernels.
// Measured against the general ones: 32 points 2^21 elements 6.5 us against 7.4
// (complex64) and 6.1 against 6.8 (FP16), 2^24 44.5 against 49.7 and 29.1 against
// 45.1; 16-bit storage at 64 and 128 points 2^22 8.6 against 8.8 and 10.6, 2^27
// 192-194 against 234-263.  Other lengths are faster there: 256 points FP16 185
// against 200, complex64 300-315 against 352-371.
bool pipe_contig(int dtype, int64_t N, int64_t total) {
    if (N == 32) return total >= ((int64_t)1 << 21);
    return dtype != WSFFT_C32 && (N == 64 || N == 128) && total >= ((int64_t)1 << 22);
}

// pipe_tile_bits for the four-step's first superstep (twid: inter-step twiddle on a
// strided store of `rows` pencils per transform) and for a contiguous
// superstep with the transposed store.  Measured per 2^27 elements, against
// the general kernels (whose first superstep takes two table reads and a
// product per element):
//   twiddle: complex64 256 points 338 us against 358, 512 364-373 against
//     402, 1024 344 against 410-530; 16-bit 64..256 points 210-225 against
//     303-330, 512 246 against 552, 1024 282 against 510 (tiles of 2^14: 327 us
//     with 32-byte rows).
//   transposed: complex64 1024 points 389 us against 452-505, shorter axes
//     equal; 16-bit 64..256 points 189-196 against 240-307, 512 214 against
//     305, 1024 225 against 389.
// From 2^22 elements (16-bit) or 2^23 (complex64) up; below, both take as long.
int pipe_tile_bits_variant(int dtype, int64_t N, int64_t rows, int64_t total, bool twid) {
    int tb = 0;
    const bool half = dtype != WSFFT_C32;
    if (twid) {
        if (N >= (half ? 64 : 256) && N <= 1024) tb = half && N == 1024 ? 14 : 13;
    } else {
        if (N == 1024 || (half && N >= 64 && N <= 512)) tb = half ? 13 : 14;
    }
    if (total < (int64_t)1 << (half ? 22 : 23)) tb = 0;
    return tb && rows % (((int64_t)1 << tb) / N) == 0 ? tb : 0;
}

// Whether a rank-2 or rank-3 transform (axes d) runs its inner axes fused on
// the tile kernels (tile_fused.cuh).  A fused trip replaces two (the inner
// axes of slabs of up to 2^13 elements) or turns three trips into two, and wins
// from 2^17 elements up (below, see build_fused: a tile keeps one block busy for
// longer than separate launches take) to 1 GiB (2^27 elements, complex64 / FP16
// storage, us):
//   64 x 64 batches 329 / 262 against 597 / 464, 32^3 623 / 410 against 962 /
//   771, 64^3 631 / 431 against 896 / 708; split middle axis: 128^3 684 / 458
//   against 919 / 734 (one cube 15.3 against 18.9), 64 x 256^2 687 / 474
//   against 907 / 686 (one of 2^22 elements 26.8 against 27.0).
// Beyond 2^22 elements per transform the outer pass would need tiles of 2^14
// elements or rows under 128 bytes (16 elements), both slower than a third trip.
struct FusedShape {
    bool use = false, outer = false;
    int zb = 0, yb = 0, y0b = 0;
};
FusedShape fused_tile_rule(const std::vector<int64_t> &d) {
    FusedShape f;
    const int r = (int)d.size();
    if (r < 2) return f;
    const int64_t n1 = d[r - 2], n2 = d[r - 1];
    if (n2 < 32 || n2 > 256 || n1 < 32) return f;
    f.zb = ilog2(n2);
    const int slab = f.zb + ilog2(n1);
    if (slab <= FUSED_TILE_BITS) {
        f.yb = ilog2(n1);
        f.use = true;
    } else if (r == 3) {
        f.yb = FUSED_TILE_BITS - f.zb;
        f.y0b = slab - FUSED_TILE_BITS;
        const int xb = ilog2(d[0]);
        // rows of at least 16 elements, within one row of the last axis (one k1)
        f.use = f.outer = xb >= 5 && f.y0b <= 4 && xb + f.y0b <= 9 && xb + f.y0b + f.zb >= FUSED_TILE_BITS;
    }
    return f;
}

// Whether a rank-2 or rank-3 transform out of place runs a digit of a long
// strided axis in the trip of its last axis (tile_wide_kernel): axis (-1: none)
// and the digit's bits.  Strided supersteps of 2048 and 4096 points have
// rows of 32-64 bytes and one block per SM (0.55 and 0.45 of the copy rate in
// complex64, 0.35 and 0.26 in 16-bit storage), those of 1024 points rows that lie
// megabytes apart; what is left of the axis after the digit is a superstep at
// the copy rate, for a last-axis trip of 0.36-0.37 ms per 2^27 elements
// (complex64) instead of 0.30-0.35.  Measured (complex64 / FP16, us): 4096^2
// 123 / 85 against 141 / 117 (8 of them 843 / 609 against 1064 / 899), 32 x
// 2048^2 684 / 495 against 889 / 741, 64 x 2048 x 1024 677 / 470 against 870 /
// 827, 1024^3 8100 / 5982 against 8766 / 7126, 1024 x 512^2 1997 against 2107;
// 1024 x 128 x 1024, whose outer stride is 2^17, 996 / 701 against 986 / 649.
// Below 2^20 elements (2^21 in 16-bit storage, and 2^21 itself for 2048 points
// beside 512) the three-stage tile's latency costs more (FP16 2048 x 512: one 14.3
// against 13.2, two 15.2 against 13.6, three 17.0 against 21.7; 4096 x 512 15.6 against
// 16.4, 2048 x 1024 15.2 against 16.8).
struct WideShape {
    int axis = -1, rb = 0;
};
WideShape wide_tile_rule(int dtype, const std::vector<int64_t> &d, int64_t total) {
    WideShape w;
    const int r = (int)d.size();
    if (r < 2 || total < ((int64_t)1 << (dtype == WSFFT_C32 ? 20 : 21))) return w;
    const int zb = ilog2(d[r - 1]);
    if (zb < 9 || zb > 12) return w;
    // the longest of the axes that qualify; the outer one where both are as long
    for (int ax = r - 2; ax >= 0; --ax) {
        const bool far = r == 3 && ax == 0 && d[0] == 1024 && d[1] * d[2] >= ((int64_t)1 << 18);
        if (dtype != WSFFT_C32 && zb == 9 && d[ax] == 2048 && total <= ((int64_t)1 << 21)) continue;
        if ((d[ax] >= 2048 || far) && (w.axis < 0 || d[ax] >= d[w.axis])) w.axis = ax;
    }
    if (w.axis < 0) return w;
    // tiles of 2^13 elements; of 2^14 only where a radix of 2 would leave 2048 points
    w.rb = zb == 12 && d[w.axis] == 4096 ? 2 : 13 - zb;
    return w;
}

// two buffers of `bytes` that share some bytes without being the same buffer
bool partial_overlap(const void *a, const void *b, size_t bytes) {
    const char *x = static_cast<const char *>(a), *y = static_cast<const char *>(b);
    return x != y && x < y + bytes && y < x + bytes;
}

}  // namespace

namespace wsfft {

// Device address of a copy of h, which flush_tables() makes: a plan's tables
// lie in blocks of at least 128 KB that are allocated and filled in one piece
// (an allocation and a synchronised copy for each table took 25 us, more
// than its roots).  Null when the memory is not there.
float2 *Plan::place_table(const std::vector<float2> &h) {
    const size_t bytes = (h.size() * sizeof(float2) + 255) & ~(size_t)255;
    if (table_blocks.empty() || table_blocks.back().used + bytes > table_blocks.back().size) {
        TableBlock b;
        b.size = std::max(bytes, (size_t)128 * 1024);
        if (cudaMalloc(&b.device, b.size) != cudaSuccess) return nullptr;
        table_blocks.push_back(std::move(b));
    }
    TableBlock &b = table_blocks.back();
    float2 *d = reinterpret_cast<float2 *>(b.device + b.used);
    const char *src = reinterpret_cast<const char *>(h.data());
    b.pending.insert(b.pending.end(), src, src + h.size() * sizeof(float2));
    b.pending.resize(b.pending.size() + bytes - h.size() * sizeof(float2));
    b.used += bytes;
    return d;
}
template <class Map, class Key>
const float2 *Plan::remember(Map &map, const Key &key, const std::vector<float2> &h) {
    float2 *d = place_table(h);
    if (d) map[key] = d;
    return d;
}
// The angles met since the last flush_tables() (null without memory: they are evaluated anew).
RootMemo *Plan::memo() {
    if (!roots) roots.reset(new (std::nothrow) RootMemo());
    return roots.get();
}
// Copy the tables placed since the last call to the device.
int Plan::flush_tables() {
    roots.reset();
    for (auto &b : table_blocks) {
        if (b.pending.empty()) continue;
        const int rc = upload(b.device + b.used - b.pending.size(), b.pending.data(), b.pending.size());
        if (rc != WSFFT_SUCCESS) return rc;
        b.pending.clear();
        b.pending.shrink_to_fit();
    }
    return WSFFT_SUCCESS;
}

const float2 *Plan::tc_table(int N) {
    if (N != 512 || dtype == WSFFT_C32) return nullptr;
    auto key = std::make_pair(N, TC_TILE);
    auto it = tables.find(key);
    if (it != tables.end()) return it->second;
    return remember(tables, key, tc_table_host(dtype));
}

// Four-step inter-superstep twiddles w_L^m, m < L, as two tables: the high
// part w_L^(i << shift) for i < L >> shift, then the low part w_L^j for
// j < 2^shift (w_L^m is their product; both from host_root).
const float2 *Plan::fourstep_table(int64_t L, int shift) {
    auto it = fs_tables.find(L);
    if (it != fs_tables.end()) return it->second;
    const int64_t nh = L >> shift, nl = (int64_t)1 << shift;
    std::vector<float2> h((size_t)(nh + nl));
    for (int64_t i = 0; i < nh; ++i) h[(size_t)i] = host_root(i << shift, L, memo());
    for (int64_t j = 0; j < nl; ++j) h[(size_t)(nh + j)] = host_root(j, L, memo());
    return remember(fs_tables, L, h);
}

// The same twiddles for the pipelined tile kernels' first superstep (length
// N, stage radices Ns and N/Ns, q < n1 = L/N pencils): w_L^(q k1) for
// k1 < Ns, then w_(L/Ns)^(q r) for r < N/Ns, rows of n1 values, neighbouring
// pencils as (re0, re1, im0, im1).  The roots are FP64 products of the two
// tables' long-double roots (a long-double root for each of the 2^16 entries
// at L = 2^20 would take the host a second), rounded once.
const float2 *Plan::fourstep_tile_table(int64_t L, int N) {
    const auto key = std::make_pair(L, N);
    auto it = fs_tile_tables.find(key);
    if (it != fs_tile_tables.end()) return it->second;
    const int64_t n1 = L / N;
    const int Ns = tile_table_E(N), shift = (ilog2(L) + 1) / 2;
    const int64_t low = (int64_t)1 << shift;
    std::vector<std::complex<double>> hi((size_t)(L >> shift)), lo((size_t)low);
    for (size_t i = 0; i < hi.size(); ++i) hi[i] = host_root_d((int64_t)i << shift, L, memo());
    for (size_t i = 0; i < lo.size(); ++i) lo[i] = host_root_d((int64_t)i, L, memo());
    std::vector<float2> h;
    h.reserve((size_t)(n1 * (Ns + N / Ns)));
    auto rows = [&](int count, int64_t step) {  // w_L^(step q j), j < count
        for (int j = 0; j < count; ++j)
            for (int64_t q = 0; q < n1; q += 2) {
                std::complex<double> w[2];
                for (int i = 0; i < 2; ++i) {
                    const int64_t m = (step * (q + i) * j) & (L - 1);
                    w[i] = hi[(size_t)(m >> shift)] * lo[(size_t)(m & (low - 1))];
                }
                h.push_back(make_float2((float)w[0].real(), (float)w[1].real()));
                h.push_back(make_float2((float)w[0].imag(), (float)w[1].imag()));
            }
    };
    rows(Ns, 1);
    rows(N / Ns, Ns);
    return remember(fs_tile_tables, key, h);
}

const float2 *Plan::table(int N, int E) {
    if (lender) return lender->table(N, E);
    auto key = std::make_pair(N, E);
    auto it = tables.find(key);
    if (it != tables.end()) return it->second;
    return remember(tables, key, stage_table(N, E, N > E ? memo() : nullptr));
}

// Twiddles of a two-stage pencil, radix R0 then N/R0: w_N^(r k) at
// (r-1)*R0 + k, r < N/R0, k < R0.
const float2 *Plan::table2(int N, int R0) {
    if (lender) return lender->table2(N, R0);
    const auto key = std::make_pair(N, 1000 + R0);
    auto it = tables.find(key);
    if (it != tables.end()) return it->second;
    std::vector<float2> h;
    h.reserve((size_t)N);
    for (int r = 1; r < N / R0; ++r)
        for (int k = 0; k < R0; ++k) h.push_back(host_root((int64_t)r * k, N, memo()));
    h.push_back(make_float2(0.f, 0.f));
    return remember(tables, key, h);
}

// Twiddles between the two parts of a split axis of n points: w_n^(y k) at
// (y-1)*(n/classes) + k for the residue classes y.
const float2 *Plan::class_table(int n, int classes) {
    if (lender) return lender->class_table(n, classes);
    const auto key = std::make_pair(n, 2000 + classes);
    auto it = tables.find(key);
    if (it != tables.end()) return it->second;
    std::vector<float2> h;
    h.reserve((size_t)n);
    for (int y = 1; y < classes; ++y)
        for (int k = 0; k < n / classes; ++k) h.push_back(host_root((int64_t)y * k, n, memo()));
    h.push_back(make_float2(0.f, 0.f));
    return remember(tables, key, h);
}

// Stage twiddles of the 2^zb points of a wide tile (TileWide): radices
// 2^(5-rb), 32 and the rest.
const float2 *Plan::wide_table(int zb, int rb) {
    if (lender) return lender->wide_table(zb, rb);
    const auto key = std::make_pair(1 << zb, 3000 + rb);
    auto it = tables.find(key);
    if (it != tables.end()) return it->second;
    std::vector<float2> h;
    h.reserve((size_t)2 << zb);
    int64_t ns = (int64_t)1 << (5 - rb);
    for (int R : {32, (1 << zb) / (32 << (5 - rb))}) {
        for (int r = 1; r < R; ++r)
            for (int64_t k = 0; k < ns; ++k) h.push_back(host_root(r * k, ns * R, memo()));
        ns *= R;
    }
    return remember(tables, key, h);
}

// Schedule with one digit of a long strided axis in the trip of the last
// axis: see wide_tile_rule.  `strided` builds the superstep of an axis of n
// points at element stride `inner`.
int Plan::build_wide(const std::vector<int64_t> &d, bool inv, const StridedBuilder &strided) {
    const int r = (int)d.size();
    const WideShape w = wide_tile_rule(dtype, d, elems * batch);
    if (w.axis < 0) return WSFFT_SUCCESS;
    std::vector<int64_t> inner((size_t)r, 1);
    for (int ax = r - 2; ax >= 0; --ax) inner[ax] = inner[ax + 1] * d[ax + 1];
    const int64_t n = d[w.axis], R = (int64_t)1 << w.rb;
    PassSpec a{};
    a.kind = PASS_TILE_WIDE;
    a.N = (int)d[r - 1];
    a.zb = ilog2(d[r - 1]);
    a.yb = w.rb;
    a.y0b = ilog2(n / R);
    a.inner = inner[w.axis];
    a.transform_elems = elems;
    a.src = SRC_IN;
    a.dst = DST_OUT;
    a.conj_in = inv;
    a.scale = axis_scale(d[r - 1] * R, dir, norm);
    a.tw = wide_table(a.zb, a.yb);
    a.tw2 = class_table((int)n, (int)R);
    if (!a.tw || !a.tw2) return WSFFT_ERR_ALLOC;
    fused.push_back(a);
    for (int ax = r - 2; ax >= 0; --ax) {
        const bool split = ax == w.axis;
        PassSpec p = strided(split ? n / R : d[ax], split ? R * inner[ax] : inner[ax]);
        p.reverse = ax == r - 2;
        p.tw = table(p.N, p.E);
        if (!p.tw) return WSFFT_ERR_ALLOC;
        fused.push_back(p);
    }
    fused.back().conj_out = inv;
    defer_scale(fused);
    return WSFFT_SUCCESS;
}

// complex64 has the range to defer every superstep's scale to the last store
// (one scaled store instead of one per pass); the reduced-precision types and
// the orthonormal scaling keep the per-superstep scale.
void Plan::defer_scale(std::vector<PassSpec> &list) const {
    if (dtype != WSFFT_C32 || norm == WSFFT_NORM_ORTHO) return;
    double total_scale = 1.0;
    for (auto &p : list) {
        total_scale *= p.scale;
        p.scale = 1.f;
    }
    list.back().scale = (float)total_scale;
}

// Fused schedule of the plan (d: its axes longer than one), beside the one
// launch per superstep in `passes`: see fused_tile_rule.
int Plan::build_fused(const std::vector<int64_t> &d, bool inv) {
    const FusedShape f = fused_tile_rule(d);
    if (!f.use) return WSFFT_SUCCESS;
    // Below 2^17 elements a block's time for 2^13 elements (about 4 us) is more than
    // two launches over many small blocks take: one 64 x 64 plane 5.5 us against
    // 3.1, 32 x 32 x 64 6.3 against 5.1.  At 2^17 itself the same holds in complex64
    // and for rank 3 (back to back and captured: 32 x 64 x 64 7.1 and 7.2 against 5.7 and
    // 5.1, thirty-two 64 x 64 planes 5.1 and 5.4 against 4.0 and 3.6; in 16-bit storage slabs
    // of 2^13 elements take 4.3 us either way).  Above: 64^3 7.6 against 8.0, eight 32^3
    // 7.0 against 9.6; up to 2^18 elements a launch less for the host, at up to 1.2 us more
    // on the GPU (twenty-four 128 x 64 planes 5.3 against 4.4).  The smaller tiles of 32 x 32 slabs make up for it from 2^15 to 2^17
    // elements in complex64: 32 planes 3.7 against 4.0, 32^3 5.5 against 5.8.
    const int r = (int)d.size();
    const int64_t total = elems * batch;
    const bool small = total < FUSED_SMALL_ELEMS || (total == FUSED_SMALL_ELEMS && (dtype == WSFFT_C32 || r == 3));
    if (small && !(dtype == WSFFT_C32 && f.zb + f.yb == 10 && total >= FUSED_SMALL_ELEMS / 4)) return WSFFT_SUCCESS;
    const int64_t n1 = d[r - 2], n2 = d[r - 1], n0 = r == 3 ? d[0] : 1;
    const int64_t rows = (int64_t)1 << f.yb;
    PassSpec a{};
    a.kind = PASS_TILE_SLAB;
    a.N = (int)n2;
    a.zb = f.zb;
    a.yb = f.yb;
    a.y0b = f.y0b;
    a.inner = n2;
    a.transform_elems = elems;
    a.src = SRC_IN;
    a.dst = DST_OUT;
    a.conj_in = inv;
    a.scale = axis_scale(n2 * rows, dir, norm);
    a.tw = table((int)n2, 16);
    a.tw2 = table((int)rows, 32);
    if (!a.tw || !a.tw2) return WSFFT_ERR_ALLOC;
    fused.push_back(a);
    if (f.outer) {
        PassSpec b{};
        b.kind = PASS_TILE_OUTER;
        b.N = (int)n0;
        b.zb = f.zb;
        b.yb = f.yb;
        b.xb = ilog2(n0);
        b.y0b = f.y0b;
        b.inner = n1 * n2;
        b.transform_elems = elems;
        b.src = SRC_OUT;
        b.dst = DST_OUT;
        b.scale = axis_scale(n0 << f.y0b, dir, norm);
        b.reverse = true;  // the slab pass wrote the last transforms last
        b.tw = table2((int)n0, 32 >> f.y0b);
        b.tw2 = class_table((int)n1, 1 << f.y0b);
        if (!b.tw || !b.tw2) return WSFFT_ERR_ALLOC;
        fused.push_back(b);
    } else if (r == 3) {
        PassSpec b = passes.back();  // x as in the one-launch schedule
        b.scale = axis_scale(n0, dir, norm);
        b.reverse = true;
        fused.push_back(b);
    }
    fused.back().conj_out = inv;
    fused_in_place = f.y0b == 0;
    defer_scale(fused);
    return WSFFT_SUCCESS;
}

// Two-launch schedule of an n^3 cube on the persistent engine.
// Pass A: per slab (fixed first index), the contiguous superstep (z) then the
// strided superstep along the middle axis (y), queued `lag` slabs apart so
// the slab is still in L2 when it is read again.  Pass B: the superstep along
// the first axis (x).
int Plan::build_engine(int64_t n0, int64_t n, bool inv) {
    int grid = eng_grid;
    if (engine_mode == 1 || engine_mode == 3) {
        int per_sm = 0;
        EngArgs dummy{};
        cudaError_t e = engine_mode == 1 ? launch_persist(dtype, (int)n, dummy, 0, &per_sm, 0, 0)
                                         : launch_wpp(dtype, (int)n, dummy, &per_sm, 0, 0);
        if (e != cudaSuccess || per_sm < 1) return WSFFT_ERR_UNSUPPORTED;
        persist_grid = per_sm * sm_count;
        grid = persist_grid;
    }
    // pencils per contiguous tile (tp) and per strided tile (tq)
    int64_t tp, tq;
    if (engine_mode == 3) {
        tp = wp_tile_z((int)n);
        tq = wp_tile_y((int)n);
    } else if (engine_mode == 1 && n == 512) {
        tp = persist512_tile_z();  // contiguous tiles: one warp per pencil
        tq = 16;                   // strided tiles: 16 pencils
    } else {
        tp = engine_tile_pencils((int)n);
        tq = tp;
    }
    const int64_t sub = engine_mode == 1 ? persist_sub((int)n) : 1;  // tiles per queue item
    const int64_t zper = n / tp / sub, yper = n / tq / sub;  // queue items per slab of each kind
    const int64_t U = batch * n0;                     // slabs
    if (U * (zper + yper) > (int64_t)1 << 30) return WSFFT_ERR_UNSUPPORTED;
    const int64_t window = engine_mode == 2 ? 3 * (int64_t)grid : 2 * (int64_t)grid;  // tiles held
    int64_t lag = (window + zper + yper - 1) / (zper + yper) + 2;  // measured: deeper lags do not help
    if (lag > U) lag = U;
    std::vector<EngItem> items;
    items.reserve((size_t)(U * (zper + yper) + batch * n * n / tq));
    for (int64_t j = 0; j < U + lag; ++j) {
        if (j < U)
            for (int64_t t = 0; t < zper; ++t)
                items.push_back(EngItem{ITEM_SIGNAL, (int)j, (int)t, 0});
        if (j >= lag)
            for (int64_t t = 0; t < yper; ++t)
                items.push_back(EngItem{ITEM_STRIDED | ITEM_WAIT, (int)(j - lag), (int)t, 0});
    }
    if (withhold) items[0].flags &= ~ITEM_SIGNAL;
    const int na = (int)items.size();
    if (engine_mode == 2)  // pipelined engine: x tiles too (cubes only, n0 == n)
        for (int64_t b = 0; b < batch; ++b)
            for (int64_t t = 0; t < n * n / tq; ++t) items.push_back(EngItem{ITEM_STRIDED, (int)b, (int)t, 0});
    const int nb = (int)items.size() - na;
    if (d_items) cudaFree(d_items);
    d_items = nullptr;
    if (cudaMalloc(&d_items, items.size() * sizeof(EngItem)) != cudaSuccess) {
        d_items = nullptr;
        return WSFFT_ERR_ALLOC;
    }
    if (upload(d_items, items.data(), items.size() * sizeof(EngItem)) != WSFFT_SUCCESS) return WSFFT_ERR_CUDA;
    if (1 + U > ctr_cap) {
        if (d_ctr) cudaFree(d_ctr);
        d_ctr = nullptr;
        ctr_cap = 0;
        if (cudaMalloc(&d_ctr, (size_t)(1 + U) * sizeof(uint32_t)) != cudaSuccess) {
            d_ctr = nullptr;
            return WSFFT_ERR_ALLOC;
        }
        ctr_cap = 1 + U;
    }
    const float sc = axis_scale(n, dir, norm), sc0 = axis_scale(n0, dir, norm);
    PassSpec a{};
    a.kind = engine_mode == 1 ? PASS_PERSIST_A : engine_mode == 3 ? PASS_WP_A : PASS_ENGINE_A;
    a.N = (int)n;
    a.E = 16;
    a.tile = (int)tp;
    a.trans_rows = zper;  // completion target of a slab
    a.items = d_items;
    a.nitems = na;
    a.units = U;
    a.conj_in = inv;
    a.c_scale = sc;
    a.s_scale = sc;
    a.transform_elems = n0 * n * n;
    PassSpec b{};
    if (engine_mode == 3 && wp_supports((int)n0)) {
        b.kind = PASS_WP_B;
        b.N = (int)n0;
        b.E = 16;
        b.inner = n * n;
        b.npencils_per_batch = n * n;
        b.src = SRC_OUT;
        b.dst = DST_OUT;
    } else if (engine_mode == 2) {
        b.kind = PASS_ENGINE_B;
        b.N = (int)n;
        b.E = 16;
        b.items = (const EngItem *)d_items + na;
        b.nitems = nb;
        b.units = 0;
    } else {
        // x: one launch of the strided superstep kernel, with the shape of
        // the one-launch-per-superstep schedule at 512 (16 pencils per block:
        // 32 values per thread in complex64, split-form pencil pairs in the
        // 16-bit types)
        b.kind = PASS_STRIDED;
        b.N = (int)n0;
        b.E = n0 == 512 ? (dtype == WSFFT_C32 ? 32 : 16) : default_E((int)n0);
        b.tile = n0 == 512 ? (dtype == WSFFT_C32 ? 16 : SPLIT_TILE + 16) : 0;
        b.inner = n * n;
        b.npencils_per_batch = n * n;
        b.src = SRC_OUT;
        b.dst = DST_OUT;
    }
    b.conj_out = inv;
    b.scale = engine_mode == 2 ? sc : sc0;
    b.transform_elems = n0 * n * n;
    passes.push_back(a);
    passes.push_back(b);
    for (auto &kv : overrides) {
        if (kv.first < (int)passes.size() && passes[kv.first].kind == PASS_STRIDED &&
            override_usable(kv.second.first, kv.second.second, passes[kv.first].N)) {
            passes[kv.first].E = kv.second.first;
            passes[kv.first].tile = kv.second.second;
        }
    }
    for (auto &p : passes) {
        p.tw = table(p.N, p.E);
        if (!p.tw) return WSFFT_ERR_ALLOC;
    }
    if (engine_mode == 1 && n == 512) {
        // the persistent 512 kernel's strided tiles have their own values per thread
        passes[0].tw2 = table(512, persist512_values_y());
        if (!passes[0].tw2) return WSFFT_ERR_ALLOC;
    }
    return WSFFT_SUCCESS;
}

// Whether the cluster-fused pass A of slab edge n can be resident on this
// plan's device (asked once per edge).
bool Plan::slab_runs(int n) {
    if (!slab_supports(n)) return false;
    int &c = slab_checked[n == 512 ? 1 : 0];
    if (c == 0) {
        SlabArgs probe{};
        int clusters = 0;
        const cudaError_t e = launch_slab(dtype, n, nullptr, nullptr, 1, probe, false, 0, &clusters);
        cudaGetLastError();  // a refused query leaves no sticky error
        c = (e == cudaSuccess && clusters > 0) ? 1 : -1;
    }
    return c > 0;
}

// Two-trip schedule of an n0 x n x n transform with the cluster-fused pass A
// (slab_cluster.cuh): the z and y supersteps of each n x n slab in one
// thread-block cluster (in -> out), then the x superstep as one launch of the
// strided kernel (out, in place).
int Plan::build_slab(int64_t n0, int64_t n, bool inv) {
    PassSpec a{};
    a.kind = PASS_SLAB_A;
    a.N = (int)n;
    a.inner = 1;
    a.npencils_per_batch = n0 * n;  // z pencils per transform
    a.units = n0;                   // slabs per transform
    a.transform_elems = n0 * n * n;
    a.src = SRC_IN;
    a.dst = DST_OUT;
    a.conj_in = inv;
    PassSpec b{};
    b.kind = PASS_STRIDED;
    b.N = (int)n0;
    b.E = default_E((int)n0);
    b.tile = 0;
    if (n0 == 512) {
        // the shape of the x superstep in the one-launch-per-superstep
        // schedule: 32 values per thread in complex64, split-form pencil
        // pairs in the 16-bit types
        b.E = dtype == WSFFT_C32 ? 32 : 16;
        b.tile = dtype == WSFFT_C32 ? 16 : SPLIT_TILE + 16;
    } else if (n0 == 1024) {
        b.E = 32;
        b.tile = 16;
    }
    b.inner = n * n;
    b.npencils_per_batch = n * n;
    b.transform_elems = n0 * n * n;
    b.src = SRC_OUT;
    b.dst = DST_OUT;
    b.conj_out = inv;
    const float sc = axis_scale(n, dir, norm), sc0 = axis_scale(n0, dir, norm);
    if (dtype == WSFFT_C32 && norm != WSFFT_NORM_ORTHO) {
        // complex64 defers every superstep's scale to the last store
        a.c_scale = a.s_scale = 1.f;
        b.scale = (float)((double)sc * (double)sc * (double)sc0);
    } else {
        a.c_scale = a.s_scale = sc;
        b.scale = sc0;
    }
    passes.push_back(a);
    passes.push_back(b);
    for (auto &kv : overrides)
        if (kv.first == 1 && override_usable(kv.second.first, kv.second.second, passes[1].N)) {
            passes[1].E = kv.second.first;
            passes[1].tile = kv.second.second;
        }
    passes[0].E = slab_ez(dtype != WSFFT_C32);
    passes[0].tw = table((int)n, passes[0].E);
    passes[0].tw2 = table((int)n, slab_ey());
    passes[1].tw = table(passes[1].N, passes[1].E);
    if (!passes[0].tw || !passes[0].tw2 || !passes[1].tw) return WSFFT_ERR_ALLOC;
    return WSFFT_SUCCESS;
}

// (Re)build the pass list from shape, direction and normalisation.
int Plan::build_schedule() {
    const int rc = make_schedule();
    const int copied = flush_tables();  // also after a failure: the tables made so far are remembered
    return rc != WSFFT_SUCCESS ? rc : copied;
}

int Plan::make_schedule() {
    passes.clear();
    fused.clear();
    fused_in_place = false;
    std::vector<int64_t> d;
    for (int i = 0; i < rank; ++i)
        if (dims[i] > 1) d.push_back(dims[i]);
    if (d.empty()) d.push_back(1);
    const int r = (int)d.size();
    const bool inv = dir == WSFFT_INVERSE;
    work_elems = 0;
    chunk = batch;

    // kernel shapes of a one-launch contiguous or strided superstep
    auto tune = [&](PassSpec &p, int64_t inner) {
        if (p.kind == PASS_CONTIG && p.N == 512) {
            // measured fastest at 512^3: 16 values per thread (radices
            // 16, 16, 2), 8 pencils per block (32 values per thread
            // matched it forward but lost 30% with the conjugate on load
            // of the inverse); complex64 one pencil per warp (256-thread
            // blocks, at the copy bandwidth), the 16-bit types as
            // split-form pairs (one pair per warp, packed FP32x2
            // butterflies: 13% faster there, the same in complex64)
            p.E = 16;
            p.tile = dtype == WSFFT_C32 ? 8 : SPLIT_TILE + 8;
        }
        if (p.N == 1024) {
            // measured at 1024^3: 32 values per thread (radix 32 x 32, one
            // exchange); contiguous: one warp per pencil, 8 per block;
            // strided: 16 pencils per block at strides of 2^17 elements
            // and more (128-byte rows: narrower tiles lost 10-50% there),
            // below that split-form pencil pairs with 16 values per pencil
            // and 8 pencils per block (two blocks per SM: 0.404 vs 0.427 ms
            // for 32 values per thread on a 1 GiB array at stride 1024)
            p.E = 32;
            p.tile = 8;
            if (p.kind == PASS_STRIDED) {
                if (inner >= ((int64_t)1 << 17)) {
                    p.tile = 16;
                } else if (inner % 8 == 0) {
                    p.E = 16;
                    p.tile = SPLIT_TILE + 8;
                } else if (dtype != WSFFT_C32) {
                    p.E = 16;
                }
            }
        }
        if (p.kind == PASS_STRIDED && p.N == 512 && inner % 16 == 0) {
            // measured fastest at 512^3: split-form pencil pairs (packed
            // FP32x2 butterflies, two adjacent elements per access), 16
            // values per pencil, 16 pencils per block, except for complex64
            // at strides of 2^17 elements and more, where 32 values per
            // thread for one pencil (one shared-memory exchange) match them
            p.E = 16;
            p.tile = SPLIT_TILE + 16;
            if (dtype == WSFFT_C32 && inner >= ((int64_t)1 << 17)) {
                p.E = 32;
                p.tile = 16;
            }
        }
        if (p.kind == PASS_CONTIG && pipe_contig(dtype, p.N, elems * batch)) {
            p.E = tile_table_E(p.N);
            p.tile = PIPE_TILE + FUSED_TILE_BITS;
        }
        if (p.kind == PASS_STRIDED) {
            // pipelined tile kernels (tile.cuh) where whole tiles fit; in 16-bit storage
            // not right after a contiguous superstep of 2048 or 4096 points while a few
            // tiles are a second wave (512 x 2048 FP16: 2^22 elements, 512 tiles for 456
            // resident blocks, 22.9 us against 20.4; 128 x 2048 in a batch of 20 23.6 against
            // 22.6; 1.5 * 2^22 elements 27.2 against 29.1; 1024 points are faster at each size)
            const bool held = dtype != WSFFT_C32 && axis_inner == 0 && p.N <= 512 && r >= 2 && inner == d[r - 1] &&
                              inner >= 2048 && elems * batch <= ((int64_t)5 << 20);
            const int tb = held ? 0 : pipe_tile_bits(dtype, p.N, inner, elems * batch);
            if (tb) {
                p.E = tile_table_E(p.N);
                p.tile = PIPE_TILE + tb;
            }
        }
    };

    // the same for a transposing contiguous superstep of `rows` pencils per transform
    auto trans_tile = [&](PassSpec &p, int64_t rows) {
        if (const int tb = pipe_tile_bits_variant(dtype, p.N, rows, elems * batch, false)) {
            p.E = tile_table_E(p.N);
            p.tile = PIPE_TILE + tb;
        }
    };

    // cluster-fused pass A (the default): the two inner axes equal and built
    // for that edge, and the kernel resident on this device
    if (layout == WSFFT_LAYOUT_NATURAL && r == 3 && engine_mode == 4 && d[1] == d[2] && slab_runs((int)d[1]))
        return build_slab(d[0], d[1], inv);
    // fused schedules: the two inner axes equal (n x n slabs); the pipelined
    // engine also runs the outer axis, so it needs a cube
    if (layout == WSFFT_LAYOUT_NATURAL && r == 3 && engine_mode >= 1 && engine_mode <= 3 && d[1] == d[2] &&
        engine_supports((int)d[1]) &&
        (engine_mode != 2 || d[0] == d[1]) && (engine_mode != 3 || wp_supports((int)d[1])) &&
        eng_grid > 0) {
        return build_engine(d[0], d[1], inv);
    }
    if (axis_inner > 0) {
        // wsfft_plan_create_axis: one superstep along an axis of length
        // dims[0] whose consecutive elements are axis_inner apart; pencils
        // (b, i) for batch index b and i < axis_inner
        PassSpec p{};
        p.N = (int)dims[0];
        p.kind = axis_inner == 1 ? PASS_CONTIG : PASS_STRIDED;
        p.E = default_E(p.N);
        tune(p, axis_inner);
        p.inner = axis_inner;
        p.npencils_per_batch = axis_inner;
        p.transform_elems = dims[0] * axis_inner;
        p.src = SRC_IN;
        p.dst = DST_OUT;
        p.conj_in = inv;
        p.conj_out = inv;
        p.scale = axis_scale(dims[0], dir, norm);
        passes.push_back(p);
    } else if (layout == WSFFT_LAYOUT_WAFER) {
        // Spectral side in the wafer's own order [n2][n0][n1] (Section 4.2:
        // after z is transformed, x and z swap places, then x and y; with the
        // PEs numbered like the input, X[k0][k1][k2] ends at k2 * n0 * n1 +
        // k0 * n1 + k1).  Built from the transposing store (pencil (t, row)
        // element k to t*N*rows + k*rows + row), three trips as in natural
        // order:
        //   forward:  z with the transposed store, rows n0*n1 (in -> work):
        //             [n0][n1][n2] -> [n2][n0][n1]; y contiguous (work ->
        //             out); x strided with stride n1 (out, in place)
        //   inverse:  y with the transposed store, rows n2*n0 (in -> work):
        //             [n2][n0][n1] -> [n1][n2][n0]; x with the transposed
        //             store, rows n1*n2 (work -> out): -> [n0][n1][n2]; z
        //             contiguous (out, in place)
        const int64_t n0 = dims[0], n1 = dims[1], n2 = dims[2];
        const int64_t total = n0 * n1 * n2;
        const int64_t per = total * elem_bytes(dtype);
        chunk = std::max<int64_t>(1, std::min<int64_t>(batch, ((int64_t)4096 << 20) / per));
        work_elems = chunk * total;
        auto trans = [&](int64_t n, int64_t rows, int src, int dst) {
            PassSpec t{};
            t.kind = PASS_CONTIG;
            t.N = (int)n;
            t.E = default_E(t.N);
            if (t.N == 1024 && dtype == WSFFT_C32) {
                t.E = 32;  // as in the four-step: one warp per pencil, 8 per block
                t.tile = 8;
            } else if (t.N == 512) {
                t.E = 32;  // half a warp per pencil, 16 per block (as in the swapped layout)
                t.tile = 16;
            }
            trans_tile(t, rows);
            t.variant = true;
            t.inner = 1;
            t.npencils_per_batch = rows;
            t.trans_rows = rows;
            t.src = src;
            t.dst = dst;
            t.scale = axis_scale(n, dir, norm);
            t.transform_elems = total;
            return t;
        };
        if (!inv) {
            passes.push_back(trans(n2, n0 * n1, SRC_IN, DST_WORK));
            PassSpec c{};
            c.kind = PASS_CONTIG;
            c.N = (int)n1;
            c.E = default_E(c.N);
            tune(c, 1);
            c.inner = 1;
            c.npencils_per_batch = n2 * n0;
            c.src = SRC_WORK;
            c.dst = DST_OUT;
            c.scale = axis_scale(n1, dir, norm);
            c.transform_elems = total;
            passes.push_back(c);
            PassSpec a{};
            a.kind = PASS_STRIDED;
            a.N = (int)n0;
            a.E = default_E(a.N);
            tune(a, n1);
            a.inner = n1;
            a.npencils_per_batch = n2 * n1;
            a.src = SRC_OUT;
            a.dst = DST_OUT;
            a.scale = axis_scale(n0, dir, norm);
            a.transform_elems = total;
            passes.push_back(a);
        } else {
            passes.push_back(trans(n1, n2 * n0, SRC_IN, DST_WORK));
            passes.push_back(trans(n0, n1 * n2, SRC_WORK, DST_OUT));
            PassSpec c{};
            c.kind = PASS_CONTIG;
            c.N = (int)n2;
            c.E = default_E(c.N);
            tune(c, 1);
            c.inner = 1;
            c.npencils_per_batch = n0 * n1;
            c.src = SRC_OUT;
            c.dst = DST_OUT;
            c.scale = axis_scale(n2, dir, norm);
            c.transform_elems = total;
            passes.push_back(c);
        }
        passes.front().conj_in = inv;
        passes.back().conj_out = inv;
        if (dtype == WSFFT_C32 && norm != WSFFT_NORM_ORTHO) {
            double total_scale = 1.0;
            for (auto &q : passes) {
                total_scale *= q.scale;
                q.scale = 1.f;
            }
            passes.back().scale = (float)total_scale;
        }
    } else if (layout == WSFFT_LAYOUT_SWAPPED) {
        // Spectral side with the last two axes swapped (the wafer's order,
        // Section 4.2).  The superstep along the last axis of the natural
        // side stores its pencils transposed (the four-step's staged store:
        // pencil (plane, row) element k to plane*N*rows + k*rows + row) into
        // the workspace, which turns the natural [a][b][c] into [a][c][b] or
        // back; the next axis is then contiguous on both sides of the swap,
        // and the first axis of a rank-3 array keeps its stride.
        //   forward:  c with the transposed store (in -> work), b contiguous
        //             (work -> out), a strided (out, in place)
        //   inverse:  b with the transposed store (in -> work), c contiguous
        //             (work -> out), a strided (out, in place)
        const int64_t A = rank == 3 ? dims[0] : 1, B = dims[rank - 2], C = dims[rank - 1];
        const int64_t total = A * B * C;
        const int64_t per = total * elem_bytes(dtype);
        chunk = std::max<int64_t>(1, std::min<int64_t>(batch, ((int64_t)4096 << 20) / per));
        work_elems = chunk * total;
        const int64_t n_t = inv ? B : C;  // axis of the transposing superstep
        const int64_t n_c = inv ? C : B;  // the other of the last two axes
        PassSpec t{};
        t.kind = PASS_CONTIG;
        t.N = (int)n_t;
        t.E = default_E(t.N);
        if (t.N == 1024 && dtype == WSFFT_C32) {
            t.E = 32;  // as in the four-step: one warp per pencil, 8 per block
            t.tile = 8;
        } else if (t.N == 512) {
            // 32 values per thread, 16 pencils per block: 0.33 against 0.39 ms
            // per GiB for the default 8 values x 16 pencils in complex64, 0.30
            // against 0.45 ms per 512 MiB in the 16-bit types (two resident
            // blocks of 256 threads against one of 1024)
            t.E = 32;
            t.tile = 16;
        }
        trans_tile(t, n_c);
        t.variant = true;
        t.inner = 1;
        t.npencils_per_batch = A * n_c;
        t.trans_rows = n_c;
        t.src = SRC_IN;
        t.dst = DST_WORK;
        t.conj_in = inv;
        t.scale = axis_scale(n_t, dir, norm);
        t.transform_elems = total;
        PassSpec c{};
        c.kind = PASS_CONTIG;
        c.N = (int)n_c;
        c.E = default_E(c.N);
        tune(c, 1);
        c.inner = 1;
        c.npencils_per_batch = A * n_t;
        c.src = SRC_WORK;
        c.dst = DST_OUT;
        c.scale = axis_scale(n_c, dir, norm);
        c.transform_elems = total;
        passes.push_back(t);
        passes.push_back(c);
        if (A > 1) {
            PassSpec a{};
            a.kind = PASS_STRIDED;
            a.N = (int)A;
            a.E = default_E(a.N);
            tune(a, B * C);
            a.inner = B * C;
            a.npencils_per_batch = B * C;
            a.src = SRC_OUT;
            a.dst = DST_OUT;
            a.scale = axis_scale(A, dir, norm);
            a.transform_elems = total;
            passes.push_back(a);
        }
        passes.back().conj_out = inv;
        if (dtype == WSFFT_C32 && norm != WSFFT_NORM_ORTHO) {
            double total_scale = 1.0;
            for (auto &q : passes) {
                total_scale *= q.scale;
                q.scale = 1.f;
            }
            passes.back().scale = (float)total_scale;
        }
    } else if (r == 1 && d[0] > 4096) {
        const int64_t n = d[0];
        const int lg = ilog2(n);
        // complex64 at n = 2^20 below 2^23 elements (where the pipelined tile
        // kernels do not take over) splits 2048 (contiguous) x 512 (strided)
        // rather than 1024 x 1024: on the general kernels the 512-point
        // strided superstep with the inter-step twiddle runs at 0.40 ms per
        // 2^27 elements against 0.53 for the 1024-point one
        const int lg1 = (lg == 20 && dtype == WSFFT_C32 && elems * batch < ((int64_t)1 << 23)) ? 11 : (lg + 1) / 2;
        const int64_t n1 = (int64_t)1 << lg1;  // contiguous length
        const int64_t n2 = n / n1;             // strided length
        const float sc = axis_scale(n, dir, norm);
        // workspace holds `chunk` transforms (at most ~4 GiB: measured 5%
        // faster than 512 MiB chunks at 512 x 2^20, fewer launch tails;
        // chunks small enough to stay in L2 were slower still)
        const int64_t per = n * elem_bytes(dtype);
        chunk = std::max<int64_t>(1, std::min<int64_t>(batch, ((int64_t)4096 << 20) / per));
        work_elems = chunk * n;
        PassSpec a{};
        a.kind = PASS_STRIDED;
        a.N = (int)n2;
        a.E = default_E((int)n2);
        if ((n2 == 1024 || n2 == 512) && dtype == WSFFT_C32) {
            // measured fastest at n = 2^20: 32 values per thread, 16 pencils per block
            a.E = 32;
            a.tile = 16;
        }
        if (const int tb = pipe_tile_bits_variant(dtype, n2, n1, elems * batch, true)) {
            a.E = tile_table_E(a.N);
            a.tile = PIPE_TILE + tb;
        }
        a.variant = true;
        a.inner = n1;
        a.npencils_per_batch = n1;
        a.src = SRC_IN;
        a.dst = DST_WORK;
        a.conj_in = inv;
        a.conj_out = false;
        a.scale = 1.f;
        a.twid_len = n;
        a.twid_shift = (lg + 1) / 2;
        a.transform_elems = n;
        PassSpec b{};
        b.kind = PASS_CONTIG;
        b.N = (int)n1;
        b.E = default_E((int)n1);
        if (n1 == 1024 && dtype == WSFFT_C32) {
            // one warp per pencil (32 values per thread), 8 pencils per block
            b.E = 32;
            b.tile = 8;
        } else if (n1 == 512) {
            // half a warp per pencil, 16 pencils per block (as in the swapped layout)
            b.E = 32;
            b.tile = 16;
        }
        trans_tile(b, n2);
        b.variant = true;
        b.inner = 1;
        b.npencils_per_batch = n2;
        b.src = SRC_WORK;
        b.dst = DST_OUT;
        b.conj_in = false;
        b.conj_out = inv;
        b.scale = sc;
        b.trans_rows = n2;
        b.transform_elems = n;
        passes.push_back(a);
        passes.push_back(b);
    } else {
        int64_t total = 1;
        for (auto v : d) total *= v;
        for (int ax = r - 1; ax >= 0; --ax) {
            int64_t inner = 1;
            for (int e = ax + 1; e < r; ++e) inner *= d[e];
            PassSpec p{};
            p.kind = ax == r - 1 ? PASS_CONTIG : PASS_STRIDED;
            p.N = (int)d[ax];
            p.E = default_E(p.N);
            p.variant = false;
            tune(p, inner);
            p.inner = inner;
            p.npencils_per_batch = total / d[ax];
            p.src = ax == r - 1 ? SRC_IN : SRC_OUT;
            p.dst = DST_OUT;
            p.conj_in = inv && ax == r - 1;
            p.conj_out = inv && ax == 0;
            p.scale = axis_scale(d[ax], dir, norm);
            p.transform_elems = total;
            passes.push_back(p);
        }
        if (dtype == WSFFT_C32 && norm != WSFFT_NORM_ORTHO) {
            // complex64 has the range to defer every superstep's 1/n to the
            // last pass (one scaled store instead of one per pass); the
            // reduced-precision types keep the per-superstep scale
            double total_scale = 1.0;
            for (auto &p : passes) {
                total_scale *= p.scale;
                p.scale = 1.f;
            }
            passes.back().scale = (float)total_scale;
        }
    }
    for (auto &kv : overrides) {
        if (kv.first < (int)passes.size() &&
            (passes[kv.first].kind == PASS_CONTIG || passes[kv.first].kind == PASS_STRIDED) &&
            override_usable(kv.second.first, kv.second.second, passes[kv.first].N)) {
            passes[kv.first].E = kv.second.first;
            passes[kv.first].tile = kv.second.second;
        }
    }
    // A strided superstep right after a contiguous one (the y superstep after
    // z) takes its tiles from the last slab down: the contiguous pass wrote
    // the last slabs last, and the first blocks then find them in L2
    // (measured at 512^3: y 0.330 -> 0.323 ms, 973 -> 967 us per transform)
    for (size_t i = 0; i < passes.size(); ++i)
        passes[i].reverse = i > 0 && passes[i].kind == PASS_STRIDED && passes[i - 1].kind == PASS_CONTIG &&
                            !passes[i].variant && !passes[i - 1].variant;
    for (auto &p : passes) {
        if (p.N > 4096 || !is_pow2(p.N)) return WSFFT_ERR_INVALID_SIZE;
        p.tw = p.tile == TC_TILE ? tc_table(p.N) : table(p.N, p.E);
        if (p.twid_len) {
            p.tw2 = p.tile >= PIPE_TILE ? fourstep_tile_table(p.twid_len, p.N)
                                        : fourstep_table(p.twid_len, p.twid_shift);
            if (!p.tw2) return WSFFT_ERR_ALLOC;
        }
        if (!p.tw) return WSFFT_ERR_ALLOC;
    }
    if (axis_inner == 0 && layout == WSFFT_LAYOUT_NATURAL && engine_mode == 0 && overrides.empty()) {
        int rc = build_fused(d, inv);
        if (rc == WSFFT_SUCCESS && fused.empty())
            rc = build_wide(d, inv, [&](int64_t n, int64_t inner) {
                PassSpec p{};
                p.kind = PASS_STRIDED;
                p.N = (int)n;
                p.E = default_E(p.N);
                tune(p, inner);
                p.inner = inner;
                p.npencils_per_batch = elems / n;
                p.src = SRC_OUT;
                p.dst = DST_OUT;
                p.scale = axis_scale(n, dir, norm);
                p.transform_elems = elems;
                return p;
            });
        if (rc != WSFFT_SUCCESS) return rc;
    }
    if (work_elems > work_cap) {
        if (work) cudaFree(work);
        work = nullptr;
        work_cap = 0;
        if (cudaMalloc(&work, (size_t)(work_elems * elem_bytes(dtype))) != cudaSuccess) {
            work = nullptr;
            return WSFFT_ERR_ALLOC;
        }
        work_cap = work_elems;
    }
    return WSFFT_SUCCESS;
}

bool Plan::overrides_launchable() const {
    for (const auto &kv : overrides) {
        if (kv.first < 0 || kv.first >= (int)passes.size()) return false;
        const PassSpec &ps = passes[kv.first];
        if (ps.E != kv.second.first || ps.tile != kv.second.second) return false;  // not applied
        TileArgs a{};
        a.npencils = 0;  // an empty launch returns before running
        if (launch(dtype, ps, nullptr, nullptr, a, 0) == cudaErrorInvalidValue) return false;
    }
    return true;
}

int Plan::run(const void *in, void *out, cudaStream_t st) {
    const int64_t eb = elem_bytes(dtype);
    const bool use_fused = !fused.empty() && (in != out || fused_in_place);
    for (int64_t b0 = 0; b0 < batch; b0 += chunk) {
        const int64_t nb = std::min(chunk, batch - b0);
        for (const auto &p : use_fused ? fused : passes) {
            if (p.kind == PASS_WP_B) {
                WpStridedArgs b{};
                b.in = out;
                b.out = out;
                b.inner = p.inner;
                b.log_inner = ilog2(p.inner);
                b.npencils = p.npencils_per_batch * batch;
                b.tw = p.tw;
                b.ci = 1.f;
                b.sx = p.scale;
                b.sy = p.conj_out ? -p.scale : p.scale;
                prof_begin(st);
                cudaError_t err = launch_wps(dtype, p.N, b, st);
                prof_end(st);
                if (err != cudaSuccess) return err == cudaErrorInvalidValue ? WSFFT_ERR_UNSUPPORTED : WSFFT_ERR_CUDA;
                continue;
            }
            if (p.kind == PASS_SLAB_A) {
                const int64_t off = b0 * p.transform_elems * eb;
                SlabArgs sa{};
                sa.ci = p.conj_in ? -1.f : 1.f;
                sa.zsx = sa.zsy = p.c_scale;
                sa.ysx = sa.ysy = p.s_scale;
                sa.tw_z = p.tw;
                sa.tw_y = p.tw2;
                const int64_t nslabs = p.units * nb;
                const bool pdl = nslabs * (int64_t)p.N * p.N * eb <= ((int64_t)2 << 30);
                prof_begin(st);
                cudaError_t e = launch_slab(dtype, p.N, (const char *)in + off, (char *)out + off, nslabs, sa, pdl,
                                            st, nullptr);
                prof_end(st);
                if (e != cudaSuccess) return e == cudaErrorInvalidValue ? WSFFT_ERR_UNSUPPORTED : WSFFT_ERR_CUDA;
                continue;
            }
            if (p.kind == PASS_ENGINE_A || p.kind == PASS_ENGINE_B || p.kind == PASS_PERSIST_A ||
                p.kind == PASS_WP_A) {
                EngArgs e{};
                e.items = (const EngItem *)p.items;
                e.nitems = p.nitems;
                e.ctr = d_ctr;
                e.status = d_status;
                e.tw_c = p.tw;
                e.tw_s = p.tw2 ? p.tw2 : p.tw;
                e.timeout_ns = (uint64_t)wait_timeout_ns;
                const int64_t n = p.N;
                if (p.kind == PASS_ENGINE_A || p.kind == PASS_PERSIST_A || p.kind == PASS_WP_A) {
                    e.c_src = in;
                    e.c_dst = out;
                    e.s_src = out;
                    e.s_dst = out;
                    e.unit_elems = n * n;
                    e.s_stride = n;
                    e.c_ci = p.conj_in ? -1.f : 1.f;
                    e.c_sx = e.c_sy = p.c_scale;
                    e.s_ci = 1.f;
                    e.s_sx = e.s_sy = p.s_scale;
                    e.dep_target = (uint32_t)p.trans_rows;
                    e.s_evict_first = 0;
                } else {
                    e.s_src = out;
                    e.s_dst = out;
                    e.unit_elems = n * n * n;
                    e.s_stride = n * n;
                    e.s_ci = 1.f;
                    e.s_sx = p.scale;
                    e.s_sy = p.conj_out ? -p.scale : p.scale;
                    e.s_evict_first = 1;
                }
                if (cudaMemsetAsync(d_ctr, 0, (size_t)(1 + p.units) * sizeof(uint32_t), st) != cudaSuccess)
                    return WSFFT_ERR_CUDA;
                prof_begin(st);
                cudaError_t err = p.kind == PASS_PERSIST_A
                                      ? launch_persist(dtype, p.N, e, 0, nullptr, persist_grid, st)
                                  : p.kind == PASS_WP_A ? launch_wpp(dtype, p.N, e, nullptr, persist_grid, st)
                                                        : launch_engine(dtype, p.N, e, eng_grid, st);
                prof_end(st);
                if (err != cudaSuccess) return err == cudaErrorInvalidValue ? WSFFT_ERR_UNSUPPORTED : WSFFT_ERR_CUDA;
                continue;
            }
            const int64_t off = b0 * p.transform_elems * eb;
            const char *src = p.src == SRC_IN ? (const char *)in + off
                              : p.src == SRC_OUT ? (const char *)out + off
                                                 : (const char *)work;
            char *dst = p.dst == DST_OUT ? (char *)out + off : (char *)work;
            TileArgs a = pass_args(p, p.npencils_per_batch * nb);
            a.elems = p.transform_elems * nb;
            prof_begin(st);
            cudaError_t e = launch(dtype, p, src, dst, a, st);
            prof_end(st);
            if (e != cudaSuccess) return e == cudaErrorInvalidValue ? WSFFT_ERR_UNSUPPORTED : WSFFT_ERR_CUDA;
        }
    }
    return WSFFT_SUCCESS;
}

TileArgs Plan::pass_args(const PassSpec &p, int64_t npencils) const {
    TileArgs a{};
    a.npencils = npencils;
    a.inner = p.inner;
    a.log_inner = ilog2(p.inner);
    a.tw = p.tw;
    a.conj_in = p.conj_in ? -1.f : 1.f;
    a.sx = p.scale;
    a.sy = p.conj_out ? -p.scale : p.scale;
    a.trans_rows = p.trans_rows;
    a.tw_hi = p.twid_len ? p.tw2 : nullptr;
    // the low table follows the high one (the tile kernels': the one over k1)
    a.tw_lo = !p.twid_len ? nullptr
              : p.tile >= PIPE_TILE ? p.tw2 + (p.twid_len / p.N) * tile_table_E(p.N)
                                    : p.tw2 + (p.twid_len >> p.twid_shift);
    a.tw_shift = p.twid_len ? p.twid_shift : 0;
    a.tw_mask = p.twid_len ? (int)(p.twid_len - 1) : 0;
    a.status = d_status;
    a.timeout_ns = (uint64_t)wait_timeout_ns;
    a.reverse = p.reverse ? 1 : 0;
    if (p.kind == PASS_TILE_SLAB) {
        a.tw2 = p.tw2;
        a.log_y0 = p.y0b;
    } else if (p.kind == PASS_TILE_WIDE) {
        a.tw_hi = p.tw2;
        a.log_y0 = p.y0b;
    } else if (p.kind == PASS_TILE_OUTER) {
        a.tw_hi = p.tw2;
        a.ystep = (int64_t)1 << (p.zb + p.yb);
        a.log_row = p.zb;
        a.log_cols = p.zb + p.yb;
        a.log_transform = ilog2(p.transform_elems);
        a.nk1 = 1 << p.yb;
    }
    return a;
}

// Host buffers, rank 3 with one launch per superstep: the copies overlap the
// supersteps.  Slab chunks (along the first axis) are copied in on a second
// stream and the z superstep of each chunk (slab-local) runs as soon as the
// chunk has arrived; the x superstep, which needs every slab, runs over the
// whole array; then the y superstep (slab-local again) runs chunk by chunk
// and each finished chunk goes back to the host with one contiguous copy, on
// a third stream, while the next is transformed.  The supersteps are taken in
// the order z, x, y (the order of axes is free, Section 1).  The data crosses
// the host link once in each direction; the x superstep and one chunk's z
// and y are the only compute of a lone transform not hidden behind a copy,
// and in a batch the next transform's copies in share the time of the
// previous one's copies out (the two directions of the link).  (Chunking the
// x superstep instead would need strided 2D copies back, measured 17% slower
// than contiguous ones on this link.)
bool Plan::can_pipeline_host() const {
    if (ragged || rank != 3 || chunk != batch || passes.size() != 3 || dims[0] < 2) return false;
    if (passes[0].kind != PASS_CONTIG || passes[1].kind != PASS_STRIDED || passes[2].kind != PASS_STRIDED)
        return false;
    for (const auto &p : passes)
        if (p.variant || p.src == SRC_WORK || p.dst == DST_WORK) return false;
    return true;
}

int Plan::run_host_pipelined(const void *hin, void *hout, cudaStream_t st) {
    constexpr int K = 8;  // chunks per direction
    // streams and events are made on first use; a call that failed half-way
    // through making them leaves nothing half-made for the next one
    if (!copy_stream && cudaStreamCreateWithFlags(&copy_stream, cudaStreamNonBlocking) != cudaSuccess) {
        copy_stream = nullptr;
        return WSFFT_ERR_CUDA;
    }
    if (!copy_out_stream && cudaStreamCreateWithFlags(&copy_out_stream, cudaStreamNonBlocking) != cudaSuccess) {
        copy_out_stream = nullptr;
        return WSFFT_ERR_CUDA;
    }
    if (pipe_ev.size() != 2 * K + 2) {
        std::vector<cudaEvent_t> evs(2 * K + 2, nullptr);
        for (auto &e : evs)
            if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
                for (auto made : evs)
                    if (made) cudaEventDestroy(made);
                return WSFFT_ERR_CUDA;
            }
        pipe_ev.swap(evs);
    }
    const int64_t eb = elem_bytes(dtype);
    const int64_t n0 = dims[0], I = dims[1] * dims[2];
    const int kz = (int)std::min<int64_t>(K, n0);
    cudaEvent_t ev_start = pipe_ev[2 * K], ev_done = pipe_ev[2 * K + 1];
    char *dev = (char *)host_buf;
    auto ck = [](cudaError_t e) { return e == cudaSuccess; };
    // Both copy streams start after the work already on `st`.  Copies in run
    // on copy_stream and copies out on copy_out_stream, so with a batch the
    // next transform's chunks come in (one direction of the link) while the
    // previous one's go out (the other): the transforms own disjoint parts of
    // the device buffer and of the host buffers (also in place: transform b
    // reads and writes only its own host slice).
    if (!ck(cudaEventRecord(ev_start, st)) || !ck(cudaStreamWaitEvent(copy_stream, ev_start, 0)) ||
        !ck(cudaStreamWaitEvent(copy_out_stream, ev_start, 0)))
        return WSFFT_ERR_CUDA;
    for (int64_t b = 0; b < batch; ++b) {
        const char *hb = (const char *)hin + b * elems * eb;
        char *ho = (char *)hout + b * elems * eb;
        char *db = dev + b * elems * eb;
        auto run_pass = [&](const PassSpec &p, char *ptr, int64_t npencils) {
            const TileArgs a = pass_args(p, npencils);
            prof_begin(st);
            cudaError_t e = launch(dtype, p, ptr, ptr, a, st);
            prof_end(st);
            return e == cudaSuccess ? WSFFT_SUCCESS : e == cudaErrorInvalidValue ? WSFFT_ERR_UNSUPPORTED : WSFFT_ERR_CUDA;
        };
        // in: slab chunks, each followed by its z superstep
        for (int c = 0; c < kz; ++c) {
            const int64_t s0 = c * n0 / kz, s1 = (c + 1) * n0 / kz;
            const int64_t o = s0 * I * eb, bytes = (s1 - s0) * I * eb;
            if (!ck(cudaMemcpyAsync(db + o, hb + o, (size_t)bytes, cudaMemcpyHostToDevice, copy_stream)) ||
                !ck(cudaEventRecord(pipe_ev[c], copy_stream)) || !ck(cudaStreamWaitEvent(st, pipe_ev[c], 0)))
                return WSFFT_ERR_CUDA;
            const int rc = run_pass(passes[0], db + o, (s1 - s0) * dims[1]);
            if (rc != WSFFT_SUCCESS) return rc;
        }
        // the x superstep over the whole array; the inverse's conjugation of
        // the output moves to the y superstep, which now runs last
        PassSpec px = passes[2], py = passes[1];
        py.conj_out = px.conj_out;
        px.conj_out = false;
        int rc = run_pass(px, db, I);
        if (rc != WSFFT_SUCCESS) return rc;
        // out: the y superstep of each slab chunk, then its copy back
        for (int c = 0; c < kz; ++c) {
            const int64_t s0 = c * n0 / kz, s1 = (c + 1) * n0 / kz;
            const int64_t o = s0 * I * eb, bytes = (s1 - s0) * I * eb;
            rc = run_pass(py, db + o, (s1 - s0) * dims[2]);
            if (rc != WSFFT_SUCCESS) return rc;
            if (!ck(cudaEventRecord(pipe_ev[K + c], st)) ||
                !ck(cudaStreamWaitEvent(copy_out_stream, pipe_ev[K + c], 0)) ||
                !ck(cudaMemcpyAsync(ho + o, db + o, (size_t)bytes, cudaMemcpyDeviceToHost, copy_out_stream)))
                return WSFFT_ERR_CUDA;
        }
    }
    // `st` ends after the last copy out (every copy in was waited for by a
    // z superstep on `st`)
    if (!ck(cudaEventRecord(ev_done, copy_out_stream)) || !ck(cudaStreamWaitEvent(st, ev_done, 0)))
        return WSFFT_ERR_CUDA;
    return WSFFT_SUCCESS;
}

// The grouped launches of a ragged plan (complex64): instances whose inner
// axes fit the fused tiles (fused_tile_rule) take two trips, one launch per
// tile shape and trip over all of them; the others (more than 2^22 elements,
// or rows shorter than a tile's) run one after the other on plans of their
// own.  256 shapes of 32..256 points per axis: 3.95 ms as one queue, whose
// tiles make three trips at 0.87 of the copy rate, 2.90 ms so; 48 shapes
// 535-749 us and 436-617, 12 shapes 114-253 and 83-238 (half of the elements in
// instances on plans of their own), 8 shapes 87-152 and 59-148, one 20.8 and 10.4.
int Plan::rag_build_groups(RagInst *inst) {
    rag_groups.clear();
    rag_single.clear();
    if (dtype != WSFFT_C32) return WSFFT_SUCCESS;
    std::map<std::array<int, 3>, std::vector<RagRef>> groups;  // kind, b0, b1
    for (int i = 0; i < rag_count; ++i) {
        const std::vector<int64_t> d(rag_dims.begin() + 3 * (size_t)i, rag_dims.begin() + 3 * (size_t)i + 3);
        const FusedShape f = fused_tile_rule(d);
        if (!f.use) {
            Plan *&sub = rag_subplans[d];
            if (!sub) {
                sub = new (std::nothrow) Plan();
                if (!sub) return WSFFT_ERR_ALLOC;
                sub->device = device;
                sub->lender = this;
                sub->sm_count = sub->eng_grid = sm_count;
                sub->rank = 3;
                sub->elems = 1;
                for (int k = 0; k < 3; ++k) sub->elems *= sub->dims[k] = d[k];
                sub->dtype = dtype;
                sub->dir = dir;
                sub->norm = norm;
                const int rc = sub->build_schedule();
                if (rc != WSFFT_SUCCESS) return rc;
            }
            rag_single.emplace_back(i, sub);
            continue;
        }
        const int64_t rows = (int64_t)1 << f.yb;
        inst[i].log_y0 = f.y0b;
        inst[i].first = axis_scale(d[2] * rows, dir, norm);
        inst[i].last = axis_scale(d[0] << f.y0b, dir, norm);
        const int tiles = (int)((d[0] * d[1] * d[2]) >> FUSED_TILE_BITS);
        auto add = [&](int kind, int b0, int b1) {
            auto &refs = groups[{kind, b0, b1}];
            const size_t at = refs.size();
            refs.resize(at + tiles);
            for (int t = 0; t < tiles; ++t) refs[at + t] = RagRef{i, t};
        };
        add(0, f.zb, f.yb);
        if (f.outer) add(1, ilog2(d[0]), f.y0b);
        else add(2, (int)d[0], 0);
    }
    std::vector<RagRef> refs;
    rag_first_groups = 0;
    for (auto &kv : groups) {  // ordered by kind: the first trips come first
        RagGroup g{};
        g.kind = kv.first[0];
        g.b0 = kv.first[1];
        g.b1 = kv.first[2];
        g.ref0 = (int64_t)refs.size();
        g.tiles = (int64_t)kv.second.size();
        refs.insert(refs.end(), kv.second.begin(), kv.second.end());
        if (g.kind == 0) {
            g.tw = table(1 << g.b0, 16);
            g.tw2 = table(1 << g.b1, 32);
            ++rag_first_groups;
        } else if (g.kind == 1) {
            g.tw = g.tw2 = table2(1 << g.b0, 32 >> g.b1);
            for (int zb = 5; zb <= 8; ++zb) {
                const int log_n1 = FUSED_TILE_BITS + g.b1 - zb;
                if (log_n1 > 8) continue;
                g.cls[zb - 5] = class_table(1 << log_n1, 1 << g.b1);
                if (!g.cls[zb - 5]) return WSFFT_ERR_ALLOC;
            }
        } else {
            g.tw = g.tw2 = table(g.b0, tile_table_E(g.b0));
        }
        if (!g.tw || !g.tw2) return WSFFT_ERR_ALLOC;
        rag_groups.push_back(g);
    }
    if (refs.empty()) return WSFFT_SUCCESS;
    if (!rag_refs && cudaMalloc(&rag_refs, refs.size() * sizeof(RagRef)) != cudaSuccess) {
        rag_refs = nullptr;
        return WSFFT_ERR_ALLOC;
    }
    return upload(rag_refs, refs.data(), refs.size() * sizeof(RagRef));
}

// The launches of one trip do not depend on each other: only its first waits
// at its start for what is before it in the stream, the others at their end.
// A launch starts once every block of the one before it has let it (after
// that one's own wait, if it has one), so all of a trip's launches start
// after what the first waited for; and a launch is complete only when the one
// before it is, so whatever waits for the last one waits for all.
int Plan::rag_run_grouped(const void *const *in, void *const *out, cudaStream_t st) {
    auto run_groups = [&](size_t from, size_t to) {
        for (size_t i = from; i < to; ++i) {
            const RagGroup &g = rag_groups[i];
            TileArgs a{};
            a.tiles = g.tiles;
            a.refs = static_cast<const RagRef *>(rag_refs) + g.ref0;
            a.inst = static_cast<const RagInst *>(rag_inst);
            a.tw = g.tw;
            a.tw2 = g.tw2;
            for (int k = 0; k < 4; ++k) a.cls[k] = g.cls[k];
            a.ystep = (int64_t)1 << FUSED_TILE_BITS;
            a.late = i > from;
            // the inverse conjugates on the first load and on the last store
            a.conj_in = g.kind == 0 && dir == WSFFT_INVERSE ? -1.f : 1.f;
            a.sx = 1.f;
            a.sy = g.kind != 0 && dir == WSFFT_INVERSE ? -1.f : 1.f;
            prof_begin(st);
            const cudaError_t e = g.kind == 0   ? launch_ragged_slab_c32(g.b0, g.b1, a, st)
                                  : g.kind == 1 ? launch_ragged_outer_c32(g.b0, g.b1, a, st)
                                                : launch_ragged_strided_c32(g.b0, a, st);
            prof_end(st);
            if (e != cudaSuccess) return WSFFT_ERR_CUDA;
        }
        return WSFFT_SUCCESS;
    };
    int rc = run_groups(0, rag_first_groups);
    for (size_t i = 0; rc == WSFFT_SUCCESS && i < rag_single.size(); ++i) {
        const auto &s = rag_single[i];
        prof_begin(st);
        rc = s.second->run(in[s.first], out[s.first], st);
        prof_end(st);
    }
    return rc == WSFFT_SUCCESS ? run_groups(rag_first_groups, rag_groups.size()) : rc;
}

// (Re)build a ragged plan's instance records and tile queue for its current
// tile-shape selection and lag: tile counts per superstep follow the chosen
// shape of each axis length; the queue holds z tiles of instance s, y tiles
// of s - lag and x tiles of s - 2*lag, so every wait is on smaller tickets.
int Plan::rag_build() {
    const int count = rag_count;
    if (wait_own_work() != WSFFT_SUCCESS) return WSFFT_ERR_CUDA;  // no execute may still read the tables
    if (rag_uploaded && cudaEventSynchronize(rag_copied) != cudaSuccess) return WSFFT_ERR_CUDA;
    for (int k = 0; k < 4; ++k)
        for (int alt = 0; alt < 2; ++alt) {
            rag_tw[k][alt] = table(32 << k, rag_E(32 << k, alt));
            if (!rag_tw[k][alt]) return WSFFT_ERR_ALLOC;
        }
    auto alt_of = [&](int64_t N) { return (rag_esel >> (ilog2(N) - 5)) & 1; };
    std::vector<RagInst> inst((size_t)count);
    for (int i = 0; i < count; ++i) {
        RagInst &I = inst[i];
        memset(&I, 0, sizeof(I));
        for (int d = 0; d < 3; ++d) I.n[d] = (int)rag_dims[3 * (size_t)i + d];
        I.log_n2 = ilog2(I.n[2]);
        I.log_n12 = ilog2((int64_t)I.n[1] * I.n[2]);
        const int64_t n0 = I.n[0], n1 = I.n[1], n2 = I.n[2];
        const int64_t P = rag_P((int)n2, alt_of(n2)), W1 = rag_W((int)n1, alt_of(n1)), W0 = rag_W((int)n0, alt_of(n0));
        I.tiles[0] = (int)((n0 * n1 + P - 1) / P);
        I.tiles[1] = (int)((n0 * n2 + W1 - 1) / W1);
        I.tiles[2] = (int)((n1 * n2 + W0 - 1) / W0);
        // scales of the z, y, x supersteps
        I.scale[0] = axis_scale(n2, dir, norm);
        I.scale[1] = axis_scale(n1, dir, norm);
        I.scale[2] = axis_scale(n0, dir, norm);
    }
    {
        const int rc = rag_build_groups(inst.data());
        const int copied = flush_tables();
        if (rc != WSFFT_SUCCESS) return rc;
        if (copied != WSFFT_SUCCESS) return copied;
    }
    const int L = rag_lag;
    size_t nitems = 0;
    for (const RagInst &I : inst) nitems += (size_t)I.tiles[0] + I.tiles[1] + I.tiles[2];
    if (nitems > (size_t)0x7fffffff) return WSFFT_ERR_UNSUPPORTED;
    std::vector<RagItem> items(nitems);
    RagItem *item = items.data();
    auto add = [&](int s, int step, int flags) {
        if (s < 0 || s >= count) return;
        for (int t = 0; t < inst[s].tiles[step]; ++t) *item++ = RagItem{flags | (step << 8), s, t, 0};
    };
    for (int s = 0; s < count + 2 * L; ++s) {
        add(s, 0, ITEM_SIGNAL);
        add(s - L, 1, ITEM_STRIDED | ITEM_WAIT | ITEM_SIGNAL);
        add(s - 2 * L, 2, ITEM_STRIDED | ITEM_WAIT);
    }
    const size_t ib = items.size() * sizeof(RagItem), nb = inst.size() * sizeof(RagInst);
    if (items.size() > (size_t)rag_items_cap) {
        if (rag_items) cudaFree(rag_items);
        rag_items = nullptr;
        rag_items_cap = 0;
        if (cudaMalloc(&rag_items, ib) != cudaSuccess) {
            rag_items = nullptr;
            return WSFFT_ERR_ALLOC;
        }
        rag_items_cap = (int64_t)items.size();
    }
    if (!rag_inst) {
        if (cudaMalloc(&rag_inst, nb) != cudaSuccess) {
            rag_inst = nullptr;
            return WSFFT_ERR_ALLOC;
        }
        if (cudaMallocHost(&rag_inst_host, nb) != cudaSuccess) {
            rag_inst_host = nullptr;
            return WSFFT_ERR_ALLOC;
        }
    } else {
        // keep the pointers of the last execute; the tile counts changed
        const RagInst *old = static_cast<const RagInst *>(rag_inst_host);
        for (int i = 0; i < count; ++i) {
            inst[i].in = old[i].in;
            inst[i].out = old[i].out;
        }
    }
    memcpy(rag_inst_host, inst.data(), nb);
    rag_uploaded = false;  // the next execute uploads the records again
    rag_nitems = (int)items.size();
    return upload(rag_items, items.data(), ib);
}

int Plan::upload(void *dst, const void *src, size_t bytes) {
    if (!setup_st && cudaStreamCreateWithFlags(&setup_st, cudaStreamNonBlocking) != cudaSuccess) {
        setup_st = nullptr;
        return WSFFT_ERR_CUDA;
    }
    if (cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, setup_st) != cudaSuccess) return WSFFT_ERR_CUDA;
    return cudaStreamSynchronize(setup_st) == cudaSuccess ? WSFFT_SUCCESS : WSFFT_ERR_CUDA;
}

int Plan::zero(void *dst, size_t bytes) {
    if (!setup_st && cudaStreamCreateWithFlags(&setup_st, cudaStreamNonBlocking) != cudaSuccess) {
        setup_st = nullptr;
        return WSFFT_ERR_CUDA;
    }
    if (cudaMemsetAsync(dst, 0, bytes, setup_st) != cudaSuccess) return WSFFT_ERR_CUDA;
    return cudaStreamSynchronize(setup_st) == cudaSuccess ? WSFFT_SUCCESS : WSFFT_ERR_CUDA;
}

void Plan::mark_done(cudaStream_t st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    if (cs != cudaStreamCaptureStatusNone) return;  // a graph's launches are the caller's to wait for
    auto it = done_ev.find(st);
    if (it == done_ev.end()) {
        cudaEvent_t e;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return;
        it = done_ev.emplace(st, e).first;
    }
    cudaEventRecord(it->second, st);
}

int Plan::wait_own_work() {
    bool ok = true;
    for (auto &kv : done_ev) ok &= cudaEventSynchronize(kv.second) == cudaSuccess;
    if (copy_stream) ok &= cudaStreamSynchronize(copy_stream) == cudaSuccess;
    if (copy_out_stream) ok &= cudaStreamSynchronize(copy_out_stream) == cudaSuccess;
    if (setup_st) ok &= cudaStreamSynchronize(setup_st) == cudaSuccess;
    return ok ? WSFFT_SUCCESS : WSFFT_ERR_CUDA;
}

void Plan::prof_begin(cudaStream_t st) {
    if (prof_used < (int)prof_ev.size() / 2) cudaEventRecord(prof_ev[2 * prof_used], st);
}

void Plan::prof_end(cudaStream_t st) {
    if (prof_used < (int)prof_ev.size() / 2) {
        cudaEventRecord(prof_ev[2 * prof_used + 1], st);
        ++prof_used;
    }
}

Plan::~Plan() {
    for (auto e : prof_ev) cudaEventDestroy(e);
    for (auto &kv : rag_subplans) delete kv.second;
    if (rag_refs) cudaFree(rag_refs);
    if (rag_items) cudaFree(rag_items);
    if (rag_inst) cudaFree(rag_inst);
    if (rag_inst_host) cudaFreeHost(rag_inst_host);
    if (rag_copied) cudaEventDestroy(rag_copied);
    if (d_items) cudaFree(d_items);
    if (d_ctr) cudaFree(d_ctr);
    for (auto &b : table_blocks) cudaFree(b.device);
    if (work) cudaFree(work);
    if (host_buf) cudaFree(host_buf);
    for (auto e : pipe_ev)
        if (e) cudaEventDestroy(e);
    if (copy_stream) cudaStreamDestroy(copy_stream);
    if (copy_out_stream) cudaStreamDestroy(copy_out_stream);
    if (d_status) cudaFree(d_status);
    for (auto &kv : done_ev) cudaEventDestroy(kv.second);
    if (setup_st) cudaStreamDestroy(setup_st);
}

}  // namespace wsfft

extern "C" {

const char *wsfft_status_string(int s) {
    switch (s) {
        case WSFFT_SUCCESS: return "success";
        case WSFFT_ERR_INVALID_ARG: return "invalid argument";
        case WSFFT_ERR_INVALID_SIZE: return "invalid size (axes must be powers of two within range)";
        case WSFFT_ERR_UNSUPPORTED: return "unsupported configuration";
        case WSFFT_ERR_ALLOC: return "allocation failed";
        case WSFFT_ERR_CUDA: return "CUDA runtime error";
        case WSFFT_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        default: return "unknown status";
    }
}

int wsfft_plan_create(wsfft_plan *plan, const int64_t *dims, int rank, int dtype, int direction,
                      int64_t batch) {
    if (!plan) return WSFFT_ERR_INVALID_ARG;
    *plan = nullptr;
    if (!dims || rank < 1 || rank > 3 || batch < 1) return WSFFT_ERR_INVALID_ARG;
    if (dtype != WSFFT_C32 && dtype != WSFFT_C16F && dtype != WSFFT_C16BF) return WSFFT_ERR_INVALID_ARG;
    if (direction != WSFFT_FORWARD && direction != WSFFT_INVERSE) return WSFFT_ERR_INVALID_ARG;
    for (int i = 0; i < rank; ++i) {
        if (!is_pow2(dims[i])) return WSFFT_ERR_INVALID_SIZE;
        if (rank > 1 && dims[i] > 4096) return WSFFT_ERR_INVALID_SIZE;
        if (rank == 1 && dims[i] > ((int64_t)1 << 24)) return WSFFT_ERR_INVALID_SIZE;
    }
    Plan *p = new (std::nothrow) Plan();
    if (!p) return WSFFT_ERR_ALLOC;
    if (cudaGetDevice(&p->device) != cudaSuccess) {
        delete p;
        return WSFFT_ERR_CUDA;
    }
    p->rank = rank;
    for (int i = 0; i < rank; ++i) p->dims[i] = dims[i];
    cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device);
    p->eng_grid = p->sm_count;  // one engine block per SM (its shared memory fills the SM)
    p->dtype = dtype;
    p->dir = direction;
    p->batch = batch;
    p->norm = dtype == WSFFT_C32 ? WSFFT_NORM_PAPER : WSFFT_NORM_ORTHO;
    p->elems = 1;
    for (int i = 0; i < rank; ++i) p->elems *= dims[i];
    if (cudaMalloc(&p->d_status, sizeof(int)) != cudaSuccess) {
        p->d_status = nullptr;
        delete p;
        return WSFFT_ERR_ALLOC;
    }
    if (p->zero(p->d_status, sizeof(int)) != WSFFT_SUCCESS) {
        delete p;
        return WSFFT_ERR_CUDA;
    }
    int rc = p->build_schedule();
    if (rc != WSFFT_SUCCESS) {
        delete p;
        return rc;
    }
    autotune_apply_cached(*p);  // a remembered choice for this key, if any
    *plan = reinterpret_cast<wsfft_plan>(p);
    return WSFFT_SUCCESS;
}

int wsfft_plan_create_axis(wsfft_plan *plan, int64_t n, int64_t inner, int dtype, int direction, int64_t batch) {
    if (!plan) return WSFFT_ERR_INVALID_ARG;
    *plan = nullptr;
    if (batch < 1 || inner < 1) return WSFFT_ERR_INVALID_ARG;
    if (dtype != WSFFT_C32 && dtype != WSFFT_C16F && dtype != WSFFT_C16BF) return WSFFT_ERR_INVALID_ARG;
    if (direction != WSFFT_FORWARD && direction != WSFFT_INVERSE) return WSFFT_ERR_INVALID_ARG;
    if (!is_pow2(n) || n > 4096 || !is_pow2(inner) || inner > ((int64_t)1 << 40)) return WSFFT_ERR_INVALID_SIZE;
    Plan *p = new (std::nothrow) Plan();
    if (!p) return WSFFT_ERR_ALLOC;
    if (cudaGetDevice(&p->device) != cudaSuccess) {
        delete p;
        return WSFFT_ERR_CUDA;
    }
    cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device);
    p->eng_grid = p->sm_count;
    p->rank = 1;
    p->dims[0] = n;
    p->axis_inner = inner;
    p->dtype = dtype;
    p->dir = direction;
    p->batch = batch;
    p->norm = dtype == WSFFT_C32 ? WSFFT_NORM_PAPER : WSFFT_NORM_ORTHO;
    p->elems = n * inner;
    if (cudaMalloc(&p->d_status, sizeof(int)) != cudaSuccess) {
        p->d_status = nullptr;
        delete p;
        return WSFFT_ERR_ALLOC;
    }
    int rc = p->zero(p->d_status, sizeof(int));
    if (rc == WSFFT_SUCCESS) rc = p->build_schedule();
    if (rc != WSFFT_SUCCESS) {
        delete p;
        return rc;
    }
    *plan = reinterpret_cast<wsfft_plan>(p);
    return WSFFT_SUCCESS;
}

int wsfft_plan_set_norm(wsfft_plan plan, int norm) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || norm < WSFFT_NORM_PAPER || norm > WSFFT_NORM_FORWARD) return WSFFT_ERR_INVALID_ARG;
    if (p->ragged) return WSFFT_ERR_UNSUPPORTED;
    p->norm = norm;
    return p->build_schedule();
}

int wsfft_plan_set_layout(wsfft_plan plan, int layout) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || (layout != WSFFT_LAYOUT_NATURAL && layout != WSFFT_LAYOUT_SWAPPED && layout != WSFFT_LAYOUT_WAFER))
        return WSFFT_ERR_INVALID_ARG;
    if (p->ragged || (p->axis_inner > 0 && layout != WSFFT_LAYOUT_NATURAL)) return WSFFT_ERR_UNSUPPORTED;
    if (layout == WSFFT_LAYOUT_WAFER) {
        // every axis passes through the transposing store in one direction
        // or the other: 64..4096 points each (its row counts, products of
        // two axes, are then multiples of its pencils per block)
        if (p->rank != 3) return WSFFT_ERR_UNSUPPORTED;
        for (int i = 0; i < 3; ++i)
            if (p->dims[i] < 64 || p->dims[i] > 4096) return WSFFT_ERR_UNSUPPORTED;
    }
    if (layout == WSFFT_LAYOUT_SWAPPED) {
        // the transposing store is built for pencils of 64..4096 points, and
        // its tiles need the row count to be a multiple of their pencils per
        // block (at most 32, so rows >= 64 suffice)
        if (p->rank < 2) return WSFFT_ERR_UNSUPPORTED;
        for (int i = p->rank - 2; i < p->rank; ++i)
            if (p->dims[i] < 64 || p->dims[i] > 4096) return WSFFT_ERR_UNSUPPORTED;
    }
    const int old_layout = p->layout;
    const auto old_over = p->overrides;
    p->layout = layout;
    p->overrides.clear();
    const int rc = p->build_schedule();
    if (rc != WSFFT_SUCCESS) {
        p->layout = old_layout;
        p->overrides = old_over;
        p->build_schedule();
    }
    return rc;
}

int wsfft_execute(wsfft_plan plan, const void *in, void *out, wsfft_stream stream) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || p->ragged || !in || !out) return WSFFT_ERR_INVALID_ARG;
    if (((uintptr_t)in & 15) || ((uintptr_t)out & 15)) return WSFFT_ERR_INVALID_ARG;
    if (partial_overlap(in, out, (size_t)(p->batch * p->elems * elem_bytes(p->dtype)))) return WSFFT_ERR_INVALID_ARG;
    const int rc = p->run(in, out, (cudaStream_t)stream);
    p->mark_done((cudaStream_t)stream);
    return rc;
}

int wsfft_execute_host(wsfft_plan plan, const void *host_in, void *host_out, wsfft_stream stream) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || p->ragged || !host_in || !host_out) return WSFFT_ERR_INVALID_ARG;
    const size_t bytes = (size_t)(p->batch * p->elems * elem_bytes(p->dtype));
    if (partial_overlap(host_in, host_out, bytes)) return WSFFT_ERR_INVALID_ARG;
    if (!p->host_buf) {
        if (cudaMalloc(&p->host_buf, bytes) != cudaSuccess) {
            p->host_buf = nullptr;
            return WSFFT_ERR_ALLOC;
        }
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (p->can_pipeline_host()) {
        const int rc = p->run_host_pipelined(host_in, host_out, st);
        if (rc != WSFFT_SUCCESS) return rc;
        return cuda_status(cudaStreamSynchronize(st));
    }
    if (!p->passes.empty() && p->passes[0].kind == PASS_SLAB_A) {
        // The host pipeline overlaps the copies with the three one-launch
        // supersteps (the slab-local z and y hide behind the chunked
        // copies); the fused pass A would leave the copy back unoverlapped.
        // Use that schedule for this call, then restore the plan's own.
        const int mode = p->engine_mode;
        const auto over = p->overrides;
        p->engine_mode = 0;
        p->overrides.clear();
        int rc = p->build_schedule();
        const bool ok = rc == WSFFT_SUCCESS && p->can_pipeline_host();
        if (ok) rc = p->run_host_pipelined(host_in, host_out, st);
        p->engine_mode = mode;
        p->overrides = over;
        const int rc2 = p->build_schedule();
        if (ok) {
            if (rc != WSFFT_SUCCESS) return rc;
            if (rc2 != WSFFT_SUCCESS) return rc2;
            return cuda_status(cudaStreamSynchronize(st));
        }
        if (rc2 != WSFFT_SUCCESS) return rc2;
    }
    if (cudaMemcpyAsync(p->host_buf, host_in, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return WSFFT_ERR_CUDA;
    int rc = p->run(p->host_buf, p->host_buf, st);
    if (rc != WSFFT_SUCCESS) return rc;
    if (cudaMemcpyAsync(host_out, p->host_buf, bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return WSFFT_ERR_CUDA;
    return cuda_status(cudaStreamSynchronize(st));
}

int wsfft_destroy(wsfft_plan plan) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p) return WSFFT_SUCCESS;
    int prev = -1;
    const int dev = p->device;
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
    const int rc = p->wait_own_work();  // this plan's executes only, not the whole device
    delete p;
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
    return rc;
}

int wsfft_plan_set_pass_variant(wsfft_plan plan, int pass, int values_per_thread, int tile) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || pass < 0 || pass >= (int)p->passes.size() || values_per_thread < 0 || tile < 0)
        return WSFFT_ERR_INVALID_ARG;
    if (values_per_thread == 0 && tile == 0) {
        p->overrides.erase(pass);
        return p->build_schedule();
    }
    const PassSpec &ps = p->passes[pass];
    if (ps.kind != PASS_CONTIG && ps.kind != PASS_STRIDED) return WSFFT_ERR_UNSUPPORTED;
    // probe: is this shape instantiated?  (an empty launch returns before running)
    TileArgs a{};
    a.npencils = 0;
    PassSpec probe = ps;
    probe.E = values_per_thread;
    probe.tile = tile;
    if (launch(p->dtype, probe, nullptr, nullptr, a, 0) == cudaErrorInvalidValue)
        return WSFFT_ERR_UNSUPPORTED;
    p->overrides[pass] = std::make_pair(values_per_thread, tile);
    return p->build_schedule();
}

int wsfft_plan_set_engine(wsfft_plan plan, int mode) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || mode < 0 || mode > 4) return WSFFT_ERR_INVALID_ARG;
    if (p->ragged) return WSFFT_ERR_UNSUPPORTED;
    p->engine_mode = mode;
    return p->build_schedule();
}

int wsfft_plan_set_wait_test(wsfft_plan plan, int withhold, int64_t timeout_ns) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || timeout_ns <= 0) return WSFFT_ERR_INVALID_ARG;
    bool uses_engine = false;
    for (auto &ps : p->passes)
        uses_engine |= ps.kind == PASS_ENGINE_A || ps.kind == PASS_PERSIST_A || ps.kind == PASS_WP_A;
    if (!uses_engine) return WSFFT_ERR_UNSUPPORTED;
    p->withhold = withhold != 0;
    p->wait_timeout_ns = timeout_ns;
    return p->build_schedule();
}

int wsfft_plan_sync_status(wsfft_plan plan, wsfft_stream stream) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p) return WSFFT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int h = 0;
    if (cudaMemcpyAsync(&h, p->d_status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return WSFFT_ERR_CUDA;
    if (h != 0 && (cudaMemsetAsync(p->d_status, 0, sizeof(int), st) != cudaSuccess ||
                   cudaStreamSynchronize(st) != cudaSuccess))
        return WSFFT_ERR_CUDA;
    return h == 0 ? WSFFT_SUCCESS : WSFFT_ERR_DEVICE_TIMEOUT;
}

int wsfft_plan_passes(wsfft_plan plan, int *passes, int64_t *bytes) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p) return WSFFT_ERR_INVALID_ARG;
    const int np = p->ragged ? 3 : (int)p->passes.size();
    if (passes) *passes = np;
    if (bytes) *bytes = (int64_t)np * 2 * p->batch * p->elems * elem_bytes(p->dtype);
    return WSFFT_SUCCESS;
}

int wsfft_plan_profile(wsfft_plan plan, int capacity) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || capacity < 0) return WSFFT_ERR_INVALID_ARG;
    for (auto e : p->prof_ev) cudaEventDestroy(e);
    p->prof_ev.clear();
    p->prof_used = 0;
    for (int i = 0; i < 2 * capacity; ++i) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return WSFFT_ERR_CUDA;
        p->prof_ev.push_back(e);
    }
    return WSFFT_SUCCESS;
}

int wsfft_plan_launch_times(wsfft_plan plan, float *ms, int capacity, int *count) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || capacity < 0) return WSFFT_ERR_INVALID_ARG;
    const int n = p->prof_used;
    if (n > 0 && cudaEventSynchronize(p->prof_ev[2 * n - 1]) != cudaSuccess) return WSFFT_ERR_CUDA;
    for (int i = 0; i < n && ms && i < capacity; ++i) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, p->prof_ev[2 * i], p->prof_ev[2 * i + 1]) != cudaSuccess)
            return WSFFT_ERR_CUDA;
        ms[i] = t;
    }
    if (count) *count = n;
    p->prof_used = 0;
    return WSFFT_SUCCESS;
}

int wsfft_plan_create_ragged(wsfft_plan *plan, int count, const int64_t *dims, int dtype,
                             int direction) {
    if (!plan) return WSFFT_ERR_INVALID_ARG;
    *plan = nullptr;
    if (!dims || count < 1 || count > (1 << 20)) return WSFFT_ERR_INVALID_ARG;
    if (dtype != WSFFT_C32 && dtype != WSFFT_C16F && dtype != WSFFT_C16BF) return WSFFT_ERR_INVALID_ARG;
    if (direction != WSFFT_FORWARD && direction != WSFFT_INVERSE) return WSFFT_ERR_INVALID_ARG;
    for (int i = 0; i < 3 * count; ++i)
        if (!is_pow2(dims[i]) || dims[i] < 32 || dims[i] > 256) return WSFFT_ERR_INVALID_SIZE;
    Plan *p = new (std::nothrow) Plan();
    if (!p) return WSFFT_ERR_ALLOC;
    p->ragged = true;
    p->rag_grouped = dtype == WSFFT_C32;
    p->rag_count = count;
    p->dtype = dtype;
    p->dir = direction;
    p->norm = dtype == WSFFT_C32 ? WSFFT_NORM_PAPER : WSFFT_NORM_ORTHO;
    p->batch = 1;
    auto fail = [&](int rc) {
        delete p;
        return rc;
    };
    if (cudaGetDevice(&p->device) != cudaSuccess) return fail(WSFFT_ERR_CUDA);
    cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device);
    if (cudaMalloc(&p->d_status, sizeof(int)) != cudaSuccess) {
        p->d_status = nullptr;
        return fail(WSFFT_ERR_ALLOC);
    }
    if (p->zero(p->d_status, sizeof(int)) != WSFFT_SUCCESS) return fail(WSFFT_ERR_CUDA);
    p->rag_dims.assign(dims, dims + 3 * (size_t)count);
    p->elems = 0;
    for (int i = 0; i < count; ++i) p->elems += dims[3 * i] * dims[3 * i + 1] * dims[3 * i + 2];
    {
        const int rc = p->rag_build();
        if (rc != WSFFT_SUCCESS) return fail(rc);
    }
    if (cudaMalloc(&p->d_ctr, (size_t)(1 + 2 * count) * sizeof(uint32_t)) != cudaSuccess) {
        p->d_ctr = nullptr;
        return fail(WSFFT_ERR_ALLOC);
    }
    p->ctr_cap = 1 + 2 * count;
    if (cudaEventCreateWithFlags(&p->rag_copied, cudaEventDisableTiming) != cudaSuccess) {
        p->rag_copied = nullptr;
        return fail(WSFFT_ERR_CUDA);
    }
    int per_sm = 0;
    RagArgs dummy{};
    cudaError_t e = dtype == WSFFT_C32 ? launch_ragged_c32(dummy, &per_sm, 0, 0)
                    : dtype == WSFFT_C16F ? launch_ragged_c16f(dummy, &per_sm, 0, 0)
                                          : launch_ragged_c16bf(dummy, &per_sm, 0, 0);
    if (e != cudaSuccess || per_sm < 1) return fail(WSFFT_ERR_CUDA);
    p->rag_grid = per_sm * p->sm_count;
    autotune_apply_cached(*p);  // a remembered tile-shape choice and lag for this shape set, if any
    *plan = reinterpret_cast<wsfft_plan>(p);
    return WSFFT_SUCCESS;
}

int wsfft_plan_set_ragged_variant(wsfft_plan plan, int shape_select, int lag) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || shape_select < 0 || shape_select > 15 || lag < 1 || lag > 64) return WSFFT_ERR_INVALID_ARG;
    if (!p->ragged) return WSFFT_ERR_UNSUPPORTED;
    const int old_sel = p->rag_esel, old_lag = p->rag_lag;
    const bool old_grouped = p->rag_grouped;
    p->rag_esel = shape_select;
    p->rag_lag = lag;
    // a chosen queue variant is what runs; the values of a new plan choose what that runs
    p->rag_grouped = p->dtype == WSFFT_C32 && shape_select == 0 && lag == 1;
    const int rc = p->rag_build();
    if (rc != WSFFT_SUCCESS) {
        p->rag_esel = old_sel;
        p->rag_lag = old_lag;
        p->rag_grouped = old_grouped;
        p->rag_build();
    }
    return rc;
}

int wsfft_execute_ragged(wsfft_plan plan, const void *const *in, void *const *out,
                         wsfft_stream stream) {
    Plan *p = reinterpret_cast<Plan *>(plan);
    if (!p || !p->ragged || !in || !out) return WSFFT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    RagInst *h = static_cast<RagInst *>(p->rag_inst_host);
    bool changed = !p->rag_uploaded, in_place = false;
    for (int i = 0; i < p->rag_count; ++i) {
        in_place |= in[i] == out[i];
        if (!in[i] || !out[i] || ((uintptr_t)in[i] & 15) || ((uintptr_t)out[i] & 15)) return WSFFT_ERR_INVALID_ARG;
        changed |= h[i].in != in[i] || h[i].out != out[i];
    }
    if (changed) {
        // the previous upload may still be reading the pinned table
        if (p->rag_uploaded && cudaEventSynchronize(p->rag_copied) != cudaSuccess) return WSFFT_ERR_CUDA;
        for (int i = 0; i < p->rag_count; ++i) {
            h[i].in = in[i];
            h[i].out = out[i];
        }
        if (cudaMemcpyAsync(p->rag_inst, h, sizeof(RagInst) * (size_t)p->rag_count, cudaMemcpyHostToDevice, st) !=
            cudaSuccess)
            return WSFFT_ERR_CUDA;
        if (cudaEventRecord(p->rag_copied, st) != cudaSuccess) return WSFFT_ERR_CUDA;
        p->rag_uploaded = true;
    }
    if (p->rag_grouped && !in_place) {
        const int rc = p->rag_run_grouped(in, out, st);
        p->mark_done(st);
        return rc;
    }
    if (cudaMemsetAsync(p->d_ctr, 0, sizeof(uint32_t) * (size_t)(1 + 2 * p->rag_count), st) != cudaSuccess)
        return WSFFT_ERR_CUDA;
    RagArgs a{};
    a.items = static_cast<const RagItem *>(p->rag_items);
    a.nitems = p->rag_nitems;
    a.inst = static_cast<const RagInst *>(p->rag_inst);
    a.ctr = p->d_ctr;
    a.status = p->d_status;
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 2; ++j) a.tw[i][j] = p->rag_tw[i][j];
    a.esel = p->rag_esel;
    a.ci = p->dir == WSFFT_INVERSE ? -1.f : 1.f;
    a.co = a.ci;
    a.timeout_ns = (uint64_t)p->wait_timeout_ns;
    p->prof_begin(st);
    cudaError_t e = p->dtype == WSFFT_C32 ? launch_ragged_c32(a, nullptr, p->rag_grid, st)
                    : p->dtype == WSFFT_C16F ? launch_ragged_c16f(a, nullptr, p->rag_grid, st)
                                             : launch_ragged_c16bf(a, nullptr, p->rag_grid, st);
    p->prof_end(st);
    p->mark_done(st);
    return e == cudaSuccess ? WSFFT_SUCCESS : WSFFT_ERR_CUDA;
}


}  // extern "C"
