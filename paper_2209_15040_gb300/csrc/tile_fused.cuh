// Fused supersteps on the pipelined tiles (tile.cuh): two axes, or one and a
// part of another, per trip through memory.
//
//  * tile_slab_kernel: n1 x n2 slabs (the two inner axes), whole ones in a
//    tile of 2^13 elements, or every (n1/R)-th row of a larger slab: R rows
//    of n2 elements, transformed along n2 and, as the first R-point digit of
//    the middle axis, across the rows.  Row y = y1 Y0 + y0 (Y0 = n1/R) goes in
//    for a fixed y0, frequency k1 comes out at row R y0 + k1: a tile stores
//    2^13 consecutive elements.
//  * tile_outer_kernel: the rest of a split middle axis (Y0 points, with the
//    twiddle w_n1^(y0 k1)) and the outer axis (n0 points), for a fixed k1 and a
//    run of adjacent columns.  It reads rows R y0 + k1 and writes rows k1 + R
//    k0, the same ones: in place.
//
// So the two inner axes of a rank-3 transform take one trip where n1 n2 <=
// 2^13, and a whole one of up to 2^22 elements takes two instead of three
// (n1 n2 = 2^13 Y0 and Y0 n0 <= 2^9 leave tiles with rows of at least 16
// elements).
#pragma once

#include "ragged_desc.h"
#include "tile.cuh"

namespace wsfft {

// ---------------------------------------------------------------------------
// Geometries with several digits per stage:
//   ngroups(s), gbits(s, g)   digits of a stage and their bits
//   nsbits(s, g), kslot(s, g, i)   frequency so far on the digit's axis, its slots
//   tbl(s, g), twoff(s, g)    the twiddle table and where the stage's start in it

// 2^YB rows of 2^ZB contiguous elements, transformed along both; spare slots
// above are further such slabs.  Three stages: the high five bits of y; the
// high four bits of z; the low bits of both.  The last stage's lanes run over
// the four bits of the first z frequency digit: 128-byte rows (complex64).
template <int TBITS, int ZB, int YB>
struct TileSlab {
    static_assert(ZB >= 5 && YB >= 5 && ZB + YB <= TBITS, "slab bits");
    static constexpr int C2 = ZB - 4, YL = YB - 5;  // low bits of z and y
    static_assert(C2 + YL <= 5, "three register stages");
    static constexpr int TB = TBITS;
    static constexpr int NST = 3;
    static constexpr int LBUF = (1 << TBITS);
    __host__ __device__ static constexpr int pair(int s) { return s == 2 ? C2 : 0; }
    __host__ __device__ static constexpr int ls(int slot) { return 1 << slot; }
    __host__ __device__ static constexpr int chunk_at(int c, int) { return c * 16; }
    __host__ __device__ static constexpr int ngroups(int s) { return s == 2 && YL > 0 ? 2 : 1; }
    __host__ __device__ static constexpr int gbits(int s, int g) { return s == 0 ? 5 : s == 1 ? 4 : g == 0 ? C2 : YL; }
    __host__ __device__ static constexpr int in(int s, int j) {
        if (s == 0) return ZB + YL + j;
        if (s == 1) return j < 4 ? C2 + j : TBITS - 1;
        if (j < C2) return j;
        if (j < C2 + YL) return ZB + j - C2;
        return TBITS - 1 - (j - C2 - YL);
    }
    __host__ __device__ static constexpr int nsbits(int s, int g) { return s < 2 ? 0 : g == 0 ? 4 : 5; }
    __host__ __device__ static constexpr int kslot(int, int g, int i) { return (g == 0 ? C2 : ZB + YL) + i; }
    __host__ __device__ static constexpr int tbl(int, int g) { return g; }
    __host__ __device__ static constexpr int twoff(int, int) { return 0; }
    __host__ __device__ static constexpr int nlead(int) { return 0; }
    __host__ __device__ static constexpr int lead(int, int) { return -1; }
    static constexpr int TABLE0 = ((1 << C2) - 1) << 4, TABLE1 = ((1 << YL) - 1) << 5;
    // where a slot's frequencies leave: z = kz1 + 16 kz2, y = ky1 + 32 ky2
    __host__ __device__ static constexpr int place(int s) {
        const int kz = ((s >> C2) & 15) | ((s & ((1 << C2) - 1)) << 4);
        const int y = s >> ZB;
        const int ky = ((y >> YL) & 31) | ((y & ((1 << YL) - 1)) << 5);
        return kz + (ky << ZB) + ((y >> YB) << (ZB + YB));
    }
};

// Contiguous axis of 2^NB points, whole pencils: the high R0 bits, then the
// low R1 bits.  The last stage's pair is the lowest frequency bit and its lanes
// run over the rest of the first digit: whole runs of a pencil per access.
template <int TBITS, int NB>
struct TileContig {
    static_assert(NB >= 5 && NB <= 8, "two register stages");
    static constexpr int R0 = NB >= 7 ? 4 : 3, R1 = NB - R0;
    static constexpr int TB = TBITS;
    static constexpr int NST = 2;
    // elements between pencils in the load buffer: the first stage's lanes
    // (2^R1 neighbours, then pencils) spread over the banks
    static constexpr int PITCH = (1 << NB) + (1 << R1);
    static constexpr int LBUF = PITCH << (TBITS - NB);
    __host__ __device__ static constexpr int pair(int s) { return s == 0 ? 0 : R1; }
    __host__ __device__ static constexpr int ls(int slot) { return slot < NB ? 1 << slot : PITCH << (slot - NB); }
    // byte in the load buffer of the tile's 16-byte chunk c
    __host__ __device__ static constexpr int chunk_at(int c, int eb) {
        const int per = (1 << NB) * eb / 16;
        return (c / per) * (PITCH * eb) + (c % per) * 16;
    }
    __host__ __device__ static constexpr int ngroups(int) { return 1; }
    __host__ __device__ static constexpr int gbits(int s, int) { return s == 0 ? R0 : R1; }
    __host__ __device__ static constexpr int in(int s, int j) {
        const int b = s == 0 ? R0 : R1;
        return j < b ? (s == 0 ? R1 : 0) + j : TBITS - 1 - (j - b);  // spares: the top pencil bits
    }
    __host__ __device__ static constexpr int nsbits(int s, int) { return s == 0 ? 0 : R0; }
    __host__ __device__ static constexpr int kslot(int, int, int i) { return R1 + i; }
    __host__ __device__ static constexpr int tbl(int, int) { return 0; }
    __host__ __device__ static constexpr int twoff(int, int) { return 0; }
    __host__ __device__ static constexpr int nlead(int) { return 0; }
    __host__ __device__ static constexpr int lead(int, int) { return -1; }
    static constexpr int TABLE0 = ((1 << R1) - 1) << R0, TABLE1 = 0;
    __host__ __device__ static constexpr int place(int s) {
        return ((s >> R1) & ((1 << R0) - 1)) + ((s & ((1 << R1) - 1)) << R0) + ((s >> NB) << NB);
    }
};

// The outer axis (2^XB points) and the low Y0B bits of the middle one, whose
// high bits a TileSlab pass has transformed: 2^LW adjacent elements per row.
template <int TBITS, int XBITS, int Y0B>
struct TileOuter {
    static constexpr int LW = TBITS - XBITS - Y0B, W = 1 << LW, XB = XBITS, YB = Y0B;
    static constexpr int XH = 5 - Y0B, XL = XB - XH;  // first and second digit of x
    static_assert(LW >= 4 && Y0B >= 1 && XH >= 1 && XL >= 1 && XL <= 5, "two register stages");
    static constexpr int TB = TBITS;
    static constexpr int NST = 2;
    static constexpr int LBUF = (1 << TBITS);
    __host__ __device__ static constexpr int pair(int) { return 0; }
    __host__ __device__ static constexpr int ls(int slot) { return 1 << slot; }
    __host__ __device__ static constexpr int ngroups(int s) { return s == 0 ? 2 : 1; }
    __host__ __device__ static constexpr int gbits(int s, int g) { return s == 0 ? (g == 0 ? XH : Y0B) : XL; }
    __host__ __device__ static constexpr int in(int s, int j) {
        if (s == 0) return LW + XL + j;  // x high bits, then the y bits above them
        return j < XL ? LW + j : TBITS - 1 - (j - XL);
    }
    __host__ __device__ static constexpr int nsbits(int s, int) { return s == 0 ? 0 : XH; }
    __host__ __device__ static constexpr int kslot(int, int, int i) { return LW + XL + i; }
    __host__ __device__ static constexpr int tbl(int, int) { return 0; }
    __host__ __device__ static constexpr int twoff(int, int) { return 0; }
    __host__ __device__ static constexpr int nlead(int) { return 0; }
    __host__ __device__ static constexpr int lead(int, int) { return -1; }
    static constexpr int TABLE0 = ((1 << XL) - 1) << XH, TABLE1 = 0;
};

// 2^(TB-ZB) rows of 2^ZB contiguous elements (512..4096), transformed along
// the row and, in one digit, across the rows.  Three stages: the high ZA bits
// of z and the rows; the next five bits of z; the low ZC bits.
template <int TBITS, int ZB>
struct TileWide {
    static constexpr int RB = TBITS - ZB, ZA = 5 - RB, ZC = TBITS - 10;
    static_assert(RB >= 1 && RB <= 4 && ZA + 5 + ZC == ZB, "three register stages");
    static constexpr int TB = TBITS;
    static constexpr int NST = 3;
    static constexpr int LBUF = (1 << TBITS);
    __host__ __device__ static constexpr int pair(int s) { return s == 2 ? ZB - ZA : 0; }
    __host__ __device__ static constexpr int ls(int slot) { return 1 << slot; }
    __host__ __device__ static constexpr int ngroups(int s) { return s == 0 ? 2 : 1; }
    __host__ __device__ static constexpr int gbits(int s, int g) { return s == 0 ? (g == 0 ? ZA : RB) : s == 1 ? 5 : ZC; }
    __host__ __device__ static constexpr int in(int s, int j) {
        if (s == 0) return TBITS - 5 + j;
        if (s == 1) return ZC + j;
        if (j < ZC) return j;
        return j - ZC < RB ? TBITS - 1 - (j - ZC) : ZC + 4 - (j - ZC - RB);  // spares: rows, then z's second digit
    }
    __host__ __device__ static constexpr int nsbits(int s, int) { return s == 0 ? 0 : s == 1 ? ZA : ZA + 5; }
    // kz = k1 + 2^ZA k2 (+ 2^(ZA+5) k3)
    __host__ __device__ static constexpr int kslot(int, int, int i) { return i < ZA ? ZB - ZA + i : ZC + i - ZA; }
    __host__ __device__ static constexpr int tbl(int, int) { return 0; }
    __host__ __device__ static constexpr int twoff(int s, int) { return s == 2 ? 31 << ZA : 0; }
    // the store's lanes: the rest of k1, then k2
    __host__ __device__ static constexpr int nlead(int s) { return s == 2 ? ZA - 1 : 0; }
    __host__ __device__ static constexpr int lead(int, int i) { return ZB - ZA + 1 + i; }
    static constexpr int TABLE0 = (31 << ZA) + (((1 << ZC) - 1) << (ZA + 5)), TABLE1 = 0;
};

// frequency so far on a group's axis that a set of slots holds
template <class G, int SG, int GR>
__host__ __device__ constexpr int tile_gk_of(int slots) {
    int k = 0;
    for (int i = 0; i < G::nsbits(SG, GR); ++i) k |= ((slots >> G::kslot(SG, GR, i)) & 1) << i;
    return k;
}

// The first register bit of a group.
template <class G>
__host__ __device__ constexpr int tile_group_lo(int s, int g) {
    int lo = 0;
    for (int i = 0; i < g; ++i) lo += G::gbits(s, i);
    return lo;
}
// One digit: its twiddles and its DFT.  The twiddles multiply all values
// before the first butterfly (interleaved with the butterflies the compiler's
// schedule was 10% slower).
template <class G, int SG, int GR, bool LDG>
__device__ __forceinline__ void tile_group(cpair (&v)[32], const float2 *__restrict__ tw, int slots) {
    constexpr int LO = tile_group_lo<G>(SG, GR), B = G::gbits(SG, GR), R = 1 << B, NSB = G::nsbits(SG, GR);
    if constexpr (NSB > 0) {
        const float2 *tk = tw + G::twoff(SG, GR) + tile_gk_of<G, SG, GR>(slots);
        // the pair may be the lowest bit of k: two neighbouring twiddles
        constexpr bool two = G::kslot(SG, GR, 0) == G::pair(SG);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int r = (i >> LO) & (R - 1);
            if (r == 0) continue;
            const float2 *p = tk + (((r - 1) << NSB) + tile_gk_of<G, SG, GR>(tile_reg_off<G, TILE_OFF_SLOT, SG>(i)));
            if constexpr (two) {
                const float4 w = LDG ? __ldg(reinterpret_cast<const float4 *>(p)) : *reinterpret_cast<const float4 *>(p);
                v[i] = cmul(v[i], cpair{make_float2(w.x, w.z), make_float2(w.y, w.w)});
            } else {
                v[i] = cmul(v[i], LDG ? __ldg(p) : *p);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if ((i >> LO) & (R - 1)) continue;
        cpair g[R];
#pragma unroll
        for (int r = 0; r < R; ++r) g[r] = v[i + (r << LO)];
        dft_fused<R>(g);
#pragma unroll
        for (int r = 0; r < R; ++r) v[i + (r << LO)] = g[r];
    }
}
template <class G, int SG, bool LDG>
__device__ __forceinline__ void tile_gstage(cpair (&v)[32], const float2 *tw0, const float2 *tw1, int slots) {
    tile_group<G, SG, 0, LDG>(v, G::tbl(SG, 0) ? tw1 : tw0, slots);
    if constexpr (G::ngroups(SG) > 1) tile_group<G, SG, 1, LDG>(v, G::tbl(SG, 1) ? tw1 : tw0, slots);
}

// Shared memory: load buffer, exchange buffer (the same bytes in tiles of
// 2^13 elements), then (16-bit storage, tables of up to 8 KB) the stage
// twiddles.
template <class G, class S>
struct TileFusedSmem {
    static constexpr int CTAS = G::TB == 14 ? 1 : sizeof(S) == 4 ? 3 : 2;  // blocks per SM
    static constexpr bool SHARED_BUF = G::TB < 14, FULL = SHARED_BUF || sizeof(S) == 4;
    static constexpr int LOAD = G::LBUF * (int)sizeof(S), XCHG = tile_xfloats<G>() * (FULL ? 8 : 4);
    static constexpr bool SHARED_TW = sizeof(S) == 4 && G::TABLE0 + G::TABLE1 <= 1024;
    static constexpr int X = SHARED_BUF ? 0 : LOAD;
    static constexpr int TW = SHARED_BUF ? (LOAD > XCHG ? LOAD : XCHG) : LOAD + XCHG;
    static constexpr int BYTES = TW + (SHARED_TW ? (G::TABLE0 + G::TABLE1) * 8 : 0);
    static_assert(BYTES <= 228 * 1024 / CTAS - 1024, "blocks per SM");
};

// The stage tables a kernel reads: in shared memory for 16-bit storage.
template <class G, class S>
__device__ __forceinline__ void tile_tables(char *sm, const TileArgs &a, const float2 *&tw0, const float2 *&tw1) {
    using SM = TileFusedSmem<G, S>;
    tw0 = a.tw;
    tw1 = a.tw2;
    if constexpr (SM::SHARED_TW) {
        // a plan's tables: no kernel writes them
        float2 *st = reinterpret_cast<float2 *>(sm + SM::TW);
        for (int i = threadIdx.x; i < G::TABLE0; i += blockDim.x) st[i] = a.tw[i];
        for (int i = threadIdx.x; i < G::TABLE1; i += blockDim.x) st[G::TABLE0 + i] = a.tw2[i];
        tw0 = st;
        tw1 = st + G::TABLE0;
    }
}
// Values of the first stage from the load buffer.
template <class G, class S>
__device__ __forceinline__ void tile_load(cpair (&v)[32], const S *lbuf, float ci) {
    static_assert(G::ls(G::pair(0)) == 1, "a pair is two neighbours in the load buffer");
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const S *p = lbuf + tile_reg_off<G, TILE_OFF_LOAD, 0>(r);
        v[r] = SplitPair<S>::load(reinterpret_cast<const typename SplitPair<S>::T *>(p));
        v[r].im = __fmul2_rn(v[r].im, f2dup(ci));
    }
}
template <class S>
__device__ __forceinline__ void tile_store(S *p, cpair z, float sx, float sy) {
    z.re = __fmul2_rn(z.re, f2dup(sx));
    z.im = __fmul2_rn(z.im, f2dup(sy));
    SplitPair<S>::store(reinterpret_cast<typename SplitPair<S>::T *>(p), z);
}

// 2^27 elements, read and write: complex64 0.330-0.345 ms, 0.92-0.96 of the copy
// rate (the two supersteps it replaces 0.60-0.67); 16-bit storage 0.235-0.27 ms
// (0.36-0.56).  What bounds it: latencies that 8 warps per SM (12 in 16-bit storage)
// cover in part; in complex64 memory is the busiest unit (67% of the DRAM peak
// from cold caches, SM 35%), in 16-bit storage the FMA and shared-memory pipes (52% and 57%).  Two
// blocks per SM (three in 16-bit storage) of 2^13 elements rather than one of
// 2^14: three stages in one block leave FP32 pipe and shared memory idle in
// turn (0.43-0.48 ms).
// Contiguous pencils alone (TileContig): 16-bit storage 32 / 64 / 128 points
// 0.197 / 0.192 / 0.194 ms against 0.341 / 0.234 / 0.263.
// WHOLE: tiles of whole slabs (or pencils) of 2^(ZB+YB) < 2^13 elements (the last tile may
// be partial); otherwise the rows of one residue class of a slab of 2^13
// << a.log_y0 elements.
template <class G, class S, bool WHOLE, bool RAG = false>
__global__ void __launch_bounds__(1 << (G::TB - 6), TileFusedSmem<G, S>::CTAS)
    tile_slab_kernel(const S *__restrict__ in, S *__restrict__ out, TileArgs a) {
    using SM = TileFusedSmem<G, S>;
    constexpr int NT = 1 << (G::TB - 6), ELEMS = 1 << G::TB;
    constexpr int EPC = 16 / (int)sizeof(S), CHUNKS = ELEMS / EPC;  // elements per 16-byte chunk, chunks per tile
    constexpr bool LDG = !SM::SHARED_TW;
    constexpr int LAST = G::NST - 1;
    extern __shared__ float4 t_smem[];
    char *sm = reinterpret_cast<char *>(t_smem);
    float *xb = reinterpret_cast<float *>(sm);
    const int tid = threadIdx.x;
    const float2 *tw0, *tw1;
    tile_tables<G, S>(sm, a, tw0, tw1);
    if (!RAG || !a.late) tile_grid_wait();
    const int64_t ntiles = a.tiles;

    RagTile rag{}, rag_next{};  // the tile in hand, the one after it
    auto issue = [&](int64_t t) {
        int64_t tile = t;
        const S *from = in;
        int log_y0 = a.log_y0;
        if constexpr (RAG) {
            tile = rag_next.tile;
            from = static_cast<const S *>(rag_next.in);
            log_y0 = rag_next.log_y0;
        }
        if constexpr (WHOLE) {
            const int64_t base = tile << G::TB, left = RAG ? ELEMS : a.elems - base;
            const S *src = from + base + tid * EPC;
            if (left >= ELEMS) {
#pragma unroll
                for (int j = 0; j < CHUNKS / NT; ++j)
                    cp_async16(sm + G::chunk_at(tid + j * NT, (int)sizeof(S)), src + j * NT * EPC);
            } else {
#pragma unroll 1
                for (int j = 0; j < CHUNKS / NT; ++j)
                    if ((tid + j * NT) * EPC < left)
                        cp_async16(sm + G::chunk_at(tid + j * NT, (int)sizeof(S)), src + j * NT * EPC);
            }
        } else {
            // slab tile >> log_y0, rows y0, y0 + Y0, ...
            constexpr int CPR = (1 << (G::C2 + 4)) / EPC, ROWS = NT / CPR;  // chunks per row, rows per round
            static_assert(CPR <= NT, "whole rounds");
            constexpr int64_t row = 1 << (G::C2 + 4);
            const int64_t rs = row << log_y0;
            const S *p = from + ((tile >> log_y0) << (G::TB + log_y0)) + (tile & ((1 << log_y0) - 1)) * row +
                         (int64_t)(tid / CPR) * rs + (tid % CPR) * EPC;
            const int64_t step = (int64_t)ROWS * rs;
#pragma unroll
            for (int j = 0; j < CHUNKS / NT; ++j) {
                cp_async16(sm + (tid + j * NT) * 16, p);
                p += step;
            }
        }
    };
    const S *lbuf = reinterpret_cast<const S *>(sm) + tile_thread_off<G, TILE_OFF_LOAD, 0>(tid);
    float *xw0 = xb + tile_thread_off<G, 0, 0>(tid), *xr0 = xb + tile_thread_off<G, 0, 1>(tid);
    float *xw1 = xb, *xr1 = xb;
    if constexpr (LAST == 2) {
        xw1 += tile_thread_off<G, 1, 1>(tid);
        xr1 += tile_thread_off<G, 1, 2>(tid);
    }
    const int slots1 = tile_thread_off<G, TILE_OFF_SLOT, 1>(tid), slots2 = tile_thread_off<G, TILE_OFF_SLOT, LAST>(tid);
    const int to = G::place(slots2);

    int64_t tile = blockIdx.x;
    if constexpr (RAG)
        if (tile < ntiles) rag_next = rag_tile(a, tile);
    if (tile < ntiles) issue(tile);
    cp_async_commit();
    // Where every block has one tile and an SM to itself, the next launch may come in
    // now and not only with the last stage: its ramp (about 1.5 us) was a fifth of a
    // small call.  Back to back, us, with one launch per axis in brackets: complex64
    // 64^3 8.7 -> 7.6 (8.0), eight of 8 x 128 x 64 9.6 -> 7.8 (7.3), 64 x 128 x 128 11.7 -> 10.8
    // (15.1); 16-bit storage 64^3 8.5 -> 7.1 (7.7), 64 x 256 x 32 10.4 -> 7.4 (8.0).  With more
    // tiles the next launch's blocks get in the way: 256 tiles of 128^3 in 16-bit
    // storage 12.9 -> 14.9; complex64 before the general strided kernel 128 tiles of 128 x
    // 128 x 64 11.0 -> 13.1, 80 of 32 x 64 x 64 8.9 -> 10.1, and 16 take 3-6% longer.
    if constexpr (!RAG)
        if (sizeof(S) == 4 || a.log_y0 > 0 ? ntiles <= 128 : ntiles >= 32 && ntiles <= 64)
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (; tile < ntiles; tile += gridDim.x) {
        cpair v[32];
        if constexpr (RAG) {
            rag = rag_next;
            if (tile + gridDim.x < ntiles) rag_next = rag_tile(a, tile + gridDim.x);
        }
        cp_async_wait_all();
        __syncthreads();
        tile_load<G, S>(v, lbuf, a.conj_in);
        __syncthreads();
        tile_gstage<G, 0, LDG>(v, tw0, tw1, 0);
        tile_exchange<G, 0, true>(v, xw0, xr0);
        if constexpr (LAST == 2) {
            tile_gstage<G, 1, LDG>(v, tw0, tw1, slots1);
            tile_exchange<G, 1, true>(v, xw1, xr1);
        }
        __syncthreads();
        if (tile + gridDim.x < ntiles) issue(tile + gridDim.x);
        else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        cp_async_commit();
        tile_gstage<G, LAST, LDG>(v, tw0, tw1, slots2);
        int64_t base = tile << G::TB;
        S *o = out;
        float sx = a.sx, sy = a.sy;
        if constexpr (RAG) {
            base = rag.tile << G::TB;
            o = static_cast<S *>(rag.out);
            sx = sy = rag.first;
        }
        o += base + to;
        int lim = ELEMS;
        if constexpr (WHOLE && !RAG)
            if (a.elems - base < ELEMS) lim = (int)(a.elems - base) - to;
#pragma unroll
        for (int r = 0; r < 32; ++r) {
            const int at = G::place(tile_reg_off<G, TILE_OFF_SLOT, LAST>(r));
            if (!WHOLE || RAG || at < lim) tile_store(o + at, v[r], sx, sy);
        }
    }
    if (RAG && a.late) tile_grid_wait();
}

// Bound like the strided tiles (0.35-0.36 ms per 2^27 elements in complex64,
// 0.19-0.21 in 16-bit storage); whole transforms of 32 MiB in L2 by the latency of
// their copies (long-scoreboard stalls 3.7 cycles per instruction).
template <class G, class S, bool RAG = false>
__global__ void __launch_bounds__(1 << (G::TB - 6), TileFusedSmem<G, S>::CTAS)
    tile_outer_kernel(const S *__restrict__ in, S *__restrict__ out, TileArgs a) {
    using SM = TileFusedSmem<G, S>;
    constexpr int NT = 1 << (G::TB - 6);
    constexpr bool LDG = !SM::SHARED_TW;
    extern __shared__ float4 t_smem[];
    char *sm = reinterpret_cast<char *>(t_smem);
    float *xb = reinterpret_cast<float *>(sm);
    const int tid = threadIdx.x;
    const float2 *tw0, *tw1;
    tile_tables<G, S>(sm, a, tw0, tw1);
    if (!RAG || !a.late) tile_grid_wait();
    const int64_t ntiles = a.tiles;

    // columns (k1, z) of a transform: 2^log_cols of them, W per tile
    auto tile_base = [&](int64_t t) -> int64_t {
        const int64_t tile = a.reverse ? ntiles - 1 - t : t;
        const int lp = a.log_cols - G::LW;
        return ((tile >> lp) << a.log_transform) + ((tile & (((int64_t)1 << lp) - 1)) << G::LW);
    };
    RagTile rag{}, rag_next{};  // the tile in hand, the one after it
    auto issue = [&](int64_t t) {
        const S *from = in;
        int64_t base, inner = a.inner;
        if constexpr (RAG) {
            from = static_cast<const S *>(rag_next.out);  // the first trip's output
            base = rag_next.tile << G::LW;
            inner = (int64_t)1 << rag_next.log_n12;
        } else {
            base = tile_base(t);
        }
        // rows of W elements: the n0 rows of a y0, then the next y0
        constexpr int EPC = 16 / (int)sizeof(S), CPR = G::W / EPC, ROWS = NT / CPR, XR = 1 << G::XB;
        static_assert(CPR <= NT && XR % ROWS == 0, "whole rounds");
        const S *src = from + base + (int64_t)(tid / CPR) * inner + (tid % CPR) * EPC;
        const int64_t step = (int64_t)ROWS * inner;
#pragma unroll
        for (int y = 0; y < (1 << G::YB); ++y) {
            const S *p = src + y * a.ystep;
#pragma unroll
            for (int j = 0; j < XR / ROWS; ++j) {
                cp_async16(sm + (tid + (y * (XR / ROWS) + j) * NT) * 16, p);
                p += step;
            }
        }
    };
    const S *lbuf = reinterpret_cast<const S *>(sm) + tile_thread_off<G, TILE_OFF_LOAD, 0>(tid);
    float *xw = xb + tile_thread_off<G, 0, 0>(tid), *xr = xb + tile_thread_off<G, 0, 1>(tid);
    const int slots = tile_thread_off<G, TILE_OFF_SLOT, 1>(tid);
    // x = kx1 + 2^XH kx2, y row k1 + R k0
    constexpr int XS = G::LW + G::XL, XM = (1 << G::XH) - 1, R = 1 << G::XL;

    int64_t tile = blockIdx.x;
    if constexpr (RAG)
        if (tile < ntiles) rag_next = rag_tile(a, tile);
    if (tile < ntiles) issue(tile);
    cp_async_commit();
    // as in tile_slab_kernel
    if constexpr (!RAG)
        if (ntiles <= 128) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (; tile < ntiles; tile += gridDim.x) {
        cpair v[32];
        if constexpr (RAG) {
            rag = rag_next;
            if (tile + gridDim.x < ntiles) rag_next = rag_tile(a, tile + gridDim.x);
        }
        int64_t base, inner = a.inner;
        int log_row = a.log_row, nk1 = a.nk1;
        const float2 *wy = a.tw_hi;
        S *o = out;
        float sx = a.sx, sy = a.sy;
        if constexpr (RAG) {
            base = rag.tile << G::LW;
            inner = (int64_t)1 << rag.log_n12;
            log_row = rag.log_n2;
            nk1 = 1 << (G::TB - log_row);
            wy = log_row == 5 ? a.cls[0] : log_row == 6 ? a.cls[1] : log_row == 7 ? a.cls[2] : a.cls[3];
            o = static_cast<S *>(rag.out);
            sx *= rag.last;
            sy *= rag.last;
        } else {
            base = tile_base(tile);
        }
        cp_async_wait_all();
        __syncthreads();
        tile_load<G, S>(v, lbuf, a.conj_in);
        __syncthreads();
        const int k1 = (int)(base >> log_row) & (nk1 - 1);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int y = i >> G::XH;
            if (y > 0) v[i] = cmul(v[i], __ldg(wy + (y - 1) * nk1 + k1));
        }
        tile_gstage<G, 0, LDG>(v, tw0, tw1, 0);
        tile_exchange<G, 0, true>(v, xw, xr);
        __syncthreads();
        if (tile + gridDim.x < ntiles) issue(tile + gridDim.x);
        else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        cp_async_commit();
        tile_gstage<G, 1, LDG>(v, tw0, tw1, slots);
        o += base + (int64_t)((slots >> XS) & XM) * inner + (slots >> (G::TB - G::YB)) * a.ystep + (slots & (G::W - 1));
        const int64_t step = inner << G::XH;
#pragma unroll
        for (int i = 0; i < 32; i += R) {
            const int sp = tile_reg_off<G, TILE_OFF_SLOT, 1>(i);
            S *p = o + (int64_t)((sp >> XS) & XM) * inner + (sp >> (G::TB - G::YB)) * a.ystep;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                tile_store(p, v[i + r], sx, sy);
                p += step;
            }
        }
    }
    if (RAG && a.late) tile_grid_wait();
}

// One digit of a strided axis of n points (element stride a.inner, a multiple
// of the row) beside the last axis: tile (o, y0, j) takes rows y1 Y0 + y0
// (Y0 = n/2^RB, j: which row of the axis' stride), and frequency k1 leaves,
// times w_n^(y0 k1), at R y0 + k1.  What is left of the axis is a strided
// superstep of Y0 points at R times the stride.  Bound by the latency of
// three stages over 13 bits (complex64 0.36-0.37 ms per 2^27 elements, 0.85 of the
// copy rate; 16-bit storage 0.285-0.295; DRAM 67%, shared memory 51%, FMA 40% busy); with
// 4096-point rows and a radix of 4, tiles of 2^14 elements, one block per SM: 0.485
// and 0.37 (DRAM 43%).
template <class G, class S>
__global__ void __launch_bounds__(1 << (G::TB - 6), TileFusedSmem<G, S>::CTAS)
    tile_wide_kernel(const S *__restrict__ in, S *__restrict__ out, TileArgs a) {
    using SM = TileFusedSmem<G, S>;
    constexpr int NT = 1 << (G::TB - 6), ZB = G::TB - G::RB;
    constexpr bool LDG = !SM::SHARED_TW;
    extern __shared__ float4 t_smem[];
    char *sm = reinterpret_cast<char *>(t_smem);
    float *xb = reinterpret_cast<float *>(sm + SM::X);
    const int tid = threadIdx.x;
    const float2 *tw0, *tw1;
    tile_tables<G, S>(sm, a, tw0, tw1);
    tile_grid_wait();
    const int64_t ntiles = a.tiles;

    const int log_m = a.log_inner - ZB;  // rows within the axis' stride
    auto y0_of = [&](int64_t tile) { return (tile >> log_m) & (((int64_t)1 << a.log_y0) - 1); };
    // first element of (o, y0 << shift, j)
    auto tile_base = [&](int64_t tile, int shift) -> int64_t {
        const int64_t o = tile >> (log_m + a.log_y0), j = tile & (((int64_t)1 << log_m) - 1);
        return (((o << (a.log_y0 + G::RB)) + (y0_of(tile) << shift)) << a.log_inner) + (j << ZB);
    };
    auto issue = [&](int64_t tile) {
        constexpr int EPC = 16 / (int)sizeof(S), PER = (1 << ZB) / EPC / NT;  // rounds per row
        static_assert(PER >= 1, "a row takes whole rounds");
        const S *src = in + tile_base(tile, 0) + tid * EPC;
        const int64_t rs = a.inner << a.log_y0;
#pragma unroll
        for (int y = 0; y < (1 << G::RB); ++y) {
#pragma unroll
            for (int j = 0; j < PER; ++j) cp_async16(sm + (tid + (y * PER + j) * NT) * 16, src + j * NT * EPC);
            src += rs;
        }
    };
    auto next = [&](int64_t tile) {
        if (tile + gridDim.x < ntiles) issue(tile + gridDim.x);
        else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        cp_async_commit();
    };
    const S *lbuf = reinterpret_cast<const S *>(sm) + tile_thread_off<G, TILE_OFF_LOAD, 0>(tid);
    float *xw0 = xb + tile_thread_off<G, 0, 0>(tid), *xr0 = xb + tile_thread_off<G, 0, 1>(tid);
    float *xw1 = xb + tile_thread_off<G, 1, 1>(tid), *xr1 = xb + tile_thread_off<G, 1, 2>(tid);
    const int slots1 = tile_thread_off<G, TILE_OFF_SLOT, 1>(tid), slots2 = tile_thread_off<G, TILE_OFF_SLOT, 2>(tid);
    // frequency along the row; the digit's sits in the slots above
    auto kz = [](int s) constexpr -> int {
        const int k1 = (s >> (ZB - G::ZA)) & ((1 << G::ZA) - 1), k2 = (s >> G::ZC) & 31, k3 = s & ((1 << G::ZC) - 1);
        return k1 + (k2 << G::ZA) + (k3 << (G::ZA + 5));
    };
    const int64_t to = (int64_t)(slots2 >> ZB) * a.inner + kz(slots2);

    int64_t tile = blockIdx.x;
    if (tile < ntiles) issue(tile);
    cp_async_commit();
    for (; tile < ntiles; tile += gridDim.x) {
        cpair v[32];
        cp_async_wait_all();
        __syncthreads();
        tile_load<G, S>(v, lbuf, a.conj_in);
        __syncthreads();
        if constexpr (!SM::SHARED_BUF) next(tile);
        tile_gstage<G, 0, LDG>(v, tw0, tw1, 0);
        const float2 *wy = a.tw_hi + y0_of(tile);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int k = i >> G::ZA;
            if (k > 0) v[i] = cmul(v[i], __ldg(wy + ((int64_t)(k - 1) << a.log_y0)));
        }
        tile_exchange<G, 0, SM::FULL>(v, xw0, xr0);
        tile_gstage<G, 1, LDG>(v, tw0, tw1, slots1);
        tile_exchange<G, 1, SM::FULL>(v, xw1, xr1);
        if constexpr (SM::SHARED_BUF) {
            __syncthreads();
            next(tile);
        }
        tile_gstage<G, 2, LDG>(v, tw0, tw1, slots2);
        S *o = out + tile_base(tile, G::RB) + to;
#pragma unroll
        for (int r = 0; r < 32; ++r) {
            const int sp = tile_reg_off<G, TILE_OFF_SLOT, 2>(r);
            tile_store(o + (int64_t)(sp >> ZB) * a.inner + kz(sp), v[r], a.sx, a.sy);
        }
    }
}

}  // namespace wsfft
