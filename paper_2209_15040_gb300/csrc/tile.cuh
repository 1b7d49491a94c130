// Pipelined supersteps over tiles of 2^13 or 2^14 elements.
//
// Persistent blocks transform one tile in registers while asynchronous copies
// bring the next tile's elements into shared memory, so the loads of tile
// i+1 run under the last stage and the stores of tile i.
//
// The TB bits of an element's index in the tile are its "slots".  In every
// stage a thread holds 64 elements: five slots index its registers (the
// digits the stage transforms, plus spare slots when they are shorter), one
// slot is the pair of elements that share packed FP32x2 instructions (cpair),
// and the others are the thread index.  A stage replaces a digit's slots
// by the digit of frequency with the same bits, so between stages only the
// roles of the slots change: an exchange writes each value to the
// shared-memory address of its slots and reads the values of the next
// stage's.  Addresses are linear in the bits, so each is one per-thread base
// plus a compile-time offset.
//
// Tiles of 2^13 elements: 128 threads, two blocks per SM in complex64, three
// in 16-bit storage.  The exchanges run through the load buffer, which takes
// the next tile once the last exchange has been read; the blocks of an SM
// are in different phases, so one's arithmetic runs under another's shared
// memory traffic.  Tiles of 2^14 elements (256 threads, one block per SM) are
// for axes whose rows would fall below 128 bytes otherwise: they have a load
// buffer of their own (128 KB in complex64), and real and imaginary parts
// pass through a 70 KB exchange buffer one after the other.
#pragma once

#include <type_traits>

#include "pass_kernels.cuh"
#include "ragged_desc.h"
#include "tile_desc.h"

namespace wsfft {

__device__ __forceinline__ void cp_async16(void *smem, const void *g) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(g) : "memory");
}
// until the grids before this one in the stream are complete
__device__ __forceinline__ void tile_grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A tile of a ragged launch and what its instance says, read from L2: a launch
// that does not wait at its start (TileArgs::late) must not meet an older line
// in L1.  The kernels read the next tile's a whole tile ahead: two dependent
// L2 reads in front of the copies and again of the stores cost 2%.
struct RagTile {
    const void *in;
    void *out;
    int64_t tile;
    int log_n2, log_n12, log_y0;
    float first, last;
};
template <class T>
__device__ __forceinline__ T *ldcg_ptr(T *const *p) {
    return reinterpret_cast<T *>(__ldcg(reinterpret_cast<const unsigned long long *>(p)));
}
__device__ __forceinline__ RagTile rag_tile(const TileArgs &a, int64_t t) {
    const int2 r = __ldcg(reinterpret_cast<const int2 *>(a.refs) + t);
    const RagInst *i = a.inst + r.x;
    return RagTile{ldcg_ptr(&i->in), ldcg_ptr(&i->out), r.y, __ldcg(&i->log_n2), __ldcg(&i->log_n12),
                   __ldcg(&i->log_y0), __ldcg(&i->first), __ldcg(&i->last)};
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Geometries: which slots each stage transforms.  A geometry G has
//   NST                stages
//   pair(s)            slot of the pair
//   in(s, j)           slot of register bit j (the digit first, then spares)
//   gbits(s)           bits of the digit
//   nsbits(s), kslot(s, i), twoff(s)  bits of the frequency so far (0: no
//                      twiddle), the slot of its bit i, and where the stage's
//                      twiddles start in the table
//   ls(slot), LBUF     load-buffer stride of a slot, elements of the buffer

// Slots of a tile of 2^NB points x 2^(TB-NB) pencils: pencil bits first, then
// the axis.  Two stages: the high R0 bits of the axis, then the low R1 bits.
template <int TBITS, int NB>
struct TileAxis {
    static_assert(NB >= 5 && NB <= 10, "two register stages");
    static constexpr int LW = TBITS - NB, W = 1 << LW, N = 1 << NB;
    static constexpr int R0 = NB >= 9 ? 5 : NB >= 7 ? 4 : 3, R1 = NB - R0;
    static constexpr int TB = TBITS;
    static constexpr int NST = 2;
    __host__ __device__ static constexpr int gbits(int s) { return s == 0 ? R0 : R1; }
    __host__ __device__ static constexpr int nsbits(int s) { return s == 0 ? 0 : R0; }
    __host__ __device__ static constexpr int kslot(int, int i) { return TBITS - R0 + i; }
    __host__ __device__ static constexpr int twoff(int) { return 0; }
    __host__ __device__ static constexpr int nlead(int) { return 0; }
    __host__ __device__ static constexpr int lead(int, int) { return -1; }
    __host__ __device__ static constexpr int in(int s, int j) {
        if (j < gbits(s)) return (s == 0 ? TBITS - R0 : LW) + j;
        // spares: the top pencil bits (a pencil's exchange then stays in fewer
        // threads); 512 points: the top frequency bit
        return NB <= 8 ? LW - 1 - (j - gbits(s)) : TBITS - 1;
    }
    static constexpr int TABLE = ((1 << R1) - 1) << R0;  // entries of the twiddle table
};

// The same for 2048 and 4096 points: three stages of four, four and the
// remaining bits.
template <int TBITS, int NB>
struct TileLongAxis {
    static_assert(NB == 11 || NB == 12, "three register stages");
    static constexpr int LW = TBITS - NB, W = 1 << LW, N = 1 << NB;
    static constexpr int R0 = 4, R1 = 4, R2 = NB - 8;
    static constexpr int TB = TBITS;
    static constexpr int NST = 3;
    __host__ __device__ static constexpr int gbits(int s) { return s == 2 ? R2 : 4; }
    __host__ __device__ static constexpr int nsbits(int s) { return 4 * s; }
    // k = k1 + 16 k2: k1 in the axis' top slots, k2 below them
    __host__ __device__ static constexpr int kslot(int, int i) { return i < 4 ? TBITS - 4 + i : TBITS - 12 + i; }
    __host__ __device__ static constexpr int twoff(int s) { return s == 2 ? 15 * 16 : 0; }
    __host__ __device__ static constexpr int nlead(int) { return 0; }
    __host__ __device__ static constexpr int lead(int, int) { return -1; }
    __host__ __device__ static constexpr int in(int s, int j) {
        if (j < gbits(s)) return (s == 0 ? TBITS - 4 : s == 1 ? TBITS - 8 : LW) + j;
        // spares: the slot below the first digit, then the top frequency bits
        return s == 0 ? TBITS - 5 : TBITS - 1 - (j - gbits(s));
    }
    static constexpr int TABLE = 15 * 16 + ((1 << R2) - 1) * 256;
};

// Strided axis: 2^LW adjacent pencils, rows of the tile copied whole.
template <int TBITS, int NB>
struct TileStrided : std::conditional_t<(NB > 10), TileLongAxis<TBITS, (NB > 10 ? NB : 11)>, TileAxis<TBITS, (NB > 10 ? 10 : NB)>> {
    static constexpr int LBUF = (1 << TBITS);
    __host__ __device__ static constexpr int pair(int) { return 0; }
    __host__ __device__ static constexpr int ls(int slot) { return 1 << slot; }
};

// Contiguous axis, transposed store: 2^LW whole pencils are copied, and leave
// as rows of 2^LW elements.  The first stage pairs neighbouring points, the
// second neighbouring pencils.  EB: bytes of a stored element.
template <int TBITS, int NB, int EB>
struct TileTrans : TileAxis<TBITS, NB> {
    using A = TileAxis<TBITS, NB>;
    static constexpr int LW = A::LW;
    // elements between pencils in the load buffer: 16 bytes more than the
    // pencil, so the first stage's lanes (pencils) spread over the banks
    static constexpr int PITCH = A::N + 16 / EB;
    static constexpr int LBUF = PITCH * A::W;
    __host__ __device__ static constexpr int pair(int s) { return s == 0 ? LW : 0; }
    __host__ __device__ static constexpr int ls(int slot) { return slot < LW ? PITCH << slot : 1 << (slot - LW); }
};

// Slot j of the thread index: the slots that are neither in a register nor
// the pair, lowest first -- after those the geometry puts in front (lead),
// where the lowest frequency bits of the last stage are not the lowest slots.
template <class G>
__host__ __device__ constexpr int tile_th(int s, int j) {
    int c = G::nlead(s);
    if (j < c) return G::lead(s, j);
    for (int slot = 0; slot < G::TB; ++slot) {
        bool used = slot == G::pair(s);
        for (int i = 0; i < 5; ++i) used |= G::in(s, i) == slot;
        for (int i = 0; i < G::nlead(s); ++i) used |= G::lead(s, i) == slot;
        if (used) continue;
        if (c == j) return slot;
        ++c;
    }
    return -1;
}

// Exchange layout after stage E: the stride (floats) of a slot.  Slots take
// positions (powers of two): the pair first where both stages have the same
// one (it moves as 8 bytes), the writing stage's lanes next - those that are
// also lanes of the reading stage first -, then the slots that are no lanes,
// and on top the reading stage's other lanes, `nr` of them.  A pad of
// 2^(5-nr) floats per step of the lowest of these gives them the banks of the
// writing stage's other lanes: writes and reads are free of bank conflicts.
template <class G>
__host__ __device__ constexpr int tile_xs(int e, int slot) {
    const bool vec = G::pair(e) == G::pair(e + 1);
    const int lanes = vec ? 4 : 5;  // lanes that share one pass of the banks
    int order[16] = {};
    bool placed[16] = {};
    int c = 0, nr = 0;
    if (vec) {
        order[c++] = G::pair(e);
        placed[G::pair(e)] = true;
    }
    for (int both = 1; both >= 0; --both)
        for (int j = 0; j < lanes; ++j) {
            const int t = tile_th<G>(e, j);
            bool in_r = false;
            for (int i = 0; i < lanes; ++i) in_r |= tile_th<G>(e + 1, i) == t;
            if (in_r == (both == 1)) {
                order[c++] = t;
                placed[t] = true;
            }
        }
    for (int j = 0; j < lanes; ++j) nr += placed[tile_th<G>(e + 1, j)] ? 0 : 1;
    for (int t = 0; t < G::TB; ++t) {
        bool r_lane = false;
        for (int j = 0; j < lanes; ++j) r_lane |= tile_th<G>(e + 1, j) == t;
        if (!placed[t] && !r_lane) order[c++] = t;
    }
    for (int j = 0; j < lanes; ++j)
        if (!placed[tile_th<G>(e + 1, j)]) order[c++] = tile_th<G>(e + 1, j);
    for (int i = 0; i < G::TB; ++i)
        if (order[i] == slot) return (1 << i) + (i >= G::TB - nr ? 1 << (i - (G::TB - nr) + 5 - nr) : 0);
    return -1;
}
template <class G>
__host__ __device__ constexpr int tile_xfloats() {
    int most = 0;
    for (int e = 0; e + 1 < G::NST; ++e) {
        int n = 1;
        for (int t = 0; t < G::TB; ++t) n += tile_xs<G>(e, t);
        most = n > most ? n : most;
    }
    return (most + 3) & ~3;
}

// Kinds of address: load buffer, exchange after stage E, slot number.
enum { TILE_OFF_LOAD = -2, TILE_OFF_SLOT = -1 };
template <class G, int KIND>
__host__ __device__ constexpr int tile_stride(int slot) {
    return KIND == TILE_OFF_LOAD ? G::ls(slot) : KIND == TILE_OFF_SLOT ? 1 << slot : tile_xs<G>(KIND, slot);
}
template <class G, int KIND, int SG, int J = 0>
__device__ __forceinline__ int tile_thread_off(int tid) {
    if constexpr (J == G::TB - 6) {
        return 0;
    } else {
        constexpr int st = tile_stride<G, KIND>(tile_th<G>(SG, J));
        return ((tid >> J) & 1) * st + tile_thread_off<G, KIND, SG, J + 1>(tid);
    }
}
template <class G, int KIND, int SG>
__host__ __device__ constexpr int tile_reg_off(int r) {
    int o = 0;
    for (int j = 0; j < 5; ++j)
        if ((r >> j) & 1) o += tile_stride<G, KIND>(G::in(SG, j));
    return o;
}
// frequency so far that a set of slots holds
template <class G, int SG>
__host__ __device__ constexpr int tile_k_of(int slots) {
    int k = 0;
    for (int i = 0; i < G::nsbits(SG); ++i) k |= ((slots >> G::kslot(SG, i)) & 1) << i;
    return k;
}

// Read one part (real or imaginary) of a stage's values, or write it.
template <class G, int E, int SG, bool IM, bool WRITE, int R = 0>
__device__ __forceinline__ void tile_part(cpair (&v)[32], float *x) {
    if constexpr (R < 32) {
        constexpr int PS = tile_xs<G>(E, G::pair(SG));
        constexpr int off = tile_reg_off<G, E, SG>(R);
        float2 &p = IM ? v[R].im : v[R].re;
        if constexpr (PS == 1) {
            if constexpr (WRITE) *reinterpret_cast<float2 *>(x + off) = p;
            else p = *reinterpret_cast<const float2 *>(x + off);
        } else if constexpr (WRITE) {
            x[off] = p.x;
            x[off + PS] = p.y;
        } else {
            p.x = x[off];
            p.y = x[off + PS];
        }
        tile_part<G, E, SG, IM, WRITE, R + 1>(v, x);
    }
}
// Exchange between stages E and E+1.  FULL: room for both parts at once (one
// barrier); otherwise they take turns in one buffer.
template <class G, int E, bool FULL>
__device__ __forceinline__ void tile_exchange(cpair (&v)[32], float *xw, float *xr) {
    constexpr int IM = FULL ? tile_xfloats<G>() : 0;
    if constexpr (E > 0) __syncthreads();  // the previous exchange has been read
    tile_part<G, E, E, false, true>(v, xw);
    if constexpr (FULL) tile_part<G, E, E, true, true>(v, xw + IM);
    __syncthreads();
    tile_part<G, E, E + 1, false, false>(v, xr);
    if constexpr (!FULL) {
        __syncthreads();
        tile_part<G, E, E, true, true>(v, xw);
        __syncthreads();
    }
    tile_part<G, E, E + 1, true, false>(v, xr + IM);
}

// Product of two split pairs of complex numbers, lane by lane.
__device__ __forceinline__ cpair cmul(cpair a, cpair w) {
    return {__ffma2_rn(a.re, w.re, f2neg(__fmul2_rn(a.im, w.im))), __ffma2_rn(a.re, w.im, __fmul2_rn(a.im, w.re))};
}
__device__ __forceinline__ cpair ld_cpair(const float4 *p) {
    const float4 t = *p;
    return {make_float2(t.x, t.y), make_float2(t.z, t.w)};
}

// A stage: the digit's twiddles and its DFT.  The twiddles multiply all
// values before the first butterfly (interleaved with the butterflies the
// compiler's schedule was 10% slower).
template <class G, int SG, bool LDG>
__device__ __forceinline__ void tile_stage(cpair (&v)[32], const float2 *__restrict__ tw, int slots) {
    constexpr int B = G::gbits(SG), R = 1 << B, NSB = G::nsbits(SG);
    if constexpr (NSB > 0) {
        const float2 *tk = tw + G::twoff(SG) + tile_k_of<G, SG>(slots);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int r = i & (R - 1);
            if (r == 0) continue;
            const float2 *p = tk + (((r - 1) << NSB) + tile_k_of<G, SG>(tile_reg_off<G, TILE_OFF_SLOT, SG>(i)));
            v[i] = cmul(v[i], LDG ? __ldg(p) : *p);
        }
    }
#pragma unroll
    for (int i = 0; i < 32; i += R) {
        cpair g[R];
#pragma unroll
        for (int r = 0; r < R; ++r) g[r] = v[i + r];
        dft_fused<R>(g);
#pragma unroll
        for (int r = 0; r < R; ++r) v[i + r] = g[r];
    }
}

// Shared memory: load buffer, exchange buffer (the same bytes in tiles of
// 2^13 elements), then (16-bit storage) the stage twiddles, then (inter-step
// twiddle) one table per digit of k, for two tiles.
template <class G, class S, int MODE>
struct TileSmem {
    static constexpr bool TWID = MODE == TILE_STRIDED_TWID;
    static constexpr int CTAS = G::TB == 14 ? 1 : sizeof(S) == 4 && !TWID ? 3 : 2;  // blocks per SM
    static constexpr bool SHARED_BUF = G::TB < 14;
    // both parts of an exchange at once where there is room (16-bit tiles of
    // 2^14: 2-4% faster)
    static constexpr bool FULL = SHARED_BUF || (sizeof(S) == 4 && !TWID);
    static constexpr int LOAD = G::LBUF * (int)sizeof(S), XCHG = tile_xfloats<G>() * (FULL ? 8 : 4);
    static constexpr int X = SHARED_BUF ? 0 : LOAD;
    static constexpr int TW = SHARED_BUF ? (LOAD > XCHG ? LOAD : XCHG) : LOAD + XCHG;
    // 16-bit storage reads its stage twiddles 5% faster from shared memory;
    // complex64 was slower so
    static constexpr bool SHARED_TW = sizeof(S) == 4;
    static constexpr int C = TW + (SHARED_TW ? G::TABLE * 8 : 0);
    static constexpr int TILE_C = TWID ? G::W * (8 << G::R0) : 0, TILE_U = TWID ? G::W * (8 << G::R1) : 0;
    static constexpr int BYTES = C + 2 * (TILE_C + TILE_U);
    static_assert(BYTES <= 228 * 1024 / CTAS - 1024, "blocks per SM");
};

// Superstep along a strided axis.  What bounds it and what it gives, 2^27
// elements, against the one-tile-per-block kernels of pass_kernels.cuh:
//   complex64, 1024 points, 16 pencils (tiles of 2^14): the memory system, on
//     128-byte rows (the same copies and stores without arithmetic take as
//     long); 0.343 ms against 0.410 (8 pencils, 64-byte rows) and 0.49-0.51
//     (16 pencils, one block per SM without the copies in flight) at a stride
//     of 2^10, 0.39 against 0.46-0.50 at 2^17;
//   16-bit storage: latencies of the FP32 pipe, shared memory and the copies (each
//     unit 45-56% busy), which the blocks of an SM overlap in part: 512 points
//     0.20 ms (tiles of 2^13), 0.227 (2^14) against 0.26-0.27; 256 points 0.187 and
//     0.205 against 0.24-0.25.
// With the four-step's inter-step twiddle w_L^(q k) on the store (pencil q,
// k = k1 + Ns r): the product of w_L^(q k1) and w_(L/Ns)^(q r), whose tables
// hold every q for the few values of k1 and of r, so a tile copies its own
// columns of both beside its elements and a pair reads them as one 16-byte
// value (gathered element by element instead: 40% slower).  complex64 1024
// points 0.344 ms against 0.41-0.53, 16-bit 512 points 0.246 against 0.55.
// Transposed store of a contiguous axis (the four-step's second superstep and
// the other spectral layouts): complex64 1024 points 0.389 ms against 0.45-
// 0.51, 16-bit 512 points 0.214 against 0.305.
template <class G, class S, int MODE>
__global__ void __launch_bounds__(1 << (G::TB - 6), TileSmem<G, S, MODE>::CTAS)
    tile_axis_kernel(const S *__restrict__ in, S *__restrict__ out, TileArgs a) {
    using SM = TileSmem<G, S, MODE>;
    using PT = typename SplitPair<S>::T;
    constexpr int NT = 1 << (G::TB - 6);
    constexpr bool LDG = !SM::SHARED_TW;
    extern __shared__ float4 t_smem[];
    char *sm = reinterpret_cast<char *>(t_smem);
    float *xb = reinterpret_cast<float *>(sm + SM::X);
    const int tid = threadIdx.x;
    const float2 *tw = a.tw;
    if constexpr (SM::SHARED_TW) {
        // a plan's table: no kernel writes it
        float2 *st = reinterpret_cast<float2 *>(sm + SM::TW);
        for (int i = tid; i < G::TABLE; i += NT) st[i] = a.tw[i];
        tw = st;
    }
    if (MODE != TILE_STRIDED_RAG || !a.late) tile_grid_wait();
    const int64_t ntiles = a.tiles;

    // first element of a tile in `in`
    auto tile_base = [&](int64_t t) -> int64_t {
        const int64_t q = (a.reverse ? ntiles - 1 - t : t) * G::W;
        if constexpr (MODE == TILE_TRANS) return q * G::N;
        else return ((q >> a.log_inner) * ((int64_t)G::N << a.log_inner)) + (q & (a.inner - 1));
    };
    constexpr int EPC = 16 / (int)sizeof(S);  // elements per 16-byte chunk
    RagTile rag{}, rag_next{};  // the tile in hand, the one after it
    auto issue = [&](int64_t tile, int half) {
        int64_t base, inner = a.inner;
        const S *from = in;
        if constexpr (MODE == TILE_STRIDED_RAG) {
            from = static_cast<const S *>(rag_next.out);  // the first trip's output
            base = rag_next.tile * G::W;
            inner = (int64_t)1 << rag_next.log_n12;
        } else {
            base = tile_base(tile);
        }
        if constexpr (MODE == TILE_TRANS) {
            constexpr int CPP = G::N / EPC;  // chunks per pencil
#pragma unroll
            for (int c = tid; c < CPP * G::W; c += NT)
                cp_async16(sm + (c / CPP) * (G::PITCH * (int)sizeof(S)) + (c % CPP) * 16, in + base + (int64_t)c * EPC);
        } else {
            constexpr int CPR = G::W / EPC, ROWS = NT / CPR;  // chunks per row, rows per round
            static_assert(CPR <= NT && G::N % ROWS == 0, "whole rounds");
            const S *p = from + base + (int64_t)(tid / CPR) * inner + (tid % CPR) * EPC;
            const int64_t step = (int64_t)ROWS * inner;
#pragma unroll
            for (int j = 0; j < G::N / ROWS; ++j) {
                cp_async16(sm + (tid + j * NT) * 16, p);
                p += step;
            }
        }
        if constexpr (MODE == TILE_STRIDED_TWID) {
            constexpr int CW = G::W / 2, TR = NT / CW, Ns = 1 << G::R0, R = 1 << G::R1;  // pairs per row, rows per round
            const int qp = ((int)(base & (a.inner - 1)) >> 1) + tid % CW, row = tid / CW;
            const int half_inner = (int)(a.inner >> 1);
            const float4 *tc = reinterpret_cast<const float4 *>(a.tw_hi) + qp;
            const float4 *tu = reinterpret_cast<const float4 *>(a.tw_lo) + qp;
            char *cu = sm + SM::C + half * (SM::TILE_C + SM::TILE_U) + tid * 16;
#pragma unroll
            for (int i = 0; i < Ns; i += TR)
                if (Ns >= TR || row < Ns) cp_async16(cu + i * CW * 16, tc + (row + i) * half_inner);
#pragma unroll
            for (int i = 0; i < R; i += TR)
                if (R >= TR || row < R) cp_async16(cu + SM::TILE_C + i * CW * 16, tu + (row + i) * half_inner);
        }
    };
    // start the copies of the tile after `tile`
    auto next = [&](int64_t tile, int half) {
        if (tile + gridDim.x < ntiles) issue(tile + gridDim.x, half ^ 1);
        else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        cp_async_commit();
    };
    constexpr int LAST = G::NST - 1;
    const S *lbuf = reinterpret_cast<const S *>(sm) + tile_thread_off<G, TILE_OFF_LOAD, 0>(tid);
    float *xw = xb + tile_thread_off<G, 0, 0>(tid), *xr = xb + tile_thread_off<G, 0, 1>(tid);
    float *xw1 = xb, *xr1 = xb;
    if constexpr (LAST == 2) {
        xw1 += tile_thread_off<G, 1, 1>(tid);
        xr1 += tile_thread_off<G, 1, 2>(tid);
    }
    const int slots1 = tile_thread_off<G, TILE_OFF_SLOT, 1>(tid), slots = tile_thread_off<G, TILE_OFF_SLOT, LAST>(tid);
    const int wcol = slots & (G::W - 1), k1 = tile_k_of<G, LAST>(slots);

    int half = 0;
    int64_t tile = blockIdx.x;
    if constexpr (MODE == TILE_STRIDED_RAG)
        if (tile < ntiles) rag_next = rag_tile(a, tile);
    if (tile < ntiles) issue(tile, 0);
    cp_async_commit();
    for (; tile < ntiles; tile += gridDim.x) {
        cpair v[32];
        if constexpr (MODE == TILE_STRIDED_RAG) {
            rag = rag_next;
            if (tile + gridDim.x < ntiles) rag_next = rag_tile(a, tile + gridDim.x);
        }
        cp_async_wait_all();
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 32; ++r) {
            const S *p = lbuf + tile_reg_off<G, TILE_OFF_LOAD, 0>(r);
            static_assert(G::ls(G::pair(0)) == 1, "a pair is two neighbours in the load buffer");
            v[r] = SplitPair<S>::load(reinterpret_cast<const PT *>(p));
            v[r].im = __fmul2_rn(v[r].im, f2dup(a.conj_in));
        }
        __syncthreads();
        if constexpr (!SM::SHARED_BUF) next(tile, half);
        tile_stage<G, 0, LDG>(v, tw, 0);
        tile_exchange<G, 0, SM::FULL>(v, xw, xr);
        if constexpr (LAST == 2) {
            tile_stage<G, 1, LDG>(v, tw, slots1);
            tile_exchange<G, 1, SM::FULL>(v, xw1, xr1);
        }
        if constexpr (SM::SHARED_BUF) {
            __syncthreads();
            next(tile, half);
        }
        tile_stage<G, LAST, LDG>(v, tw, slots);
        // row k = k1 + Ns r: the last digit r in the registers
        constexpr int Ns = 1 << G::nsbits(LAST), R = 1 << G::gbits(LAST);
        int64_t ob, ostride = MODE == TILE_TRANS ? a.trans_rows : a.inner;
        S *o = out;
        float sx = a.sx, sy = a.sy;
        if constexpr (MODE == TILE_STRIDED_RAG) {
            ob = rag.tile * G::W;
            ostride = (int64_t)1 << rag.log_n12;
            o = static_cast<S *>(rag.out);
            sx *= rag.last;
            sy *= rag.last;
        } else {
            ob = tile_base(tile);
        }
        if constexpr (MODE == TILE_TRANS) {
            // rows per transform are a multiple of W: a tile's rows share one
            const int64_t q0 = ob / G::N, b = q0 / a.trans_rows;
            ob = b * G::N * a.trans_rows + (q0 - b * a.trans_rows);
        }
        o += ob + (int64_t)k1 * ostride + wcol;
        const int64_t step = (int64_t)Ns * ostride;
#pragma unroll
        for (int i = 0; i < 32; i += R) {
            const int sp = tile_reg_off<G, TILE_OFF_SLOT, LAST>(i);
            const int kc = tile_k_of<G, LAST>(sp), wc = sp & (G::W - 1);
            S *p = o + (int64_t)kc * ostride + wc;
            const float4 *cu =
                reinterpret_cast<const float4 *>(sm + SM::C + half * (SM::TILE_C + SM::TILE_U)) + (wcol + wc) / 2;
            cpair c;
            if constexpr (MODE == TILE_STRIDED_TWID) c = ld_cpair(cu + (k1 + kc) * (G::W / 2));
#pragma unroll
            for (int r = 0; r < R; ++r) {
                cpair z = v[i + r];
                if constexpr (MODE == TILE_STRIDED_TWID)
                    z = cmul(z, cmul(c, ld_cpair(cu + SM::TILE_C / 16 + r * (G::W / 2))));
                z.re = __fmul2_rn(z.re, f2dup(sx));
                z.im = __fmul2_rn(z.im, f2dup(sy));
                SplitPair<S>::store(reinterpret_cast<PT *>(p), z);
                p += step;
            }
        }
        half ^= 1;
    }
    if (MODE == TILE_STRIDED_RAG && a.late) tile_grid_wait();
}

}  // namespace wsfft
