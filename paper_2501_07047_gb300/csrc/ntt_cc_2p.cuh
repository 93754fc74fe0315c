// CUDA-core NTT / INTT in two launches through L2 (path a, the two-pass schedule).
//
// The radix-2 Cooley-Tukey forward transform (App. A; the same butterflies, twiddles and lazy
// ranges as ntt_cc_impl.cuh) of N = 2^LOGN, LOGN = 14 .. 17, is cut at stage A = LOGN - 10, the
// row / column factorisation of the matrix NTT (MAT, Sec. IV-B) with the twiddle step folded
// into the butterflies' own twiddles:
//  - strided pass, stages 0 .. A-1: a thread runs radix-2^A sub-transforms over the elements
//    j + 1024 k of one to four consecutive positions j in registers, 64 or 32 elements in all
//    (where 2^A is twice that, two warps share the positions and exchange halves once through
//    shared memory).  Whole 128-byte lines; the 2^A - 1 twiddles are the row's first ones;
//  - block pass, stages A .. LOGN-1: a warp owns a block of 1024 consecutive elements, 32 per
//    lane: a radix-32 sub-transform over the elements lane + 32 k, an exchange in the warp's own
//    4 KiB of shared memory, one over 32 consecutive elements, and a second exchange so that the
//    results leave as whole lines.  No CTA barrier: a CTA is one warp.
// The inverse (Gentleman-Sande) runs the same passes in the other order.  The intermediate goes
// through the output buffer, which stays in the 129 MB L2 between the launches up to about 64 MiB.
//
// What bounds it (192 rows of 2^16, 48 MiB): the strided pass is at HBM speed (18.4 us alone, 16.8
// with the butterflies left out, 6 TB/s); the block pass takes 21 to 25 us of which 13 are the
// multiply pipe's: L2 and shared-memory latency with 20 warps an SM, and more warps (64
// registers) or fewer change nothing.  In all 39.6 us forward and 39.4 inverse, against 43.1 and
// 49.0 on the cluster schedule at the outset and 49.7 and 45.1 for the 8 + 8 split it replaces
// (columns of 64-byte pieces, 64-byte-strided block stores: 48 us of its 50 were data movement).
// Distributed shared memory is what the cluster kernel pays for instead: its cross-CTA step moves
// 44 MB at about 3 TB/s, 15 us (31.6 us without butterflies, 17.0 with the exchange kept inside
// the CTA), where an L2 read runs at 18 TB/s.  Parts of it, forward / inverse: CTAs of one warp
// in the block pass instead of four 40.5 / 41.1 -> 39.6 / 40.9; the inverse's first 24 twiddles
// requested with the data, before the first exchange, 40.9 -> 39.4 (and 52.8 -> 50.3 with a
// Hadamard product).  Tried: both passes in one launch by tickets and flags (41.4 / 42.6 us); the
// polynomials of one limb side by side to share twiddles in L1 (42.4 / 48.5).
#pragma once
#include "ntt_cc_impl.cuh"

namespace hefx {
namespace cc2 {

using cc::KRows;
using cc::fwd_first;
using cc::inv_offset;
using cc::inv_sum;
using cc::reduce_out;
using cc::row_had;
using cc::row_in;
using cc::row_lc;
using cc::row_out;
using cc::row_twf;
using cc::row_twi;
using cc::twmul;

constexpr int LOGB = 10, BLOCK = 1 << LOGB;  // elements of a block

constexpr int SM_WARPS = 20;                 // warps an SM that the register budget is sized for (96 registers)

// Twiddles g, g + 1 of a stage (base in shared memory, 16-byte aligned for even g).
__device__ __forceinline__ void tw_pair(uint2 (&w)[2], const uint2* base) {
    const uint4 t = *reinterpret_cast<const uint4*>(base);
    w[0] = make_uint2(t.x, t.y);
    w[1] = make_uint2(t.z, t.w);
}

// Forward stages S0 .. S0+R-1 of sub-transform h (of 2^S0) on its elements x, twiddles from shared memory.
template <int S0, int R, int LOGN, int F>
__device__ __forceinline__ void fwd_strided(uint32_t (&x)[1 << R], int h, const uint2* tws, const LimbConst& lc) {
    const uint32_t two_q = lc.q2;
#pragma unroll
    for (int v = 0; v < R; ++v) {
        const int half = 1 << (R - 1 - v);
        const uint2* base = tws + (1 << (S0 + v)) + (h << v);
        uint2 w[2];
        w[0] = w[1] = v == 0 ? *base : make_uint2(0, 0);
#pragma unroll
        for (int b = 0; b < (1 << (R - 1)); ++b) {
            const int g = b >> (R - 1 - v);
            const int k = (g << (R - v)) + (b & (half - 1));
            if (v > 0 && (g & 1) == 0 && (b & (half - 1)) == 0) tw_pair(w, base + g);
            const uint32_t xa = fwd_first<LOGN, F>(x[k], S0 + v, lc);
            const uint32_t t = twmul<F>(x[k + half], w[g & 1], lc);
            x[k] = xa + t;
            x[k + half] = xa - t + two_q;
        }
    }
}

// The inverse's last A stages but the very last S0 (0 or 1) likewise; N^-1 (SCALE 1) or N^-1 2^32 (2)
// goes into the transform's last stage, inv_last.
template <int SCALE, int F>
__device__ __forceinline__ void inv_last(uint32_t& X, uint32_t& Y, uint32_t cq, const LimbConst& lc) {
    const uint32_t s = SCALE == 1 ? lc.ninv : lc.ninvR, ssh = SCALE == 1 ? lc.ninv_sh : lc.ninvR_sh;
    const uint32_t w = SCALE == 1 ? lc.ninvw : lc.ninvRw, wsh = SCALE == 1 ? lc.ninvw_sh : lc.ninvRw_sh;
    const uint32_t a = X + Y, b = X - Y + cq;
    X = csub(mul_shoup_lazy(a, s, ssh, lc.q), lc.q);
    Y = csub(mul_shoup_lazy(b, w, wsh, lc.q), lc.q);
}
template <int S0, int R, int LOGN, int SCALE, int F>
__device__ __forceinline__ void inv_strided(uint32_t (&x)[1 << R], int h, const uint2* tws, const LimbConst& lc) {
    constexpr int A = R + S0;
#pragma unroll
    for (int v = 0; v < R; ++v) {
        const int d = 1 << v;
        if (v == A - 1) {
#pragma unroll
            for (int k = 0; k < (1 << (R - 1)); ++k) inv_last<SCALE, F>(x[k], x[k + d], inv_offset<F>(lc, v, k), lc);
            continue;
        }
        const uint2* base = tws + (1 << (A - 1 - v)) + (h << (R - 1 - v));
        uint2 w[2];
        w[0] = w[1] = v == R - 1 ? *base : make_uint2(0, 0);
#pragma unroll
        for (int b = 0; b < (1 << (R - 1)); ++b) {
            const int g = b >> v;
            const int k = (g << (v + 1)) + (b & (d - 1));
            if (v < R - 1 && (g & 1) == 0 && (b & (d - 1)) == 0) tw_pair(w, base + g);
            const uint32_t X = x[k], Y = x[k + d];
            x[k] = inv_sum<A, F>(X + Y, v, k, lc);
            x[k + d] = twmul<F>(X - Y + inv_offset<F>(lc, v, k), w[g & 1], lc);
        }
    }
}

// Stages s0 .. s0+4 of a block's elements lane + 32 k: every lane of the warp has the same twiddles
// (2^s + blk 2^v + g), read in pairs.
template <int LOGN, int s0, int F>
__device__ __forceinline__ void fwd_uniform(uint32_t (&x)[32], uint32_t blk, const uint2* tw, const LimbConst& lc) {
    const uint32_t two_q = lc.q2;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        const int half = 1 << (4 - v);
        const uint2* base = tw + (1u << (s0 + v)) + (blk << v);
        uint2 w[2];
        w[0] = w[1] = v == 0 ? __ldg(base) : make_uint2(0, 0);
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const int g = b >> (4 - v);
            const int k = (g << (5 - v)) + (b & (half - 1));
            if (v > 0 && (g & 1) == 0 && (b & (half - 1)) == 0) {
                const uint4 t = __ldg(reinterpret_cast<const uint4*>(base + g));
                w[0] = make_uint2(t.x, t.y);
                w[1] = make_uint2(t.z, t.w);
            }
            const uint32_t xa = fwd_first<LOGN, F>(x[k], s0 + v, lc);
            const uint32_t t = twmul<F>(x[k + half], w[g & 1], lc);
            x[k] = xa + t;
            x[k + half] = xa - t + two_q;
        }
    }
}
template <int LOGN, int e0, int F>
__device__ __forceinline__ void inv_uniform(uint32_t (&x)[32], uint32_t blk, const uint2* tw, const LimbConst& lc) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        const int h = 1 << v;
        const uint2* base = tw + ((1u << LOGN) >> (e0 + v + 1)) + (blk << (4 - v));
        uint2 w[2];
        w[0] = w[1] = v == 4 ? __ldg(base) : make_uint2(0, 0);
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const int g = b >> v;
            const int k = (g << (v + 1)) + (b & (h - 1));
            if (v < 4 && (g & 1) == 0 && (b & (h - 1)) == 0) {
                const uint4 t = __ldg(reinterpret_cast<const uint4*>(base + g));
                w[0] = make_uint2(t.x, t.y);
                w[1] = make_uint2(t.z, t.w);
            }
            const uint32_t X = x[k], Y = x[k + h];
            x[k] = inv_sum<5, F>(X + Y, v, k, lc);
            x[k + h] = twmul<F>(X - Y + inv_offset<F>(lc, v, k), w[g & 1], lc);
        }
    }
}

// Strided-pass task of a CTA of 64 threads.  SPLIT 0: positions (part * 64 + thread) * V .. of one row, the
// 2^A elements of each of its V positions in a thread.  SPLIT 1: position part * 32 + lane, whose
// 2^A elements the two warps share, half each: the stage between the halves runs on k, k + 2^(A-1)
// of one quarter, then the warps exchange 2^(A-2) elements through shared memory and run the rest
// on their own half (the inverse: in the other order).  SMALL: half the elements per thread.
constexpr int THREADS = 64;
template <int LOGN, int SMALL>
struct Strided {
    static constexpr int A = LOGN - LOGB;
    static constexpr int LOGE = SMALL ? 5 : 6;                // elements per thread
    static constexpr int SPLIT = A > LOGE ? A - LOGE : 0;
    static constexpr int R = A - SPLIT;
    static constexpr int V = 1 << (LOGE - R);                 // positions per thread
    static constexpr int POS = (THREADS >> SPLIT) * V;        // positions per CTA
    static constexpr int PARTS = BLOCK / POS;                 // tasks of a row
    static_assert(SPLIT <= 1 && V <= 4, "one, two or four positions per thread, two threads per position at most");
};

template <int V>
struct Vec;
template <>
struct Vec<1> { typedef uint32_t T; };
template <>
struct Vec<2> { typedef uint2 T; };
template <>
struct Vec<4> { typedef uint4 T; };
__device__ __forceinline__ void unpack(uint32_t v, uint32_t (&x)[1]) { x[0] = v; }
__device__ __forceinline__ void unpack(uint2 v, uint32_t (&x)[2]) { x[0] = v.x, x[1] = v.y; }
__device__ __forceinline__ void unpack(uint4 v, uint32_t (&x)[4]) { x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w; }
__device__ __forceinline__ uint32_t pack(const uint32_t (&x)[1]) { return x[0]; }
__device__ __forceinline__ uint2 pack(const uint32_t (&x)[2]) { return make_uint2(x[0], x[1]); }
__device__ __forceinline__ uint4 pack(const uint32_t (&x)[4]) { return make_uint4(x[0], x[1], x[2], x[3]); }

// Forward in -> out (RS: rescaling on the way in), inverse in place in out.
template <int LOGN, int MODE, int F, int SMALL>
__device__ __forceinline__ void strided_task(uint2* tws, uint32_t* swap, uint32_t row, uint32_t part, const KRows& a) {
    typedef Strided<LOGN, SMALL> S;
    constexpr int N = 1 << LOGN, A = S::A, V = S::V, R = S::R, E = 1 << R, RA = 1 << A;
    constexpr bool INV = MODE == MODE_INV || MODE == MODE_HAD_INV, RS = MODE == MODE_RS_FWD;
    constexpr int SCALE = MODE == MODE_INV ? 1 : 2;
    typedef typename Vec<V>::T T;
    const uint2* tw = INV ? row_twi<N, F>(a, row) : row_twf<N, F>(a, row);
    for (int i = threadIdx.x; i < RA; i += THREADS) tws[i] = __ldg(tw + i);
    const int h = S::SPLIT ? threadIdx.x >> 5 : 0;
    const uint32_t j = S::SPLIT ? part * 32 + (threadIdx.x & 31) : (part * THREADS + threadIdx.x) * V;
    const LimbConst& lc = row_lc<F>(a, row);
    // x[c][i] is element pos(i): all of a position's 2^A, or the quarters h and h + 2
    const uint32_t base = j + (S::SPLIT ? h * (E / 2) * BLOCK : 0);
    auto pos = [](int i) { return (i + (S::SPLIT && i >= E / 2 ? E / 2 : 0)) * BLOCK; };
    uint32_t* out = row_out<N, F>(a, row) + base;
    uint32_t x[V][E];
    const uint32_t* in = out;
    if constexpr (!INV && !RS) in = row_in<N, F>(a, row) + base;
    if constexpr (RS) in = a.in + ((size_t)(row / a.L) * a.in_rows + row % a.L) * N + base;  // (b, limb) of [B][in_rows]
    // the inverse runs on its own half first: elements h E + i
    const uint32_t* src = S::SPLIT && INV ? in + h * (E / 2) * BLOCK : in;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        uint32_t t[V];
        unpack(__ldcg(reinterpret_cast<const T*>(src + (INV ? i * BLOCK : pos(i)))), t);
#pragma unroll
        for (int c = 0; c < V; ++c) x[c][i] = t[c];
    }
    if constexpr (RS) {
        const uint32_t* last = a.in + ((size_t)(row / a.L) * a.in_rows + a.in_rows - 1) * N + base;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            uint32_t t[V];
            unpack(__ldcg(reinterpret_cast<const T*>(last + pos(i))), t);
#pragma unroll
            for (int c = 0; c < V; ++c) x[c][i] = cc::rescale_one(x[c][i], t[c], lc);
        }
    }
    __syncthreads();
    // warp 0's upper quarter for warp 1's lower one, both ways round
    auto exchange = [&]() {
        uint32_t* mine = swap + threadIdx.x;
        const uint32_t* other = swap + (threadIdx.x ^ 32);
#pragma unroll
        for (int i = 0; i < E / 2; ++i) mine[i * THREADS] = h ? x[0][i] : x[0][E / 2 + i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const uint32_t v = other[i * THREADS];
            x[0][i] = h ? v : x[0][i];
            x[0][E / 2 + i] = h ? x[0][E / 2 + i] : v;
        }
    };
    if constexpr (S::SPLIT && !INV) {
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const uint32_t xa = fwd_first<LOGN, F>(x[0][i], 0, lc), t = twmul<F>(x[0][E / 2 + i], tws[1], lc);
            x[0][i] = xa + t;
            x[0][E / 2 + i] = xa - t + lc.q2;
        }
        exchange();
    }
#pragma unroll
    for (int c = 0; c < V; ++c) {
        if constexpr (INV) inv_strided<S::SPLIT, R, LOGN, SCALE, F>(x[c], h, tws, lc);
        else fwd_strided<S::SPLIT, R, LOGN, F>(x[c], h, tws, lc);
    }
    if constexpr (S::SPLIT && INV) {
        exchange();
#pragma unroll
        for (int i = 0; i < E / 2; ++i)  // the offset of warp 0's elements covers warp 1's, which are products (below 2q)
            inv_last<SCALE, F>(x[0][i], x[0][E / 2 + i], inv_offset<F>(lc, A - 1, i), lc);
    }
    uint32_t* dst = S::SPLIT && !INV ? out + h * (E / 2) * BLOCK : out;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        uint32_t t[V];
#pragma unroll
        for (int c = 0; c < V; ++c) t[c] = x[c][i];
        *reinterpret_cast<T*>(dst + (INV ? pos(i) : i * BLOCK)) = pack(t);
    }
}

// Word of element e of a block in its warp's 4 KiB: swz keeps the three patterns (a lane's 32
// consecutive elements, lanes over consecutive elements, lanes over consecutive 16-byte groups) free of
// bank conflicts.
__device__ __forceinline__ uint4* chunk_of(uint32_t* sm, int e) { return reinterpret_cast<uint4*>(&sm[cc::swz(e)]); }

// Twiddles of inverse stages E0 .. E1-1 of sub-transform J over 32 consecutive elements (as
// cc::load_tw_inv): requested in two parts, the first with the data, which 96 registers allow.
template <int LOGN, int E0, int E1>
__device__ __forceinline__ void load_tw_block(uint2 (&w)[31], uint32_t J, const uint2* tw) {
#pragma unroll
    for (int e = E0; e < E1; ++e)
#pragma unroll
        for (int g = 0; g < (16 >> e); ++g)
            w[cc::inv_tw_off(5, e) + g] = __ldg(tw + ((1u << LOGN) >> (e + 1)) + J + (g << (LOGN - 5)));
}

// Block-pass task of a warp: block blk of one row, through the warp's 4 KiB of shared memory.  Forward in
// place in out (canonical results), inverse in -> out (HAD: the Montgomery product of two inputs on
// the way in).
template <int LOGN, int MODE, int F>
__device__ __forceinline__ void block_task(uint32_t* sm, uint32_t row, uint32_t blk, const KRows& a) {
    constexpr int N = 1 << LOGN, A = LOGN - LOGB;
    constexpr bool INV = MODE == MODE_INV || MODE == MODE_HAD_INV, HAD = MODE == MODE_HAD_INV;
    const int lane = threadIdx.x & 31;
    const LimbConst& lc = row_lc<F>(a, row);
    uint32_t* out = row_out<N, F>(a, row) + blk * BLOCK;
    uint32_t x[32];
    if constexpr (!INV) {
        const uint2* tw = row_twf<N, F>(a, row);
#pragma unroll
        for (int k = 0; k < 32; ++k) x[k] = __ldcg(out + lane + 32 * k);
        fwd_uniform<LOGN, A, F>(x, blk, tw, lc);
#pragma unroll
        for (int k = 0; k < 32; ++k) sm[cc::swz(lane + 32 * k)] = x[k];
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint4 v = *chunk_of(sm, 32 * lane + 4 * c);
            x[4 * c] = v.x;
            x[4 * c + 1] = v.y;
            x[4 * c + 2] = v.z;
            x[4 * c + 3] = v.w;
        }
        cc::fwd_stages<5, LOGN, LOGN - 5, F>(x, blk * 32 + lane, tw, lc);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            *chunk_of(sm, 32 * lane + 4 * c) = make_uint4(reduce_out<F>(x[4 * c], lc), reduce_out<F>(x[4 * c + 1], lc),
                                                          reduce_out<F>(x[4 * c + 2], lc), reduce_out<F>(x[4 * c + 3], lc));
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int e = (c * 32 + lane) * 4;
            *reinterpret_cast<uint4*>(out + e) = *chunk_of(sm, e);
        }
    } else {
        const uint2* tw = row_twi<N, F>(a, row);
        const uint32_t* in = row_in<N, F>(a, row) + blk * BLOCK;
        uint4 v[8];
        uint2 w[31];
        load_tw_block<LOGN, 0, 2>(w, blk * 32 + lane, tw);
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = __ldcg(reinterpret_cast<const uint4*>(in) + c * 32 + lane);
        if constexpr (HAD) {
            const uint4* had = reinterpret_cast<const uint4*>(row_had<N, F>(a, row) + blk * BLOCK);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 h = __ldcg(had + c * 32 + lane);
                v[c] = make_uint4(mul_mont_lazy(v[c].x, h.x, lc.q, lc.qinv_neg), mul_mont_lazy(v[c].y, h.y, lc.q, lc.qinv_neg),
                                  mul_mont_lazy(v[c].z, h.z, lc.q, lc.qinv_neg), mul_mont_lazy(v[c].w, h.w, lc.q, lc.qinv_neg));
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) *chunk_of(sm, (c * 32 + lane) * 4) = v[c];
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint4 t = *chunk_of(sm, 32 * lane + 4 * c);
            x[4 * c] = t.x;
            x[4 * c + 1] = t.y;
            x[4 * c + 2] = t.z;
            x[4 * c + 3] = t.w;
        }
        load_tw_block<LOGN, 2, 5>(w, blk * 32 + lane, tw);
        cc::inv_stages_w<5, LOGN, 0, 0, F>(x, w, lc);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            *chunk_of(sm, 32 * lane + 4 * c) = make_uint4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 32; ++k) x[k] = sm[cc::swz(lane + 32 * k)];
        inv_uniform<LOGN, 5, F>(x, blk, tw, lc);
#pragma unroll
        for (int k = 0; k < 32; ++k) out[lane + 32 * k] = x[k];
    }
}

template <int LOGN, int MODE, int F, int SMALL>
__global__ void __launch_bounds__(THREADS, SM_WARPS * 32 / THREADS) strided_kernel(const __grid_constant__ KRows a) {
    typedef Strided<LOGN, SMALL> S;
    __shared__ __align__(16) uint2 tws[1 << S::A];
    __shared__ uint32_t swap[S::SPLIT ? (1 << (S::R - 1)) * THREADS : 1];
    griddep_wait();
    strided_task<LOGN, MODE, F, SMALL>(tws, swap, blockIdx.x / S::PARTS, blockIdx.x % S::PARTS, a);
}

template <int LOGN, int MODE, int F>
__global__ void __launch_bounds__(32, SM_WARPS) block_kernel(const __grid_constant__ KRows a) {
    __shared__ __align__(16) uint32_t sm[BLOCK];
    constexpr uint32_t BLOCKS = (1u << LOGN) / BLOCK;
    griddep_wait();
    block_task<LOGN, MODE, F>(sm, blockIdx.x / BLOCKS, blockIdx.x % BLOCKS, a);
}

template <int LOGN, int MODE, int F, int SMALL>
cudaError_t launch_pair_t(const KRows& a, size_t rows, cudaStream_t s) {
    constexpr bool INV = MODE != MODE_FWD && MODE != MODE_RS_FWD;
    // the scale N^-1 2^32 is the strided pass's only difference, the product the block pass's
    constexpr int MS = MODE == MODE_INV_R ? MODE_HAD_INV : MODE, MB = MODE == MODE_INV_R ? MODE_INV : MODE;
    const dim3 gs((unsigned)(rows * Strided<LOGN, SMALL>::PARTS)), gb((unsigned)(rows << (LOGN - LOGB)));
    if (!INV) {
        cudaError_t e = launch_pdl(strided_kernel<LOGN, MS, F, SMALL>, gs, dim3(THREADS), 0, s, a);
        return e != cudaSuccess ? e : launch_pdl(block_kernel<LOGN, MB, F>, gb, dim3(32), 0, s, a);
    }
    cudaError_t e = launch_pdl(block_kernel<LOGN, MB, F>, gb, dim3(32), 0, s, a);
    return e != cudaSuccess ? e : launch_pdl(strided_kernel<LOGN, MS, F, SMALL>, gs, dim3(THREADS), 0, s, a);
}
// SMALL, 32 elements per thread of the strided pass: twice the warps, half the serial chain, and two
// warps per position at N = 2^16.  Forward up to 44 rows of 2^16 elements, the inverse forms to
// 256, the rescaling form (whose second operand fills the registers) always.  us, 64 / 32
// elements, N = 2^16:
//   rows       1          8          24         48           192          384
//   forward    5.7 / 5.2  6.2 / 5.6  8.7 / 8.5  12.4 / 12.6  39.6 / 40.4  77.8 / 79.8
//   inverse    6.4 / 5.2  6.9 / 5.7  9.5 / 8.7  13.6 / 13.2  39.5 / 39.0  81.1 / 83.8
//   rescaling             7.6 / 6.0  10.2/ 9.3  14.6 / 13.3  47.0 / 45.7  92.9 / 87.8
template <int LOGN, int MODE, int F>
cudaError_t launch_pair(const KRows& a, size_t rows, cudaStream_t s) {
    constexpr bool RS = MODE == MODE_RS_FWD;
    const size_t rows16 = (rows << LOGN) >> 16;
    if constexpr (LOGN == 17) return launch_pair_t<LOGN, MODE, F, 0>(a, rows, s);
    else if constexpr (RS) return launch_pair_t<LOGN, MODE, F, 1>(a, rows, s);
    else return rows16 <= (MODE == MODE_FWD ? 44u : 256u) ? launch_pair_t<LOGN, MODE, F, 1>(a, rows, s)
                                                          : launch_pair_t<LOGN, MODE, F, 0>(a, rows, s);
}

// rows == 0 launches nothing
template <int LOGN, int F>
cudaError_t launch_mode(NttMode mode, const KRows& a, size_t rows, cudaStream_t s) {
    switch (mode) {
        case MODE_FWD: return launch_pair<LOGN, MODE_FWD, F>(a, rows, s);
        case MODE_INV: return launch_pair<LOGN, MODE_INV, F>(a, rows, s);
        case MODE_HAD_INV: return launch_pair<LOGN, MODE_HAD_INV, F>(a, rows, s);
        case MODE_INV_R: return launch_pair<LOGN, MODE_INV_R, F>(a, rows, s);
        case MODE_RS_FWD:
            if constexpr ((F & 1) == 0) return launch_pair<LOGN, MODE_RS_FWD, F>(a, rows, s);
            else return cudaErrorNotSupported;
        default: return cudaErrorNotSupported;
    }
}

// lazy: every modulus of the parameter set is below 2^28
template <int LOGN>
cudaError_t launch_logn(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy) {
    if (rows == 0) return cudaSuccess;
    if (a.desc) return lazy ? launch_mode<LOGN, 3>(mode, a, rows, s) : launch_mode<LOGN, 1>(mode, a, rows, s);
    return lazy ? launch_mode<LOGN, 2>(mode, a, rows, s) : launch_mode<LOGN, 0>(mode, a, rows, s);
}

// One ring degree each, compiled in its own translation unit (build time).
cudaError_t launch_14(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy);
cudaError_t launch_15(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy);
cudaError_t launch_16(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy);
cudaError_t launch_17(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy);

}  // namespace cc2
}  // namespace hefx
