// Tensor-core basis conversion (path c): App. B's BConv with its step-2 MatModMul turned
// into a BAT digit-split matrix product (Sec. IV-A3, "High-Precision MatModMul in BConv").
//
//   D[n][(j, o)] = sum_{(i, d)} byte_d(b_{n,i}) * chunk_o([qhat_i]_{p_j} 2^(8d) mod p_j) + bias[(j, o)]
//   out_{n,j}    = ( sum_o D[n][(j, o)] 2^(8o) ) mod p_j
//
// b_{n,i} = [a_{n,i} qhat_i^-1]_{q_i} is step 1 (a Shoup product).  One kernel runs the plain
// conversion, ModDown (its epilogue returns (x_j - out_j) P^-1, or x_j - out_j P^-1 where x_j carries
// the factor already) and ModUp (every digit in one
// launch).
//
// What bounds it: memory, once the work per (coefficient, limb) is small enough.  The MMAs are
// a few percent of the tensor pipe; the threads' work is what counts, about 10 instructions per
// source residue and 14 per output, so it is cut down at both ends:
//  - The digits are the residue's four bytes, stored as fp16 words without a conversion: the
//    bits of a byte are the subnormal fp16 value byte * 2^-24, so one byte permute makes two
//    digits.  The constants' chunks are signed bytes times 2^8 (exact in fp16), so that the
//    integer a column sums is scaled by 2^-16.
//  - A column's sum lies in an interval shorter than 2^23 (L * 828 * 128 at most); three constant
//    columns of A times the bias rows of B shift it to [2^23, 2^24) units, where the accumulator's
//    low 23 bits are the integer itself: no conversion instruction.  Every partial sum is a whole
//    number of units below 2^24, so the fp32 accumulation is exact.
//  - The biases of a target are chosen with sum_o bias_o 2^(8o) = 0 mod p_j, so the merged value
//    U < 2^48 is the result mod p_j.  With x = U >> 16 (below 2^31.1) and mu = floor(2^48 / p), the
//    quotient estimate floor(x mu / 2^32) is short of U / p by less than 1.76 for p >= 2^18:
//    one multiply-high, one multiply and one conditional subtraction finish (a plan with a smaller
//    target takes a 64-bit Barrett reduction).
//
// GB300 mapping: one persistent CTA per SM walks tiles of 128 coefficients.  One warp keeps a ring
// of raw tiles (L rows x 512 bytes, TMA) in flight; producer groups of four warps take every PG-th
// tile, write its digits into a ring of K-major 128B-swizzled A buffers (two sources per 16-byte
// store, conflict free); one thread issues the tcgen05 MMAs against the constant B operand
// (resident for the whole kernel) into a ring of TMEM accumulators; epilogue groups of four warps
// merge, reduce and store.  The groups are split between the two roles by the plan's sources
// and targets.
//
// Measured at N = 2^16, against the kernel before it (7-bit digits converted with HSUB2, MMAs issued
// under `if (lane == 0)`, one epilogue group) or the CUDA-core kernel, whichever was taken: 24 -> 8 at
// batch 16 48.1 -> 30.5 us (4.4 TB/s of inputs and outputs; 20 us with the digits and the epilogue left
// out), 24 -> 56 at batch 8 129 -> 41.2 us (the epilogue's four groups bind), ModUp of three digits
// 16 -> 48 46 -> 20 us, ModDown of two polynomials 16 -> 48 40 -> 21 us.  Four or six groups
// instead of five: 36.6 / 42.0 and 34.6 / 42.2 us.  MMAs of two tiles issued in turn, to hide the
// accumulator's latency: no gain at 8 targets, 53 us at 56.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "bconv_common.h"
#include "host_nt.h"
#include "modarith.cuh"
#include "tc_common.cuh"

namespace hefx {

namespace {

constexpr int KO = 4;                // chunks per constant
constexpr int TILE = 128;            // coefficients per tile: MMA rows
constexpr int GROUP = 128;           // threads of a producer or epilogue group
#ifndef HEFX_BT_GROUPS
#define HEFX_BT_GROUPS 5
#endif
constexpr uint32_t GROUPS = HEFX_BT_GROUPS;
constexpr int THREADS = GROUPS * GROUP + 64;  // and the copy and MMA warps
constexpr uint32_t MAX_A = 4, MAX_ACC = 4;    // rings of A buffers and accumulators
constexpr uint32_t MAX_L = 48, MAX_LP = 64;  // MMA N <= 256
constexpr uint32_t CHUNK_BYTES = TILE * 128;  // 64 fp16 columns of a 128-row A tile
constexpr uint32_t MAX_STAGES = 8;
constexpr uint32_t SMEM_MAX = 232448;

// One conversion's constants (device).
struct BcTcConst {
    uint32_t L, Lp;
    uint32_t achunks;            // 64-column chunks of an A buffer
    uint32_t kc;                 // first of the constant columns (a multiple of 16)
    uint32_t npad;               // MMA N: KO columns per target, padded to 16
    uint32_t skip_lo, skip_len;  // ModUp: the digit's own rows of the output
    uint32_t pad;
    uint4 src[MAX_LP];           // (q_i, qhat_i^-1, Shoup companion, 0)
    uint4 tgt[MAX_LP];           // (p_j, floor(2^48 / p_j), (prod q)^-1 mod p_j, Shoup companion)
    uint64_t mu64[MAX_LP];       // floor(2^64 / p_j)
};
static_assert(sizeof(BcTcConst) % 16 == 0, "copied as uint4");

// BT_SMALL: the plain conversion with a target below 2^18.
enum : int { BT_FAST = 0, BT_MODDOWN = 1, BT_MODUP = 2, BT_SMALL = 3, BT_MODDOWN_SCALED = 4 };
template <int MODE>
constexpr bool kModDown = MODE == BT_MODDOWN || MODE == BT_MODDOWN_SCALED;

// Shared-memory layout of a launch, sized for its largest conversion (bytes from a 1 KiB-aligned base).
struct BcTcLayout {
    uint32_t a_bytes;    // one A buffer
    uint32_t ac_off;     // the shared constant chunk (0: inside the A buffers)
    uint32_t b_off, raw_off, bar_off, total;
    uint32_t raw_bytes, stages, abufs, accs, tmem_cols;  // ring sizes
    uint32_t producers, esplit;  // producer groups; epilogue groups that share a tile
};

struct BcTcArgs {
    BcTcLayout lay;
    const BcTcConst* consts;   // [conversions of the launch]
    const uint8_t* image;      // their B operands, image_stride apart
    size_t image_stride;
    uint32_t* out;
    const uint32_t* xq;        // ModDown: the target-basis limbs
    size_t xq_stride, out_stride, digit_stride;  // words
    uint32_t in_rows, in_row0;  // input rows of a polynomial, and its first source row
    uint32_t log2n, batch;
    uint32_t* err;
};

uint32_t a_chunks(uint32_t L) { return (L + 15) / 16; }
uint32_t const_col(uint32_t L) { return 16 * ((L + 3) / 4); }
bool const_apart(uint32_t L) { return const_col(L) == 64 * a_chunks(L); }
uint32_t b_chunks(uint32_t L) { return a_chunks(L) + (const_apart(L) ? 1 : 0); }
uint32_t n_pad(uint32_t Lp) { return (KO * Lp + 15) / 16 * 16; }
uint32_t image_size(uint32_t L, uint32_t npad) { return b_chunks(L) * npad * 128; }

// The layout of a launch: A buffers first (more let the MMAs and the producers run apart), then as
// many raw buffers as fit; stages == 0 where one CTA's shared memory does not hold two of each.
// apart: some conversion keeps its constant columns in the shared chunk.
BcTcLayout layout_for(uint32_t L, uint32_t Lp, uint32_t npad, uint32_t bimage, bool apart) {
    BcTcLayout l = {};
    l.a_bytes = a_chunks(L) * CHUNK_BYTES;
    l.raw_bytes = L * TILE * 4;
    const uint32_t room = SMEM_MAX - (uint32_t)sizeof(BcTcConst) - 64;
    for (l.abufs = MAX_A; l.abufs >= 2; --l.abufs) {
        uint32_t off = l.abufs * l.a_bytes;
        l.ac_off = apart ? off : 0;
        off += apart ? CHUNK_BYTES : 0;
        l.b_off = off;
        off += bimage;
        l.raw_off = off;
        const uint32_t fixed = off + 512 + 1024;  // barriers, and the alignment of the base
        const uint32_t want = l.abufs > 2 ? 4 : 2;
        if (fixed + want * l.raw_bytes > room) continue;
        l.stages = std::min(MAX_STAGES, (room - fixed) / l.raw_bytes);
        l.bar_off = off + l.stages * l.raw_bytes;
        l.total = l.bar_off + 512 + 1024;
        l.accs = std::min(MAX_ACC, 512 / npad);
        l.tmem_cols = 32;
        while (l.tmem_cols < l.accs * npad) l.tmem_cols *= 2;
        // groups in proportion to the instructions of a tile's two halves.  A waiter must not fall two
        // rounds behind a barrier (a parity says no more than odd or even), so a role has no more
        // groups at work on different tiles than its ring has slots (the MMAs, which fill and
        // free those rings, complete in order), and a raw buffer, whose copies may complete out of
        // order, always serves the same producer group
        const uint32_t wp = 11 * L + 40, we = 15 * Lp + 60;
        uint32_t prod = std::min(GROUPS - 1, std::max(1u, (GROUPS * wp + (wp + we) / 2) / (wp + we)));
        l.esplit = 1;
        if (GROUPS - prod > l.accs) {
            l.esplit = 2;
            if ((GROUPS - prod) % 2) ++prod;  // GROUPS - prod even and at most 2 accs
            while (GROUPS - prod > 2 * l.accs) prod += 2;
        }
        while (prod > l.abufs || prod > l.stages) prod -= l.esplit;
        l.producers = prod;
        l.stages -= l.stages % prod;
        return l;
    }
    l.stages = 0;
    return l;
}

// 1 in one thread of a converged warp (always the same one).
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p;
}

// tc::mma_f16 in the elected thread of a converged warp.
__device__ __forceinline__ void mma_elected(uint32_t leader, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                            uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}

// A ring's slot and the parity of its current round.
struct Ring {
    uint32_t i, ph;
    __device__ void advance(uint32_t by, uint32_t size) {
        i += by;
        while (i >= size) {
            i -= size;
            ph ^= 1u;
        }
    }
};

// byte b of x as two fp16 words: bits of bytes (0, 1) or (2, 3)
__device__ __forceinline__ uint2 byte_digits(uint32_t x) {
    return make_uint2(__byte_perm(x, 0, 0x4140), __byte_perm(x, 0, 0x4342));
}

template <int MODE>
__global__ void __launch_bounds__(THREADS, 1)
    bconv_tc_kernel(const __grid_constant__ BcTcArgs a, const __grid_constant__ CUtensorMap in_map) {
    extern __shared__ uint8_t smem_raw[];
    // aligned by an offset, not through an integer cast: the compiler keeps the shared address space
    uint8_t* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(16) BcTcConst c;
    const uint32_t tid = threadIdx.x, lane = tid & 31, nthreads = THREADS;
    const uint32_t stages = a.lay.stages, abufs = a.lay.abufs, accs = a.lay.accs;
    // the conversion of this CTA, and its place among the CTAs of that conversion
    const BcTcConst* gc = a.consts;
    const uint8_t* image = a.image;
    uint32_t* out = a.out;
    const uint32_t blk = blockIdx.x, nblk = gridDim.x;
    uint32_t* const err = a.err;
    if constexpr (MODE == BT_MODUP) {
        gc += blockIdx.y;
        image += blockIdx.y * a.image_stride;
        out += blockIdx.y * a.digit_stride;
    }
    for (uint32_t i = tid; i < sizeof(BcTcConst) / 16; i += nthreads)
        reinterpret_cast<uint4*>(&c)[i] = __ldg(reinterpret_cast<const uint4*>(gc) + i);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + a.lay.bar_off);
    uint64_t* raw_full = bars;                    // [stages] copies -> producers
    uint64_t* raw_empty = raw_full + MAX_STAGES;  // [stages] producers -> copies
    uint64_t* a_full = raw_empty + MAX_STAGES;    // [abufs] producers -> MMAs
    uint64_t* a_empty = a_full + MAX_A;           // [abufs] MMAs -> producers
    uint64_t* acc_full = a_empty + MAX_A;         // [accs] MMAs -> epilogue
    uint64_t* acc_empty = acc_full + MAX_ACC;     // [accs] epilogue -> MMAs
    uint64_t* mma_done = acc_empty + MAX_ACC;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    const uint32_t warp = tid >> 5;
    constexpr uint32_t COPY_WARP = GROUPS * 4, MMA_WARP = COPY_WARP + 1;
    for (uint32_t i = tid; i < abufs * a.lay.a_bytes / 16; i += nthreads)
        reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    if (a.lay.ac_off)
        for (uint32_t i = tid; i < CHUNK_BYTES / 16; i += nthreads)
            reinterpret_cast<uint4*>(smem + a.lay.ac_off)[i] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (uint32_t s = 0; s < MAX_STAGES; ++s) {
            tc::mbar_init(&raw_full[s], 1);
            tc::mbar_init(&raw_empty[s], 4);
        }
        for (uint32_t s = 0; s < MAX_A; ++s) {
            tc::mbar_init(&a_full[s], 4);
            tc::mbar_init(&a_empty[s], 1);
        }
        for (uint32_t s = 0; s < MAX_ACC; ++s) {
            tc::mbar_init(&acc_full[s], 1);
            tc::mbar_init(&acc_empty[s], 4 * a.lay.esplit);
        }
        tc::mbar_init(mma_done, 1);
        tc::fence_mbar_init();
    }
    if (warp == MMA_WARP) tc::tmem_alloc(tmem_slot, a.lay.tmem_cols);
    __syncthreads();
    const uint32_t L = c.L, Lp = c.Lp, npad = c.npad, kc = c.kc;
    const bool apart = kc == 64 * c.achunks;
    // constant operand B, and the constant columns of A (2^-16, 2^-5, 64: units of the bias digits)
    {
        const uint32_t bytes = (c.achunks + (apart ? 1u : 0u)) * npad * 128;
        for (uint32_t i = tid; i < bytes / 16; i += nthreads)
            reinterpret_cast<uint4*>(smem + a.lay.b_off)[i] = __ldg(reinterpret_cast<const uint4*>(image) + i);
        const uint32_t nbuf = apart ? 1u : abufs;
        for (uint32_t i = tid; i < nbuf * TILE; i += nthreads) {
            const uint32_t row = i & (TILE - 1);
            uint8_t* base = apart ? smem + a.lay.ac_off : smem + (i / TILE) * a.lay.a_bytes + (kc >> 6) * CHUNK_BYTES;
            *reinterpret_cast<uint2*>(base + tc::sw128_offset(row, kc & 63)) = make_uint2(0x28000100u, 0x00005400u);
        }
    }
    tc::fence_proxy_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // constants and images are written at plan creation; everything else waits for the stream's
    // preceding kernel
    griddep_wait();
    const uint32_t logt = a.log2n - 7;  // log2 of the tiles of a polynomial
    const uint32_t ntiles = a.batch << logt;

    const uint32_t group = tid / GROUP, row = tid & (TILE - 1), producers = a.lay.producers;
    const uint32_t row_bytes = 4u << a.log2n;

    if (warp == COPY_WARP) {  // ---- raw tiles
        Ring r = {0, 0};
        uint32_t used = 0;
        for (uint32_t t = blk; t < ntiles; t += nblk) {
            if (!tc::mbar_wait_warp(&raw_empty[r.i], r.ph ^ 1u, err, tc::ERR_TIMEOUT_EMPTY)) break;
            uint8_t* dst = smem + a.lay.raw_off + r.i * a.lay.raw_bytes;
            if (lane == 0) {
                // one 2D copy: 128 words x the map's box of rows (rows past a ragged digit go unused)
                tc::mbar_arrive_expect_tx(&raw_full[r.i], a.lay.raw_bytes);
                const uint32_t y = (t >> logt) * a.in_rows + a.in_row0 + (MODE == BT_MODUP ? c.skip_lo : 0u);
                tc::tma_load_2d(dst, &in_map, (int32_t)((t & ((1u << logt) - 1)) * TILE), (int32_t)y, &raw_full[r.i]);
            }
            used = used < stages ? used + 1 : used;
            r.advance(1, stages);
        }
        // no copy may still be writing shared memory when the CTA exits
        for (uint32_t k = 0; k < used; ++k) {
            if (r.i == 0) {
                r.i = stages;
                r.ph ^= 1u;
            }
            --r.i;
            tc::mbar_drain(&raw_full[r.i], r.ph);
        }
    } else if (warp == MMA_WARP) {  // ---- MMAs
        // One thread issues about eight MMAs a tile, so what it takes to issue one is a tile's shortest
        // time.  The whole warp runs the loop and only the instruction itself is elected: in
        // uniform code the descriptors stay in uniform registers, where the instruction takes them
        // (inside `if (lane == 0)` each was moved there first: 65-100 cycles an MMA).
        const uint32_t leader = elect_one();
        const uint32_t idesc = tc::idesc_f16_f32(TILE, npad);
        const uint64_t a0 = tc::sw128_desc(tc::smem_u32(smem)), a_step = a.lay.a_bytes >> 4;
        const uint64_t b0 = tc::sw128_desc(tc::smem_u32(smem + a.lay.b_off)), b_chunk = npad * 8;
        const uint32_t kin = (kc & 63) >> 3;  // the constant columns inside their chunk (16-byte units)
        const uint64_t bk = b0 + (kc >> 6) * b_chunk + kin;
        const uint64_t ak = apart ? tc::sw128_desc(tc::smem_u32(smem + a.lay.ac_off)) : 0;
        const uint32_t full = kc >> 6, rest = (kc & 63) >> 4;  // 64-column chunks of digits, steps of the last
        Ring ra = {0, 0}, rc = {0, 0};
        for (uint32_t t = blk; t < ntiles; t += nblk) {
            if (!tc::mbar_wait_warp(&a_full[ra.i], ra.ph, err, tc::ERR_TIMEOUT_FULL) ||
                !tc::mbar_wait_warp(&acc_empty[rc.i], rc.ph ^ 1u, err, tc::ERR_TIMEOUT_ACC))
                break;
            tc::tc_fence_after();
            const uint64_t ab = a0 + ra.i * a_step;
            const uint32_t acc = tmem + rc.i * npad;
            mma_elected(leader, acc, apart ? ak : ab + full * (CHUNK_BYTES >> 4) + kin, bk, idesc, 0);
            uint64_t ad = ab, bd = b0;
            for (uint32_t ch = 0; ch < full; ++ch) {
#pragma unroll
                for (uint32_t k = 0; k < 8; k += 2) mma_elected(leader, acc, ad + k, bd + k, idesc, 1);
                ad += CHUNK_BYTES >> 4;
                bd += b_chunk;
            }
#pragma unroll
            for (uint32_t k = 0; k < 3; ++k)
                if (k < rest) mma_elected(leader, acc, ad + 2 * k, bd + 2 * k, idesc, 1);
            if (leader) {
                tc::mma_commit(&acc_full[rc.i]);
                tc::mma_commit(&a_empty[ra.i]);
            }
            __syncwarp();
            ra.advance(1, abufs);
            rc.advance(1, accs);
        }
        if (leader) tc::mma_commit(mma_done);
        __syncwarp();
        tc::mbar_drain(mma_done, 0);  // before TMEM is released, whatever the error flag says
    } else if (group < producers) {  // ---- step 1 and digits
        const uint32_t rx = (row & 7) << 4;
        Ring rr = {0, 0}, ra = {0, 0};
        rr.advance(group, stages);
        ra.advance(group, abufs);
        for (uint64_t t = blk + (uint64_t)group * nblk; t < ntiles; t += (uint64_t)producers * nblk) {
            if (!tc::mbar_wait_warp(&raw_full[rr.i], rr.ph, err, tc::ERR_TIMEOUT_FULL)) break;
            if (!tc::mbar_wait_warp(&a_empty[ra.i], ra.ph ^ 1u, err, tc::ERR_TIMEOUT_EMPTY)) break;
            const uint32_t* raw = reinterpret_cast<const uint32_t*>(smem + a.lay.raw_off + rr.i * a.lay.raw_bytes) + row;
            uint8_t* A = smem + ra.i * a.lay.a_bytes + row * 128;
            char* own = nullptr;  // ModUp copies the digit's own limbs
            if constexpr (MODE == BT_MODUP)
                own = reinterpret_cast<char*>(out + ((uint32_t)t >> logt) * a.out_stride + ((size_t)c.skip_lo << a.log2n) +
                                              ((uint32_t)t & ((1u << logt) - 1)) * TILE + row);
            // sources i0 .. i0+7: four 16-byte stores.  All loads before the first store: the compiler
            // cannot move a shared-memory load over a store to A, and a tile's digits would then be
            // one chain of load latencies
            auto eight = [&](uint32_t i0, auto full) {
                uint32_t x[8];
                uint4 k[8];
#pragma unroll
                for (uint32_t u = 0; u < 8; ++u) {
                    const bool in_l = decltype(full)::value || i0 + u < L;
                    x[u] = in_l ? raw[(i0 + u) * TILE] : 0u;
                    k[u] = c.src[i0 + u];  // zeros past L
                }
                uint8_t* Ac = A + (i0 >> 4) * CHUNK_BYTES;
#pragma unroll
                for (uint32_t u = 0; u < 8; u += 2) {
                    uint2 d[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        d[e] = byte_digits(csub(mul_shoup_lazy(x[u + e], k[u + e].y, k[u + e].z, k[u + e].x), k[u + e].x));
                    if (decltype(full)::value || i0 + u < L)
                        *reinterpret_cast<uint4*>(Ac + (((i0 << 3) & 64) ^ ((u << 3) ^ rx))) = make_uint4(d[0].x, d[0].y, d[1].x, d[1].y);
                }
                if constexpr (MODE == BT_MODUP) {
#pragma unroll
                    for (uint32_t u = 0; u < 8; ++u)
                        if (decltype(full)::value || i0 + u < L)
                            *reinterpret_cast<uint32_t*>(own + (uint64_t)(i0 + u) * row_bytes) = x[u];
                }
            };
            uint32_t i0 = 0;
            for (; i0 + 8 <= L; i0 += 8) eight(i0, std::true_type{});
            if (i0 < L) eight(i0, std::false_type{});
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(&raw_empty[rr.i]);
                tc::mbar_arrive(&a_full[ra.i]);
            }
            rr.advance(producers, stages);
            ra.advance(producers, abufs);
        }
    } else {  // ---- merge, reduce, store
        const uint32_t esplit = a.lay.esplit, eg = (group - producers) / esplit, epis = (GROUPS - producers) / esplit;
        const uint32_t es = (group - producers) % esplit;  // this group takes every esplit-th column group
        const uint32_t quad = (warp & 3) << 21;  // TMEM lanes of this warp (lane << 16)
        Ring rc = {0, 0};
        rc.advance(eg, accs);
        auto epilogue = [&](uint32_t t, uint32_t cols) {
            const size_t x = (size_t)(t & ((1u << logt) - 1)) * TILE + row;
            char* dst = reinterpret_cast<char*>(out + (size_t)(t >> logt) * a.out_stride + x);
            [[maybe_unused]] const char* xq = nullptr;
            if constexpr (kModDown<MODE>)
                xq = reinterpret_cast<const char*>(a.xq + (size_t)(t >> logt) * a.xq_stride + x);
            // eight targets (two 16-column reads) at a time
            auto group8 = [&](uint32_t j0, auto full) {
                uint32_t r[32], v[8];
                tc::tmem_ld16(cols + j0 * 4, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
                if (decltype(full)::value || j0 + 4 < Lp)
                    tc::tmem_ld16(cols + j0 * 4 + 16, *reinterpret_cast<uint32_t(*)[16]>(&r[16]));
                [[maybe_unused]] uint32_t xv[8];
                if constexpr (kModDown<MODE>) {
#pragma unroll
                    for (uint32_t h = 0; h < 8; ++h)
                        xv[h] = decltype(full)::value || j0 + h < Lp
                                    ? __ldg(reinterpret_cast<const uint32_t*>(xq + (uint64_t)(j0 + h) * row_bytes)) : 0u;
                }
                tc::tmem_ld_wait();
#pragma unroll
                for (uint32_t h = 0; h < 8; ++h) {
                    // accumulator bits: 0x43000000 | integer (2^23 units of 2^-16 is 128)
                    const uint2 q = *reinterpret_cast<const uint2*>(&c.tgt[j0 + h]);  // zeros past Lp
                    const uint32_t lo = r[4 * h] + (r[4 * h + 1] << 8) - 0x43000000u;
                    const uint32_t hr = r[4 * h + 2] + (r[4 * h + 3] << 8);  // - 0x43000000
                    if constexpr (MODE != BT_SMALL) {
                        const uint32_t y = hr + (lo >> 16) - 0x43000000u;  // U >> 16
                        v[h] = csub(lo + (hr << 16) - __umulhi(y, q.y) * q.x, q.x);
                    } else {
                        v[h] = barrett64((uint64_t)lo + ((uint64_t)(hr - 0x43000000u) << 16), q.x, c.mu64[j0 + h]);
                    }
                    if constexpr (kModDown<MODE>) {
                        const uint2 w = *(reinterpret_cast<const uint2*>(&c.tgt[j0 + h]) + 1);
                        if constexpr (MODE == BT_MODDOWN)
                            v[h] = csub(mul_shoup_lazy(xv[h] + q.x - v[h], w.x, w.y, q.x), q.x);
                        else
                            v[h] = csub(xv[h] + q.x - csub(mul_shoup_lazy(v[h], w.x, w.y, q.x), q.x), q.x);
                    }
                }
#pragma unroll
                for (uint32_t h = 0; h < 8; ++h) {
                    const uint32_t j = j0 + h;
                    const uint32_t jr = MODE == BT_MODUP && j >= c.skip_lo ? j + c.skip_len : j;
                    if (decltype(full)::value || j < Lp)
                        *reinterpret_cast<uint32_t*>(dst + (uint64_t)jr * row_bytes) = v[h];
                }
            };
            uint32_t j0 = 8 * es;
            for (; j0 + 8 <= Lp; j0 += 8 * esplit) group8(j0, std::true_type{});
            if (j0 < Lp) group8(j0, std::false_type{});
        };
        for (uint64_t t = blk + (uint64_t)eg * nblk; t < ntiles; t += (uint64_t)epis * nblk) {
            if (!tc::mbar_wait_warp(&acc_full[rc.i], rc.ph, err, tc::ERR_TIMEOUT_ACC)) break;
            tc::tc_fence_after();
            const uint32_t cols = tmem + quad + rc.i * npad;
            epilogue((uint32_t)t, cols);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acc_empty[rc.i]);
            rc.advance(epis, accs);
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, a.lay.tmem_cols);
    }
}

uint16_t half_bits_int(int v) {  // |v| <= 2048, times 2^0
    if (v == 0) return 0;
    const uint32_t m = (uint32_t)(v < 0 ? -v : v);
    const int e = 31 - __builtin_clz(m);
    return (uint16_t)((v < 0 ? 0x8000u : 0u) | ((uint32_t)(e + 15) << 10) | ((m << 10 >> e) & 0x3FFu));
}

uint32_t sw128_offset_host(uint32_t row, uint32_t k) {
    const uint32_t chunk = (k >> 3) & 7u;
    return row * 128u + ((chunk ^ (row & 7u)) << 4) + ((k & 7u) << 1);
}

// Constants and B operand of one conversion (h: its sources, targets and matrix).  Lmax and npad
// are the launch's, for the digits of one ModUp; img is image_size(Lmax, npad) bytes, zeroed.
void fill_tc(const BConvConst& h, uint32_t Lmax, uint32_t npad, BcTcConst& c, uint8_t* img) {
    memset(&c, 0, sizeof c);
    c.L = h.L;
    c.Lp = h.Lp;
    c.achunks = a_chunks(Lmax);
    c.kc = const_col(Lmax);
    c.npad = npad;
    c.skip_lo = h.skip_lo;
    c.skip_len = h.skip_len;
    for (uint32_t i = 0; i < h.L; ++i) c.src[i] = make_uint4(h.q[i], h.qhat_inv[i], h.qhat_inv_sh[i], 0);
    auto put = [&](uint32_t row, uint32_t k, uint16_t bits) {
        memcpy(img + (size_t)(k / 64) * (npad * 128) + sw128_offset_host(row, k % 64), &bits, 2);
    };
    for (uint32_t j = 0; j < h.Lp; ++j) {
        const uint64_t p = h.p[j];
        c.tgt[j] = make_uint4((uint32_t)p, p >= (1u << 18) ? (uint32_t)(((uint64_t)1 << 48) / p) : 0u, h.pinv[j], h.pinv_sh[j]);
        c.mu64[j] = h.p_mu[j];
        int64_t low[KO] = {0, 0, 0, 0};  // the least value of each column's sum
        for (uint32_t i = 0; i < h.L; ++i) {
            uint64_t cst = h.qhat_p[i * kBConvMaxLimbs + j];
            for (uint32_t d = 0; d < 4; ++d) {
                const int64_t dmax = d < 3 ? 255 : (h.q[i] - 1) >> 24;
                int64_t rest = (int64_t)cst;
                for (int o = 0; o < KO; ++o) {  // signed bytes
                    int64_t ch = o < KO - 1 ? (int64_t)(int8_t)(rest & 255) : rest;
                    rest = (rest - ch) >> 8;
                    if (ch < 0) low[o] += dmax * ch;
                    // chunk * 2^8: eight more in the exponent
                    const uint16_t hb = half_bits_int((int)ch);
                    put(KO * j + o, 4 * i + d, ch ? (uint16_t)(hb + (8u << 10)) : (uint16_t)0);
                }
                cst = (cst << 8) % p;
            }
        }
        // biases: -low, and what makes sum_o bias_o 2^(8o) a multiple of p (less than p, in bytes)
        uint64_t sum = 0;
        for (int o = KO - 1; o >= 0; --o) sum = (sum * 256 + (uint64_t)(-low[o]) % p) % p;
        const uint64_t add = sum ? p - sum : 0;
        for (int o = 0; o < KO; ++o) {
            const uint32_t b = (uint32_t)(-low[o]) + (uint32_t)(o < KO - 1 ? (add >> (8 * o)) & 255 : add >> (8 * o));
            put(KO * j + o, c.kc, half_bits_int((int)(b & 2047)));
            put(KO * j + o, c.kc + 1, half_bits_int((int)((b >> 11) & 2047)));
            put(KO * j + o, c.kc + 2, half_bits_int((int)(b >> 22) + 2));  // + 2^23 units
        }
    }
}

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

template <int MODE>
cudaError_t launch_mode(const BcTcArgs& a, const CUtensorMap& in_map, dim3 grid, cudaStream_t s) {
    static bool attr_set[64] = {};  // per device; benign race (idempotent)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(bconv_tc_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(SMEM_MAX - sizeof(BcTcConst) - 64));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    return launch_pdl(bconv_tc_kernel<MODE>, grid, dim3(THREADS), a.lay.total, s, a, in_map);
}

}  // namespace

struct BcTcPlan {
    BcTcConst* d_const = nullptr;
    uint8_t* d_image = nullptr;  // constant B operands, already in the swizzled smem layout
    size_t image_stride = 0;
    BcTcLayout lay = {};
    uint32_t L = 0, npad = 0;    // of the largest conversion
    bool small_sources = false;  // every source below 2^28
    bool small_target = false;   // some target below 2^18: plain conversions only (BT_SMALL)
};

bool bconv_tc_engine(const BcTcPlan* tp, uint32_t log2n) { return tp != nullptr && log2n >= 7; }

// HEFX_PATH_TENSOR is offered where every source prime is below 2^28.
bool bconv_tc_available(const hefx_bconv_plan* plan) {
    return bconv_tc_engine(plan->tc, plan->log2n) && plan->tc->small_sources;
}

// Where the tensor kernel is the faster one.  The CUDA-core kernel makes one pass over the sources per
// 8 targets, at about the cost of the products, so beyond 8 targets it loses from the smallest call
// on (12 -> 28: 6.2 against 4.3 us for 2 tiles, 26.3 against 14.0 us for 2048; 24 -> 56 at 4096 tiles 129
// against 42 us); with up to 8 it is ahead while a call is less than seven tiles an SM
// (24 -> 8: 3.8 against 4.4 us at 128 tiles, 8.5 against 7.3 us at 1024, 48.2 against 30.7 us at
// 8192) or has few sources, whose tiles cost the tensor kernel 0.36 us an SM whatever
// they hold (4 -> 4 at 8192 tiles: 15.7 against 19.6 us).
static bool faster_on_tc(uint32_t L, uint32_t Lp, size_t ntiles) {
    return Lp > 8 ? L >= 4 : L >= 8 && L * Lp >= 64 && ntiles >= 1024;
}

bool bconv_prefer_tc(const hefx_bconv_plan* plan, size_t batch) {
    return bconv_tc_engine(plan->tc, plan->log2n) && faster_on_tc(plan->L, plan->Lp, (batch << plan->log2n) / TILE);
}

// Uploads the tensor form of `count` conversions of one launch; leaves *out null where it does
// not fit one CTA's shared memory (the CUDA-core kernels then run).
cudaError_t bconv_tc_create(const BConvConst* h, uint32_t count, BcTcPlan** out) {
    *out = nullptr;
    uint32_t L = 0, Lp = 0;
    bool small = true, small_target = false;
    for (uint32_t k = 0; k < count; ++k) {
        L = std::max(L, h[k].L);
        Lp = std::max(Lp, h[k].Lp);
        for (uint32_t i = 0; i < h[k].L; ++i) small = small && h[k].q[i] < (1u << 28);
        for (uint32_t j = 0; j < h[k].Lp; ++j) small_target = small_target || h[k].p[j] < (1u << 18);
    }
    if (L > MAX_L || Lp > MAX_LP) return cudaSuccess;
    const uint32_t npad = n_pad(Lp), size = image_size(L, npad);
    const BcTcLayout lay = layout_for(L, Lp, npad, size, const_apart(L));
    if (!lay.stages) return cudaSuccess;
    std::vector<BcTcConst> hc(count);
    std::vector<uint8_t> img((size_t)size * count, 0);
    for (uint32_t k = 0; k < count; ++k) fill_tc(h[k], L, npad, hc[k], img.data() + (size_t)k * size);
    BcTcPlan* tp = new BcTcPlan();
    tp->image_stride = size;
    tp->lay = lay;
    tp->L = L;
    tp->npad = npad;
    tp->small_sources = small;
    tp->small_target = small_target;
    cudaError_t e = cudaMalloc(&tp->d_const, sizeof(BcTcConst) * count);
    if (e == cudaSuccess) e = cudaMemcpy(tp->d_const, hc.data(), sizeof(BcTcConst) * count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&tp->d_image, img.size());
    if (e == cudaSuccess) e = cudaMemcpy(tp->d_image, img.data(), img.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        bconv_tc_free(tp);
        return e;
    }
    *out = tp;
    return cudaSuccess;
}

void bconv_tc_free(BcTcPlan* tp) {
    if (!tp) return;
    if (tp->d_const) cudaFree(tp->d_const);
    if (tp->d_image) cudaFree(tp->d_image);
    delete tp;
}

namespace {

// The launch of a plan's conversions over [batch][in_rows][n] inputs whose source rows start at in_row0.
template <int MODE>
cudaError_t launch_plan(const BcTcPlan* tp, BcTcArgs a, const uint32_t* in, uint32_t in_rows, uint32_t in_row0,
                        uint32_t log2n, size_t batch, size_t blocks, uint32_t ny, cudaStream_t stream) {
    const size_t ntiles = (batch << log2n) / TILE;
    if (ntiles == 0) return cudaSuccess;
    if (ntiles > 0x3fffffffull || batch * in_rows > 0x3fffffffull) return cudaErrorInvalidValue;
    CUtensorMap map;
    if (!encode_map_2d(&map, CU_TENSOR_MAP_DATA_TYPE_UINT32, const_cast<uint32_t*>(in), (uint64_t)1 << log2n,
                       batch * in_rows, (uint64_t)4 << log2n, TILE, tp->L, CU_TENSOR_MAP_SWIZZLE_NONE))
        return cudaErrorInvalidValue;
    a.lay = tp->lay;
    a.consts = tp->d_const;
    a.image = tp->d_image;
    a.image_stride = tp->image_stride;
    a.in_rows = in_rows;
    a.in_row0 = in_row0;
    a.log2n = log2n;
    a.batch = (uint32_t)batch;
    return launch_mode<MODE>(a, map, dim3((unsigned)std::min(ntiles, blocks), ny), stream);
}

}  // namespace

cudaError_t launch_bconv_tc(const hefx_bconv_plan* plan, const uint32_t* in, uint32_t* out, size_t batch,
                            cudaStream_t stream) {
    if (!bconv_tc_engine(plan->tc, plan->log2n)) return cudaErrorNotSupported;
    BcTcArgs a = {};
    a.out = out;
    a.out_stride = (size_t)plan->Lp << plan->log2n;
    a.err = plan->d_err;
    if (plan->tc->small_target)
        return launch_plan<BT_SMALL>(plan->tc, a, in, plan->L, 0, plan->log2n, batch, (size_t)sm_count(), 1, stream);
    return launch_plan<BT_FAST>(plan->tc, a, in, plan->L, 0, plan->log2n, batch, (size_t)sm_count(), 1, stream);
}

cudaError_t launch_mod_down_tc(const hefx_bconv_plan* plan, const uint32_t* x, uint32_t* out, size_t batch,
                               bool scaled, cudaStream_t stream) {
    if (plan->mod_down_cc || !bconv_prefer_tc(plan, batch) || plan->tc->small_target) return cudaErrorNotSupported;
    BcTcArgs a = {};
    a.out = out;
    a.xq = x;
    a.xq_stride = (size_t)(plan->L + plan->Lp) << plan->log2n;
    a.out_stride = (size_t)plan->Lp << plan->log2n;
    a.err = plan->d_err;
    if (scaled)
        return launch_plan<BT_MODDOWN_SCALED>(plan->tc, a, x, plan->L + plan->Lp, plan->Lp, plan->log2n, batch,
                                              (size_t)sm_count(), 1, stream);
    return launch_plan<BT_MODDOWN>(plan->tc, a, x, plan->L + plan->Lp, plan->Lp, plan->log2n, batch,
                                   (size_t)sm_count(), 1, stream);
}

cudaError_t launch_mod_up_tc(const hefx_modup_plan* mp, const uint32_t* c, uint32_t* U, size_t batch,
                             cudaStream_t stream) {
    if (mp->cc || !bconv_tc_engine(mp->tc, mp->log2n) || mp->tc->small_target ||
        !faster_on_tc(mp->alpha, mp->L + mp->K - mp->alpha, (batch * mp->dnum << mp->log2n) / TILE))
        return cudaErrorNotSupported;
    BcTcArgs a = {};
    a.out = U;
    a.digit_stride = (size_t)(mp->L + mp->K) << mp->log2n;
    a.out_stride = a.digit_stride * mp->dnum;
    a.err = mp->d_err;
    return launch_plan<BT_MODUP>(mp->tc, a, c, mp->L, 0, mp->log2n, batch,
                                 std::max<size_t>(1, (size_t)sm_count() / mp->dnum), mp->dnum, stream);
}

}  // namespace hefx
