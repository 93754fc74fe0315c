// CUDA-core NTT dispatcher and public launchers; the kernels are in ntt_cc_impl.cuh and are
// instantiated per ring-degree range in ntt_cc_range_*.cu (parallel compilation).
#include <cstring>

#include "ntt_cc_2p.cuh"
#include "ntt_cc_impl.cuh"

namespace hefx {

// max_prime: the largest modulus of the rows, which decides between the lazy ranges (below 2^28) and Harvey's
cudaError_t launch_dispatch(uint32_t log2n, uint32_t max_prime, NttMode mode, const cc::KArgs& a, size_t rows,
                            cudaStream_t stream);

namespace {

// The two-pass schedule (ntt_cc_2p.cuh) is built for N = 2^14 .. 2^17 and every mode but the product's
// second half, which would need a workspace for NTT(b).  AUTO takes it always at N = 2^17 and for the
// inverse of a Hadamard product; else while the rows' elements are at most: forward 256 x 2^16,
// inverse 320 x 2^16 (at N = 2^16 always), rescaling forward 144 x 2^16.  Beyond, the
// intermediate leaves L2 between the launches and the cluster kernel's single trip through HBM
// wins (us, cluster / two-pass):
//   N = 2^16   24 rows     96          144         240         288         384
//   forward    10.1 / 8.5  27.0 / 22.8 33.1 / 31.0 50.2 / 48.8 59.2 / 59.3 75.4 / 77.8
//   inverse    11.9 / 8.7  31.0 / 23.3 39.2 / 30.9 57.3 / 48.1 67.7 / 61.6 85.9 / 81.1
//   Hadamard   13.4 / 9.2  40.7 / 27.5 49.6 / 38.0 73.6 / 61.7 91.8 / 74.3 116 / 95.0
//   rescaling  11.1 / 9.3  29.6 / 25.6 35.8 / 35.4 53.3 / 57.1 65.6 / 68.8 84.2 / 87.8
//   N = 2^15   24 rows     192         384         576         N = 2^17    24 rows     96          384
//   forward    7.9 / 6.1   24.4 / 19.8 41.1 / 38.9 55.9 / 57.2             17.6 / 14.0 52.3 / 44.8 191 / 173
//   inverse    9.3 / 6.3   26.0 / 20.5 44.6 / 36.8 60.7 / 57.3             22.0 / 14.8 62.2 / 43.7 219 / 170
//   rescaling  9.3 / 6.7   27.8 / 24.0 45.7 / 44.0 63.1 / 64.9             19.5 / 16.4 56.3 / 52.6 209 / 196
// and at N = 2^14 768 rows 43.1 / 38.3 and 40.8 / 34.3, 15 rows 7.9 / 5.0 and 8.7 / 5.2.
//
// A lone forward call (a call of its own, on a stream that is not being captured) of at most 32 rows of
// 2^15 stays one cluster launch.  A launch costs the host 1.4 us, and a PyTorch program that looks its
// current stream up for each call (2.8 us) is bound by the host with two of them: 8.5 us a call, 4
// rows, against 7.4 with one.  Where the program keeps the stream the device decides, 4.7 against
// 7.4 us, so captured calls, row lists and the halves of a product take two launches.  The other
// forms and sizes are level or better with two either way (one / two launches, stream looked up:
// N = 2^14 forward 8.5 / 8.5, inverse 8.7 / 8.6; 2^15 inverse 8.5 / 8.6).
bool two_pass(const hefx_params* p, NttMode mode, size_t rows, bool lone = false) {
    if (p->log2n < 14 || p->log2n > 17 || mode == MODE_FWD_HAD_INV || mode == MODE_PRODUCT ||
        rows > (1u << 24))
        return false;
    if (p->cc_schedule != HEFX_CC_AUTO) return p->cc_schedule == HEFX_CC_TWO_PASS;
    if (lone && mode == MODE_FWD && p->log2n == 15 && rows <= 32) return false;
    if (p->log2n == 17 || mode == MODE_HAD_INV || (p->log2n == 16 && mode == MODE_INV)) return true;
    return (rows << p->log2n) >> 16 <= (mode == MODE_FWD ? 256u : mode == MODE_INV ? 320u : 144u);
}

cudaError_t launch_two_pass(uint32_t log2n, uint32_t max_prime, NttMode mode, const cc::KArgs& a, size_t rows,
                            cudaStream_t stream) {
    const bool lazy = max_prime < (1u << 28);
    return log2n == 14 ? cc2::launch_14(mode, a, rows, stream, lazy)
           : log2n == 15 ? cc2::launch_15(mode, a, rows, stream, lazy)
           : log2n == 16 ? cc2::launch_16(mode, a, rows, stream, lazy)
                         : cc2::launch_17(mode, a, rows, stream, lazy);
}

// The product's second half, INTT(NTT(b) o c) with c in the output, as the cluster forward transform
// that multiplies on its way out and the two-pass inverse, instead of one cluster launch with two
// cross-CTA steps.  The whole product of two polynomials, us, one launch / this:
//   N = 2^17   1 row 29.3 / 25.5   24 rows 55.1 / 51.2   96 rows 163 / 149
//   N = 2^16   1 row 21.0 / 18.9   48 rows 44.0 / 44.7   96 rows 80.1 / 75.4   384 rows 249 / 244
//   N = 2^15   1 row 19.8 / 17.4   96 rows 38.7 / 38.4   192 rows 71.3 / 67.9  384 rows 123 / 121
//   N = 2^14   1 row 19.5 / 17.2   96 rows 26.8 / 26.1   192 rows 37.0 / 37.3  768 rows 117 / 118
bool halves(const hefx_params* p, NttMode mode, size_t rows) {
    return mode == MODE_FWD_HAD_INV && p->log2n >= 14 && p->log2n <= 17 && p->cc_schedule != HEFX_CC_CLUSTER &&
           rows <= (p->log2n == 14 ? 128u : 1u << 24);
}

cudaError_t launch_halves(const hefx_params* p, cc::KArgs& a, size_t rows, cudaStream_t stream) {
    cudaError_t e = launch_dispatch(p->log2n, p->max_prime, MODE_FWD_HAD, a, rows, stream);
    if (e != cudaSuccess) return e;
    a.in = a.out;
    return launch_two_pass(p->log2n, p->max_prime, MODE_INV_R, a, rows, stream);
}

}  // namespace

// Tensor map of a contiguous [rows][N] input for the inverse transforms' TMA loads.
cudaError_t encode_input_map(const hefx_params* p, const uint32_t* in, size_t rows, CUtensorMap* map) {
    const uint64_t lines = (uint64_t)rows * p->n / 32;  // 128-byte lines of 32 words
    if (!encode_map_2d(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, const_cast<uint32_t*>(in), 32, lines, 128, 32, 256,
                       CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorNotSupported;
    return cudaSuccess;
}

cudaError_t launch_ntt_cc(const hefx_params* p, NttMode mode, const uint32_t* in, const uint32_t* had, uint32_t* out,
                          size_t rows, cudaStream_t stream, bool lone) {
    cc::KArgs a;
    memset(&a.tmap_in, 0, sizeof a.tmap_in);
    memset(&a.tmap_out, 0, sizeof a.tmap_out);
    a.err = p->d_err_cc;
    const bool tp = two_pass(p, mode, rows, lone);
    if (mode == MODE_INV && rows > 0 && p->log2n >= 13 && !tp) {
        cudaError_t e = encode_input_map(p, in, rows, &a.tmap_in);
        if (e != cudaSuccess) return e;
    }
    if (mode == MODE_FWD && rows > 0 && p->log2n >= 13 && !tp) {
        cudaError_t e = encode_input_map(p, out, rows, &a.tmap_out);
        if (e != cudaSuccess) return e;
    }
    a.in = in;
    a.had = had;
    a.out = out;
    a.tw_f = p->d_tw_fwd;
    a.tw_i = p->d_tw_inv;
    a.lc = p->d_lc;
    a.desc = nullptr;
    a.rows = (uint32_t)rows;
    a.L = p->nlimbs;
    a.in_rows = 0;
    if (rows == 0) return cudaSuccess;
    if (halves(p, mode, rows)) return launch_halves(p, a, rows, stream);
    return tp ? launch_two_pass(p->log2n, p->max_prime, mode, a, rows, stream)
              : launch_dispatch(p->log2n, p->max_prime, mode, a, rows, stream);
}

bool one_launch_if_lone(const hefx_params* p, NttMode mode, size_t rows) {
    return two_pass(p, mode, rows) && !two_pass(p, mode, rows, true);
}

uint32_t ntt_cc_launches(const hefx_params* p, NttMode mode, size_t rows, bool lone, bool row_list) {
    if (rows == 0) return 0;
    if (!row_list && halves(p, mode, rows)) return 3;
    if (mode == MODE_RS_FWD && p->log2n <= 13) return 2;  // rescaled, then transformed
    return two_pass(p, mode, rows, lone) ? 2 : 1;
}

cudaError_t launch_ntt_cc_rescale(const hefx_params* p, const uint32_t* in, uint32_t* out, size_t batch,
                                  cudaStream_t stream) {
    const uint32_t L = p->nlimbs;
    const size_t rows = batch * (L - 1);
    if (rows == 0) return cudaSuccess;
    cc::KArgs a;
    memset(&a.tmap_in, 0, sizeof a.tmap_in);
    memset(&a.tmap_out, 0, sizeof a.tmap_out);
    a.err = p->d_err_cc;
    const bool tp = two_pass(p, MODE_RS_FWD, rows);
    if (p->log2n >= 13 && !tp) {
        cudaError_t e = encode_input_map(p, out, rows, &a.tmap_out);
        if (e != cudaSuccess) return e;
    }
    a.in = in;
    a.had = nullptr;
    a.out = out;
    a.tw_f = p->d_tw_fwd;  // limbs 0 .. L-2 of the full set: the tables of q_0 .. q_{L-2}
    a.tw_i = p->d_tw_inv;
    a.lc = p->d_lc;        // rs_inv: q_{L-1}^-1 mod q_i
    a.desc = nullptr;
    a.rows = (uint32_t)rows;
    a.L = L - 1;
    a.in_rows = L;
    if (tp) return launch_two_pass(p->log2n, p->max_prime, MODE_RS_FWD, a, rows, stream);
    cudaError_t e = launch_dispatch(p->log2n, p->max_prime, MODE_RS_FWD, a, rows, stream);
    if (e != cudaErrorNotSupported) return e;
    // not fused at this N: rescale into out, then the forward transform of its L - 1 limbs
    e = launch_rescale(p, in, out, batch, stream);
    if (e != cudaSuccess) return e;
    a.in = out;
    a.in_rows = 0;
    return launch_dispatch(p->log2n, p->max_prime, MODE_FWD, a, rows, stream);
}

cudaError_t prepare_ntt_cc(const hefx_params* p, NttMode mode) {
    static const RowDesc dummy = {};
    cc::KArgs a = {};
    a.err = p->d_err_cc;
    a.desc = &dummy;  // selects the row-list kernels; rows == 0 sets attributes without launching
    return launch_dispatch(p->log2n, p->max_prime, mode, a, 0, nullptr);
}

cudaError_t launch_ntt_cc_rows(const hefx_params* p, uint32_t max_prime, NttMode mode, const RowDesc* d_rows, size_t nrows,
                               cudaStream_t stream) {
    cc::KArgs a;
    memset(&a.tmap_in, 0, sizeof a.tmap_in);
    memset(&a.tmap_out, 0, sizeof a.tmap_out);
    a.err = p->d_err_cc;
    a.in = nullptr;
    a.had = nullptr;
    a.out = nullptr;
    a.tw_f = p->d_tw_fwd;
    a.tw_i = p->d_tw_inv;
    a.lc = p->d_lc;
    a.desc = d_rows;
    a.rows = (uint32_t)nrows;
    a.L = p->nlimbs;
    a.in_rows = 0;
    if (nrows == 0) return cudaSuccess;
    return two_pass(p, mode, nrows) ? launch_two_pass(p->log2n, max_prime, mode, a, nrows, stream)
                                    : launch_dispatch(p->log2n, max_prime, mode, a, nrows, stream);
}

cudaError_t launch_dispatch(uint32_t log2n, uint32_t max_prime, NttMode mode, const cc::KArgs& a, size_t rows,
                            cudaStream_t stream) {
    const bool lazy = max_prime < (1u << 28);
    const int L = (int)log2n;
    if (L >= 3 && L <= 11) return cc::launch_range_a(L, mode, a, rows, stream, lazy);
    if (L >= 12 && L <= 14) return cc::launch_range_b(L, mode, a, rows, stream, lazy);
    if (L == 15) return cc::launch_range_c(L, mode, a, rows, stream, lazy);
    if (L == 16) return cc::launch_range_d(L, mode, a, rows, stream, lazy);
    if (L == 17) return cc::launch_range_e(L, mode, a, rows, stream, lazy);
    return cudaErrorInvalidValue;
}

}  // namespace hefx
