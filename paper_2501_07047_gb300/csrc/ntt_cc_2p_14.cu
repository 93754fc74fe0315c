// Two-pass transforms of N = 2^14 (the kernels are in ntt_cc_2p.cuh).
#include "ntt_cc_2p.cuh"

namespace hefx {
namespace cc2 {

cudaError_t launch_14(NttMode mode, const KRows& a, size_t rows, cudaStream_t s, bool lazy) {
    return launch_logn<14>(mode, a, rows, s, lazy);
}

}  // namespace cc2
}  // namespace hefx
