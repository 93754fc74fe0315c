// Self-check of the failure-detection path shared by the tcgen05 / TMA kernels: one 32-thread
// block takes TMEM, waits on an mbarrier with the same bounded wait (tc::mbar_wait) the
// pipelines use, then frees TMEM and returns.  With `arrive` the block arrives on the barrier
// first and the wait succeeds; without it nothing ever arrives, the wait gives up after
// `limit_ns` and records tc::ERR_WAIT_CHECK in the parameter set's error flag, which
// hefx_stream_check reports as HEFX_ETIMEOUT.  Nothing else is in flight when the wait gives
// up, so the kernel ends cleanly and the context stays usable.
#include "hefx_internal.h"
#include "tc_common.cuh"

namespace hefx {
namespace {

__global__ void __launch_bounds__(32, 1) wait_check_kernel(uint32_t* err, uint64_t limit_ns, int arrive) {
    __shared__ uint64_t bar;
    __shared__ uint32_t tmem_slot;
    if (threadIdx.x == 0) {
        tc::mbar_init(&bar, 1);
        tc::fence_mbar_init();
    }
    tc::tmem_alloc(&tmem_slot, 32);  // warp-wide; the waiting pipeline role holds TMEM like this
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (threadIdx.x == 0) {
        if (arrive) tc::mbar_arrive(&bar);
        tc::mbar_wait(&bar, 0, err, tc::ERR_WAIT_CHECK, limit_ns);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 32);
}

// The wait of a warp whose lanes go on together (tc::mbar_wait_warp): a lane whose bit of `lanes` is set
// waits on a barrier that has completed, the others on one that nothing arrives on.  Lanes that
// decide differently are recorded as tc::ERR_WAIT_SPLIT.
__global__ void __launch_bounds__(32, 1) wait_check_warp_kernel(uint32_t* err, uint64_t limit_ns, uint32_t lanes) {
    __shared__ uint64_t bar[2];
    if (threadIdx.x == 0) {
        tc::mbar_init(&bar[0], 1);
        tc::mbar_init(&bar[1], 1);
        tc::fence_mbar_init();
        tc::mbar_arrive(&bar[1]);
    }
    __syncthreads();
    const bool ok = tc::mbar_wait_warp(&bar[(lanes >> threadIdx.x) & 1u], 0, err, tc::ERR_WAIT_CHECK, limit_ns);
    const uint32_t went_on = __ballot_sync(0xffffffffu, ok);
    if (threadIdx.x == 0 && went_on != 0u && went_on != 0xffffffffu) atomicExch(err, (uint32_t)tc::ERR_WAIT_SPLIT);
}

}  // namespace

cudaError_t launch_wait_check_warp(uint32_t* err, uint64_t limit_ns, uint32_t lanes, cudaStream_t s) {
    wait_check_warp_kernel<<<1, 32, 0, s>>>(err, limit_ns, lanes);
    return cudaGetLastError();
}

cudaError_t launch_wait_check(uint32_t* err, uint64_t limit_ns, int arrive, cudaStream_t s) {
    wait_check_kernel<<<1, 32, 0, s>>>(err, limit_ns, arrive);
    return cudaGetLastError();
}

}  // namespace hefx
