// Self-test of the bounded device-side wait: one thread waits, with the same wait routine the attention
// kernel uses, on an mbarrier that nothing ever arrives on, each time until the wait gives up, and again until
// `limit_ns` have passed.  It then records PEVLM_ETIMEOUT and the id of the wait in the workspace header exactly as the
// attention kernel does, and the kernel ends normally: no trap, no fault, the context stays usable.
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

constexpr int kWaitSelfTest = 99;  // wait id reported in the detail word: 99 * 1000000 + CTA index

__global__ void wait_selftest_kernel(WorkspaceHeader* hdr, uint32_t limit_ns) {
    __shared__ uint64_t bar;
    __shared__ WaitState state;
    if (threadIdx.x == 0) {
        state.tries = kGraceTries;
        state.expired = 0;
        mbar_init(smem_u32(&bar), 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t t0 = globaltimer_lo();
        do mbar_wait(smem_u32(&bar), 0, state, kWaitSelfTest);  // gives up after a few tries
        while (globaltimer_lo() - t0 < limit_ns);
        if (state.expired != 0 && atomicCAS(&hdr->status, 0, PEVLM_ETIMEOUT) == 0) hdr->detail = state.expired * 1000000 + blockIdx.x;
    }
}

cudaError_t launch_wait_selftest(WorkspaceHeader* hdr, uint32_t limit_ns, cudaStream_t stream) {
    wait_selftest_kernel<<<1, 32, 0, stream>>>(hdr, limit_ns);
    return cudaGetLastError();
}

}  // namespace pevlm
