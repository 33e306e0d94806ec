// KV-cache assembly (the key/value set s + c_all + q of Eq. 5): a coalesced 16-byte-vector
// copy of up to four segments (K video, K question, V video, V question) into the two
// contiguous caches, one launch.  Pure HBM traffic: reads and writes each byte once.
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 4;

// An ordinary load, not one through the non-coherent path (.nc): this kernel may be on the GPU while the one that writes its
// sources still runs (launch_chained), and grid_wait() orders ordinary accesses only.
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) {
    asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// The segments are indexed where they are, in the parameters: a copy of them that the thread changes (to the sequence's own
// addresses) ends up in local memory, with a load from it before every access.  K and V of 15,360 tokens of 4 heads of 128
// 6.4 us (20.9 with such a copy), of 50,000 tokens 34.2 (54.2) = 6.0 TB/s.
// The first addresses are formed before the next kernel may come and before the wait, since they take a chain of reads of the
// parameters: a decode step, whose copy is one row, 24.97 us; 25.73 with the next kernel let in first, 26.08 with the wait
// first as well, 25.54 with the next kernel let in after the wait.
__global__ void __launch_bounds__(kCopyThreads) copy_segments_kernel(const __grid_constant__ CopySegments s) {
    const int64_t seq = blockIdx.y;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kCopyThreads * kCopyUnroll;
    bool waited = false;
    for (int64_t base = static_cast<int64_t>(blockIdx.x) * kCopyThreads * kCopyUnroll + threadIdx.x; base < s.total;
         base += stride) {
        const uint4* src[kCopyUnroll];
        uint4* dst[kCopyUnroll];
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u) {
            int64_t i = base + static_cast<int64_t>(u) * kCopyThreads;
            dst[u] = nullptr;
            if (i < s.total) {
                int seg = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if (seg == k && i >= s.n_vec[k]) {
                        i -= s.n_vec[k];
                        seg = k + 1;
                    }
                }
                src[u] = s.src[seg] + seq * s.src_stride[seg] + i;
                dst[u] = s.dst[seg] + seq * s.dst_stride + i;
            }
        }
        if (!waited) {
            grid_launch_dependents();
            grid_wait();
        }
        waited = true;
        uint4 v[kCopyUnroll];
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u)
            if (dst[u]) v[u] = ld_stream(src[u]);
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u)
            if (dst[u]) st_stream(dst[u], v[u]);
    }
    if (!waited) grid_wait();
}

cudaError_t launch_copy_segments(const CopySegments& s, cudaStream_t stream) {
    if (s.total <= 0) return cudaSuccess;
    const int64_t per_cta = static_cast<int64_t>(kCopyThreads) * kCopyUnroll;
    int64_t ctas = (s.total + per_cta - 1) / per_cta;
    const int64_t cap = 148 * 16;  // a few waves of the 148 SMs; the loop strides over the rest
    if (ctas > cap) ctas = cap;
    return launch_chained<copy_segments_kernel>(dim3(static_cast<unsigned>(ctas), static_cast<unsigned>(s.batch)), kCopyThreads, 0, stream, s);
}

}  // namespace pevlm
