// LSE merge of the key-range partials of the question attention (Eq. 5): each split s left
// a locally normalised output o_s and lse_s for every question row; the whole-range result is
//   lse = log sum_s exp(lse_s),   o = sum_s exp(lse_s - lse) o_s.
// A split with no visible key for a row has lse_s = -inf and contributes nothing.
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

constexpr int kMergeThreads = 256;
constexpr int kMergeChunk = 8;       // partial rows of a warp whose loads are in flight together
// most splits of the form for few rows (its weights are an array in shared memory).  The tile kernel alone and the decode kernel
// make 148 at most; beside a prefill part there can be more (one kv head, 1,024 question tokens, 1.3M keys: 161), which
// launch_merge gives to the other form
constexpr int kMergeMaxParts = 160;

// Many rows (a prefill-sized question block): one thread per (row, 4 output columns), the splits one after
// another; tens of thousands of threads hide the latency of the dependent loads.
__global__ void merge_kernel(MergeParams p) {
    grid_wait();
    grid_launch_dependents();
    const int vec_per_row = p.d / 4;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t rows = static_cast<int64_t>(p.Q) * p.Hq;
    if (idx >= rows * vec_per_row) return;
    const int64_t row = idx / vec_per_row;  // = tok * Hq + head
    const int v = static_cast<int>(idx % vec_per_row);
    const int n = p.n_splits;
    const int64_t seq = blockIdx.y;
    p.part_o += seq * n * rows * p.d;
    p.part_lse += seq * n * rows;
    p.o += seq * rows * p.d;
    if (p.lse) p.lse += seq * rows;
    float m = -INFINITY;
    for (int s = 0; s < n; ++s) m = fmaxf(m, p.part_lse[s * rows + row]);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.f;
    if (m != -INFINITY) {
        for (int s = 0; s < n; ++s) {
            const float ls = p.part_lse[s * rows + row];
            if (ls == -INFINITY) continue;
            const float w = __expf(ls - m);
            l += w;
            const float4 o = reinterpret_cast<const float4*>(p.part_o + (s * rows + row) * p.d)[v];
            acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        }
    }
    const float inv = (l > 0.f) ? 1.f / l : 0.f;
    uint2 out;
    out.x = pack_bf16x2(acc.x * inv, acc.y * inv);
    out.y = pack_bf16x2(acc.z * inv, acc.w * inv);
    reinterpret_cast<uint2*>(p.o + row * p.d)[v] = out;
    if (p.lse && v == 0) {
        const int tok = static_cast<int>(row / p.Hq), head = static_cast<int>(row % p.Hq);
        p.lse[static_cast<int64_t>(head) * p.Q + tok] = (l > 0.f) ? m + logf(l) : -INFINITY;
    }
}

// Few rows (a decode step has Hq of them): one CTA per question row (token, head).  With few rows the time is the chain of
// dependent L2 round trips, so there is only one: every warp takes all lse_s of the row (lane l splits l, l + 32, ...) and,
// at the same time, its share of the partial rows (warp w splits w, w + 8, ..., kMergeChunk of them in flight; lane l output
// columns [4l, 4l + 4), lanes 0-15 at d = 64), and the warps' sums meet in shared memory.  (One warp per row, with the
// chunks of partial rows one after another, took 4-5 us behind a decode step of 37 splits.)
__global__ void __launch_bounds__(kMergeThreads) merge_rows_kernel(MergeParams p) {
    __shared__ float4 sums[kMergeThreads / 32][32];
    __shared__ float weights[kMergeMaxParts];
    grid_wait();
    grid_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = blockIdx.x, rows = static_cast<int64_t>(p.Q) * p.Hq, seq = blockIdx.y;
    const int n = p.n_splits;
    p.part_o += seq * n * rows * p.d;
    p.part_lse += seq * n * rows;
    const bool col_ok = lane * 4 < p.d;
    constexpr int kWarps = kMergeThreads / 32;
    auto load_chunk = [&](int s0, float4 (&o)[kMergeChunk]) {
#pragma unroll
        for (int u = 0; u < kMergeChunk; ++u) {
            const int s = s0 + u * kWarps;
            o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (s < n && col_ok) o[u] = __ldcg(reinterpret_cast<const float4*>(p.part_o + (s * rows + row) * p.d) + lane);
        }
    };
    float4 o[kMergeChunk];
    load_chunk(warp, o);
    float ls[kMergeMaxParts / 32], m = -INFINITY;
#pragma unroll
    for (int i = 0; i < kMergeMaxParts / 32; ++i) {
        ls[i] = lane + 32 * i < n ? __ldcg(p.part_lse + (lane + 32 * i) * rows + row) : -INFINITY;
        m = fmaxf(m, ls[i]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    float l = 0.f;
#pragma unroll
    for (int i = 0; i < kMergeMaxParts / 32; ++i) {
        const float e = ls[i] == -INFINITY ? 0.f : __expf(ls[i] - m);  // an empty split contributes nothing
        if (warp == 0) weights[lane + 32 * i] = e;
        l += e;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    __syncthreads();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = warp; s0 < n; s0 += kMergeChunk * kWarps) {
        if (s0 != warp) load_chunk(s0, o);
#pragma unroll
        for (int u = 0; u < kMergeChunk; ++u) {
            const float wt = s0 + u * kWarps < n ? weights[s0 + u * kWarps] : 0.f;
            if (wt == 0.f) continue;  // an empty split's partial row is zero anyway
            acc.x += wt * o[u].x; acc.y += wt * o[u].y; acc.z += wt * o[u].z; acc.w += wt * o[u].w;
        }
    }
    sums[warp][lane] = acc;
    __syncthreads();
    if (warp != 0) return;
    const float inv = (l > 0.f) ? 1.f / l : 0.f;
    if (col_ok) {
#pragma unroll
        for (int w = 1; w < kWarps; ++w) {
            const float4 x = sums[w][lane];
            acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
        }
        uint2 out;
        out.x = pack_bf16x2(acc.x * inv, acc.y * inv);
        out.y = pack_bf16x2(acc.z * inv, acc.w * inv);
        reinterpret_cast<uint2*>(p.o + (seq * rows + row) * p.d)[lane] = out;
    }
    if (p.lse && lane == 0) {
        const int tok = static_cast<int>(row / p.Hq), head = static_cast<int>(row % p.Hq);
        p.lse[seq * rows + static_cast<int64_t>(head) * p.Q + tok] = (l > 0.f) ? m + logf(l) : -INFINITY;
    }
}

cudaError_t launch_merge(const MergeParams& p, cudaStream_t stream) {
    const int64_t rows = static_cast<int64_t>(p.Q) * p.Hq;
    if (rows <= 0) return cudaSuccess;
    const unsigned batch = static_cast<unsigned>(p.batch);
    // few rows: the latency-oriented form
    if (rows * batch <= kMergeRows && p.n_splits <= kMergeMaxParts)
        return launch_chained<merge_rows_kernel>(dim3(static_cast<unsigned>(rows), batch), kMergeThreads, 0, stream, p);
    const int64_t n = rows * (p.d / 4);
    return launch_chained<merge_kernel>(dim3(static_cast<unsigned>((n + kMergeThreads - 1) / kMergeThreads), batch), kMergeThreads, 0,
                          stream, p);
}

}  // namespace pevlm
