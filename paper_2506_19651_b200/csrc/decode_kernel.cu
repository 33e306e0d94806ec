// Question attention of a few rows (Eq. 5 with a decode-sized question): the group's heads x the question's tokens make at
// most 32 rows per kv head, so the step is one pass over the K/V cache and bound by HBM alone.
//
// The tile kernel (attn_kernel.cu) spends 128-row tiles and a softmax of 128 x 128 scores on 7 rows and holds a pair of SMs
// per item: 30 us for a 103 MB cache that takes 16 us to read.  Here a CTA takes one kv head and one range of keys; its
// eight warps take the 16-key pieces of the range in turn, each with a private ring of stages in shared memory that it
// fills by cp.async and reads itself, so no warp ever waits for another and no barrier stands in the loop: 128 KB are in
// flight per SM.  Per piece a warp forms S = Q K^T and O += P V with mma.sync m16n8k16 (its 16 rows are the question's,
// two such tiles above 16 rows; operands of this size are nowhere near a bound, and tcgen05's smallest tile is 128 rows), with a running reference maximum that
// moves only when it grows by more than 2^8.  At the end the warps' (m, l, O) are merged in shared memory and the CTA
// leaves one partial for the merge of the splits.
// Measured (B200, whole call with the merge, back to back): 50K keys, 28/4 heads of 128, one token 36.3 -> 23.1 us
// (4.5 TB/s of cache), four tokens 36.5 -> 28.5; 12.5K keys 22.7 -> 11.2; heads of 64 45.9 -> 21.5.  Above 32 rows the
// tile kernel is the faster one (56 rows at 50K keys: 33.8 us, and it needs no accumulator of rows x head size per warp).
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

constexpr int kDecodeThreads = 256;
constexpr int kDecodeWarps = kDecodeThreads / 32;
constexpr int kPiece = 16;  // keys a warp takes at a time
constexpr int kEarlyPieces = 8;  // of a warp, fetched into L2 ahead (50K keys: a step takes 27.2 us with 0, 26.7 with 4, 26.4 with 8)

// MT: 16-row tiles
template <int D, int MT>
struct DecodeSmem {
    static constexpr int kRows = 16 * MT;
    static constexpr int kStageBytes = 2 * kPiece * D * 2;                      // K and V rows of a piece
    static constexpr int kStages = D == 128 ? 3 : 6;
    static constexpr int kRingBytes = kDecodeWarps * kStages * kStageBytes;     // 192 KB
    static constexpr int kQBytes = kRows * D * 2;                               // behind the rings
    static constexpr int kMergeBytes = kDecodeWarps * kRows * (D + 2) * 4;      // overlays the rings
    static constexpr int kTotal = kRingBytes + kQBytes;
    static_assert(kMergeBytes <= kRingBytes, "merge area");
};

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int D, int MT>
__global__ void __launch_bounds__(kDecodeThreads, 1) decode_kernel(const __grid_constant__ DecodeParams p) {
    using L = DecodeSmem<D, MT>;
    constexpr int ROWS = L::kRows;
    constexpr int CH = D / 8;          // 16-byte chunks of a row; stored at chunk ^ (row & 7)
    constexpr int ROW = D * 2;
    extern __shared__ __align__(128) uint8_t raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = blockIdx.x, g = blockIdx.y;
    const int64_t seq = blockIdx.z;
    const uint32_t ring = smem_u32(raw) + warp * L::kStages * L::kStageBytes;
    const int piece0 = split * p.pieces_per_split;
    const int pieces = min(p.pieces_per_split, p.pieces - piece0);
    const int mine = pieces > warp ? (pieces - warp + kDecodeWarps - 1) / kDecodeWarps : 0;  // pieces of this warp
    const int64_t row_stride = static_cast<int64_t>(p.Hkv) * D;
    const __nv_bfloat16* k = p.k + seq * p.L * row_stride + g * D;
    const __nv_bfloat16* v = p.v + seq * p.L * row_stride + g * D;
    // While the kernels before this one finish (a decode step's RoPE and copy of one token leave nearly all SMs idle), the
    // first pieces are brought into L2: that reads nothing, so what those kernels still write is seen all the same.
    for (int n = 0; n < min(mine, kEarlyPieces); ++n) {
        const int key0 = (piece0 + warp + n * kDecodeWarps) * kPiece;
        constexpr int kLines = D * 2 / 128;  // lines of a row
        for (int i = lane; i < kPiece * kLines; i += 32) {
            const int64_t key = min(key0 + i / kLines, p.L - 1);
            const int64_t off = key * row_stride + i % kLines * 64;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(k + off));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(v + off));
        }
    }
    grid_wait();
    grid_launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0) p.hdr->status = p.hdr->detail = 0;

    auto fetch = [&](int n) {  // the warp's n-th piece
        if (n < mine) {
            const int key0 = (piece0 + warp + n * kDecodeWarps) * kPiece;
            const uint32_t stage = ring + (n % L::kStages) * L::kStageBytes;
#pragma unroll
            for (int i = 0; i < kPiece * CH / 32; ++i) {
                const int row = (i * 32 + lane) / CH, c = lane % CH;
                const int64_t key = key0 + row;
                const uint32_t dst = stage + row * ROW + ((c ^ (row & 7)) << 4);
                const int n_bytes = key < p.L ? 16 : 0;  // past the end: zeros
                const int64_t off = (key < p.L ? key : 0) * row_stride + c * 8;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(k + off), "r"(n_bytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + kPiece * ROW), "l"(v + off), "r"(n_bytes) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int n = 0; n < L::kStages - 1; ++n) fetch(n);

    // the rows: r -> token r / G, head g * G + r % G; in shared memory like K (rows that do not exist are zeros).  This
    // thread holds parts of rows r0 + 8 h of every tile
    const int r0 = lane >> 2, rows = p.Q * p.G;
    const uint32_t sq = smem_u32(raw) + L::kRingBytes;
    for (int i = tid; i < ROWS * CH; i += kDecodeThreads) {
        const int r = i / CH, c = i % CH, tok = r / p.G;
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (r < rows) x = *reinterpret_cast<const uint4*>(p.q + ((seq * p.Q + tok) * p.Hq + g * p.G + (r - tok * p.G)) * D + c * 8);
        *reinterpret_cast<uint4*>(raw + L::kRingBytes + r * ROW + ((c ^ (r & 7)) << 4)) = x;
    }
    int limit[MT][2];  // last visible key
    float o[MT][D / 8][4], m[MT][2], l[MT][2];
#pragma unroll
    for (int t = 0; t < MT; ++t) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            limit[t][h] = p.n_video + (16 * t + 8 * h + r0) / p.G;
            m[t][h] = -INFINITY;
            l[t][h] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < D / 8; ++i) o[t][i][0] = o[t][i][1] = o[t][i][2] = o[t][i][3] = 0.f;
    }
    __syncthreads();
    const int mat = lane >> 3, mrow = lane & 7;  // ldmatrix: this lane's matrix and row
    for (int n = 0; n < mine; ++n) {
        fetch(n + L::kStages - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(L::kStages - 1) : "memory");
        __syncwarp();
        const uint32_t stage = ring + (n % L::kStages) * L::kStageBytes;
        const int key0 = (piece0 + warp + n * kDecodeWarps) * kPiece;
        float s[MT][2][4] = {};  // keys [0, 8) and [8, 16)
        const int krow = (mat >> 1) * 8 + mrow, vrow = (mat & 1) * 8 + mrow;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            uint32_t b[4], a[4];
            ldmatrix4(b, stage + krow * ROW + (((2 * ks + (mat & 1)) ^ (krow & 7)) << 4));
#pragma unroll
            for (int t = 0; t < MT; ++t) {
                const int qrow = 16 * t + vrow;
                ldmatrix4(a, sq + qrow * ROW + (((2 * ks + (mat >> 1)) ^ (qrow & 7)) << 4));
                mma16816(s[t][0], a, b[0], b[1]);
                mma16816(s[t][1], a, b[2], b[3]);
            }
        }
        uint32_t pa[MT][4];
#pragma unroll
        for (int t = 0; t < MT; ++t) {
            if (key0 + kPiece > p.n_video) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (key0 + i * 8 + (lane & 3) * 2 + (e & 1) > limit[t][e >> 1]) s[t][i][e] = -INFINITY;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float mt = fmaxf(fmaxf(s[t][0][2 * h], s[t][0][2 * h + 1]), fmaxf(s[t][1][2 * h], s[t][1][2 * h + 1]));
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
                const bool moves = (mt - m[t][h]) * p.scale_log2 > 8.f || (m[t][h] == -INFINITY && mt != -INFINITY);
                if (__any_sync(0xffffffffu, moves)) {
                    const float alpha = moves ? fast_exp2((m[t][h] - mt) * p.scale_log2) : 1.f;
                    if (moves) m[t][h] = mt;
                    l[t][h] *= alpha;
#pragma unroll
                    for (int i = 0; i < D / 8; ++i) {
                        o[t][i][2 * h] *= alpha;
                        o[t][i][2 * h + 1] *= alpha;
                    }
                }
                const float neg = m[t][h] == -INFINITY ? 0.f : -m[t][h] * p.scale_log2;
                float e[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) e[i] = fast_exp2(fmaf(s[t][i >> 1][2 * h + (i & 1)], p.scale_log2, neg));
                l[t][h] += (e[0] + e[1]) + (e[2] + e[3]);
                pa[t][h] = pack_bf16x2(e[0], e[1]);
                pa[t][2 + h] = pack_bf16x2(e[2], e[3]);
            }
        }
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
            uint32_t b[4];
            ldmatrix4_trans(b, stage + kPiece * ROW + vrow * ROW + (((2 * c + (mat >> 1)) ^ (vrow & 7)) << 4));
#pragma unroll
            for (int t = 0; t < MT; ++t) {
                mma16816(o[t][2 * c], pa[t], b[0], b[1]);
                mma16816(o[t][2 * c + 1], pa[t], b[2], b[3]);
            }
        }
        __syncwarp();  // every lane has read the stage before it is filled again
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // merge of the warps: (m, l) and O through shared memory, over the rings
    float* so = reinterpret_cast<float*>(raw);                                  // [warp][row][D]
    float* sm = so + kDecodeWarps * ROWS * D;                            // [warp][row]
    float* sl = sm + kDecodeWarps * ROWS;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < MT; ++t) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            l[t][h] += __shfl_xor_sync(0xffffffffu, l[t][h], 1);
            l[t][h] += __shfl_xor_sync(0xffffffffu, l[t][h], 2);
            const int r = 16 * t + 8 * h + r0;
            if ((lane & 3) == 0) {
                sm[warp * ROWS + r] = m[t][h];
                sl[warp * ROWS + r] = l[t][h];
            }
#pragma unroll
            for (int i = 0; i < D / 8; ++i)
                *reinterpret_cast<float2*>(so + (warp * ROWS + r) * D + i * 8 + (lane & 3) * 2) = make_float2(o[t][i][2 * h], o[t][i][2 * h + 1]);
        }
    }
    __syncthreads();
    for (int i = tid; i < rows * (D / 4); i += kDecodeThreads) {
        const int r = i / (D / 4), c = i % (D / 4), tok = r / p.G;
        float mx = -INFINITY, sum = 0.f;
#pragma unroll
        for (int w = 0; w < kDecodeWarps; ++w) mx = fmaxf(mx, sm[w * ROWS + r]);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (mx != -INFINITY) {
#pragma unroll
            for (int w = 0; w < kDecodeWarps; ++w) {
                const float f = fast_exp2((sm[w * ROWS + r] - mx) * p.scale_log2);
                sum += f * sl[w * ROWS + r];
                const float4 x = *reinterpret_cast<const float4*>(so + (w * ROWS + r) * D + c * 4);
                acc.x += f * x.x; acc.y += f * x.y; acc.z += f * x.z; acc.w += f * x.w;
            }
        }
        const float inv = sum > 0.f ? 1.f / sum : 0.f;
        const int64_t row = ((seq * p.n_splits + split) * p.Q + tok) * p.Hq + g * p.G + (r - tok * p.G);
        reinterpret_cast<float4*>(p.part_o + row * D)[c] = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        if (c == 0) p.part_lse[row] = sum > 0.f ? mx * p.scale + logf(sum) : -INFINITY;
    }
}

cudaError_t launch_decode(const DecodeParams& p, int head_dim, cudaStream_t stream) {
    const dim3 grid(static_cast<unsigned>(p.n_splits), static_cast<unsigned>(p.Hkv), static_cast<unsigned>(p.batch));
    const bool two = p.Q * p.G > 16;
    if (head_dim == 128)
        return two ? launch_chained<decode_kernel<128, 2>>(grid, kDecodeThreads, DecodeSmem<128, 2>::kTotal, stream, p)
                   : launch_chained<decode_kernel<128, 1>>(grid, kDecodeThreads, DecodeSmem<128, 1>::kTotal, stream, p);
    return two ? launch_chained<decode_kernel<64, 2>>(grid, kDecodeThreads, DecodeSmem<64, 2>::kTotal, stream, p)
               : launch_chained<decode_kernel<64, 1>>(grid, kDecodeThreads, DecodeSmem<64, 1>::kTotal, stream, p);
}

}  // namespace pevlm
