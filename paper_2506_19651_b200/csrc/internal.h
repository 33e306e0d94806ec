// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/pevlm.h"

namespace pevlm {

constexpr int kTile = 128;        // query-tile rows (MMA M) and key-tile columns (MMA N max)
constexpr int kStatusBytes = 256; // first bytes of every workspace: status word + detail
constexpr int kNumSms = 148;      // B200; used only to size the key splits of the question attention

// Workspace header (device memory, first kStatusBytes of the workspace).
struct WorkspaceHeader {
    int32_t status;  // 0 or PEVLM_ETIMEOUT
    int32_t detail;  // which wait expired (kernel-specific code)
    int32_t pad[62];
};

// a / b for 0 <= a < 2^31 without a divide: (a * mul) >> (31 + shift), shift = ceil(log2 b), mul = ceil(2^(31 + shift) / b)
// < 2^32.  Exact: mul exceeds 2^(31 + shift) / b by less than 1, which adds less than a / 2^(31 + shift) < 1 / b.
struct Divisor {
    uint32_t mul;
    uint32_t shift;
};
inline Divisor make_divisor(int b) {  // b = 0 (a quantity the launch does not use) gives quotient 0
    Divisor d{0, 0};
    if (b <= 0) return d;
    while ((1ll << d.shift) < b) ++d.shift;
    d.mul = static_cast<uint32_t>(((1ull << (31 + d.shift)) + static_cast<uint64_t>(b) - 1) / static_cast<uint64_t>(b));
    return d;
}

#ifdef __CUDACC__
__device__ __forceinline__ int quotient(int a, const Divisor& b) {
    return static_cast<int>((static_cast<uint64_t>(static_cast<uint32_t>(a)) * b.mul) >> 31 >> b.shift);
}
#endif

// The calling thread's context: a number that no other context of the process ever has; 0 if it has none yet (or if the driver does not say).
uint64_t context_id();

// Launch of one of the library's kernels behind another.  The kernel may be brought onto the GPU while the one before it
// in the stream still runs, so that its launch costs nothing; every kernel therefore calls grid_wait() before it reads or writes
// global memory (the decode kernel prefetches keys into L2 before, which reads nothing into registers or shared memory).  Most let the next kernel come before their own wait; the decode kernel and the merge only after it,
// because the launches behind them would otherwise arrive two steps early and hold the SMs that the step needs whole
// (a decode step 25.2 us so, 27.4 with all of them early, 26.5 with none).  All kernels ask for the same split of the SM's memory (as much shared memory as there is), because an
// SM has to run empty before it can change the split.
template <auto Kernel, typename... Args>
inline cudaError_t launch_chained(dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, const Args&... args) {
    // attributes of a kernel: once in each context (a second one on a device, or the one after a reset, has its own; smem
    // is the same in every launch of a kernel).  Contexts whose ids share a place take turns in it.
    static std::atomic<uint64_t> prepared[64] = {};
    const uint64_t context = context_id();
    std::atomic<uint64_t>& place = prepared[context % 64];
    cudaError_t e = cudaSuccess;
    if (context == 0 || place.load(std::memory_order_acquire) != context) {
        e = cudaFuncSetAttribute(Kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e == cudaSuccess && smem > 48 * 1024)
            e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        place.store(context, std::memory_order_release);
    }
    cudaLaunchAttribute chained;
    chained.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    chained.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config{};
    config.gridDim = grid;
    config.blockDim = dim3(threads);
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &chained;
    config.numAttrs = 1;
    e = cudaLaunchKernelEx(&config, Kernel, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// How the query tiles of one position of a segment follow one another: `toks` tokens of `heads` q heads of one kv group
// each (a full position: 128 of one), the next tile head_step heads or tok_step tokens on.
struct QTile {
    int32_t heads, toks, head_step, tok_step, box_rows;
};

// One kind of prefill segment (full context blocks, a shorter last block, the sink) and its work items.
struct Segment {
    int32_t items;       // work items, padded: (per_chunk =) blocks * Hkv * pair_chunk, times chunks
    int32_t len;         // tokens of a segment
    int32_t q0;          // row of q / o where the first one starts
    int32_t key0;        // row where the first one starts in the tensor map of its keys
    int32_t a_end;       // keys of the shared range (the sink) that its rows see
    int32_t own_map;     // which K / V map its own keys are in: 0 blocks, 1 sink
    int32_t full_tiles;  // query tile positions without the packed tail
    int32_t entries;     // query tiles of one (segment, kv head): tail_tiles + G * full_tiles
    int32_t tail_tiles;  // tiles of a ragged last position (len % 128 rows) whose rows are packed; 0 = no packing
    QTile form[2];       // of a full position, of a packed tail
    int32_t pair_chunk;  // pairs of one (segment, kv head) handed out together (see decode_item)
    int32_t per_chunk;
    Divisor div_per_chunk, div_pair_chunk;
};

// What one launch of the attention kernel does, bit 0 of mode: prefill rows (sink + blocks, or full causal); bit 1:
// question rows against the assembled cache, split over keys.
struct AttnParams {
    int32_t mode;
    int32_t batch;          // sequences, each with n_items work items
    Segment seg[3];         // prefill: full blocks (full causal: the whole stream as one), shorter last block, sink
    int32_t n_video;        // S + N*B (+ the last block)
    int32_t sink_len;       // prefill (host only): S,
    int32_t block_rows;     // rows of all blocks
    int32_t blk_key0;       // and K/V row of the first block (S, or the cache row of a block range)
    int32_t q_rows;         // prefill: rows of q / o (and columns of lse) of a sequence
    int32_t kv_rows;        // prefill (host only): rows of k / v of a sequence
    int32_t Q, L;           // question length, total length
    int32_t Hq, Hkv, G;
    int32_t items_question; // question work items
    int32_t n_items;        // all work items of a sequence
    int32_t tok_per_tile;   // question: tokens per query tile = 128 / G
    int32_t q_tiles;        // question: ceil(Q / tok_per_tile)
    int32_t n_splits;       // question
    int32_t tiles_per_split;// question
    Divisor div_items, div_hkv, div_g, div_splits, div_q_pairs;  // decode_item
    int32_t wait_tries;     // limit of a single device-side wait before the launch reports PEVLM_ETIMEOUT
    float scale;            // softmax scale
    float scale_log2;       // scale * log2(e)
    __nv_bfloat16* o;       // prefill: [batch * q_rows, Hq, d]
    float* lse;             // prefill: [batch, Hq, q_rows] or NULL
    __nv_bfloat16* o_question;  // question, n_splits = 1: [batch, Q, Hq, d]
    float* lse_question;        // and [batch, Hq, Q] or NULL
    float* part_o;          // question, n_splits > 1: [batch, n_splits, Q, Hq, d] fp32
    float* part_lse;        // and [batch, n_splits, Q, Hq]
    WorkspaceHeader* hdr;
    WorkspaceHeader* hdr_question;  // mode 3: header of the question's workspace
    int32_t keep_status;    // a later launch of the same call
};

constexpr int kMergeRows = 8 * kNumSms;  // most rows of the merge that takes a CTA for each (as many as are resident)
constexpr int kDecodeRows = 32;  // most rows (question tokens x heads of a kv group) of the decode kernel

// Question attention of a few rows, see decode_kernel.cu.
struct DecodeParams {
    const __nv_bfloat16* q;  // [batch, Q, Hq, d]
    const __nv_bfloat16* k;  // [batch, L, Hkv, d]
    const __nv_bfloat16* v;
    float* part_o;           // [batch, n_splits, Q, Hq, d]
    float* part_lse;         // [batch, n_splits, Q, Hq]
    WorkspaceHeader* hdr;
    int32_t batch, Q, L, n_video, Hq, Hkv, G;
    int32_t pieces;            // ceil(L / 16)
    int32_t pieces_per_split;
    int32_t n_splits;
    float scale, scale_log2;
};

struct MergeParams {
    int32_t batch, Q, Hq, d, n_splits;
    const float* part_o;
    const float* part_lse;
    __nv_bfloat16* o;  // [batch, Q, Hq, d]
    float* lse;        // [batch, Hq, Q] or NULL
};

struct RopeParams {
    double inv_freq[64];  // theta^(-2i/d), i < d/2, computed on the host in fp64
    const __nv_bfloat16* q_in;
    const __nv_bfloat16* k_in;
    __nv_bfloat16* q_out;
    __nv_bfloat16* k_out;
    const int32_t* pos_ids;
    int64_t first_token;
    int64_t n_tokens;
    int32_t Hq, Hkv;  // heads to process of each tensor (0 = skip tensor)
    // q rows of tokens from split_token on go to the same place counted from q_out2
    __nv_bfloat16* q_out2;
    int64_t split_token;
    const __nv_bfloat16* v_in;  // rows copied along: Hv heads of v_in to v_out (0 = none)
    __nv_bfloat16* v_out;
    int32_t Hv;
    int32_t seq_len;  // tokens of a sequence, n_tokens = batch * seq_len (pos_ids [batch, seq_len], pos3 [batch, 3, seq_len])
    Divisor div_seq;
    int32_t group;  // tokens per CTA (this and the divisors are set by launch_rope)
    Divisor div_hq, div_hkv;
    // multimodal RoPE: pos3 != NULL selects it; rotary pair i takes its position from component 0 for
    // i < sec_end0, component 1 for i < sec_end1, else component 2
    const int32_t* pos3;
    int32_t sec_end0, sec_end1;
};

struct CopySegments {
    const uint4* src[4];
    uint4* dst[4];
    int64_t n_vec[4];  // 16-byte vectors per segment
    int64_t total;
    int64_t src_stride[4], dst_stride;  // vectors from one sequence to the next
    int32_t batch;
};

cudaError_t launch_rope(const RopeParams& p, int head_dim, cudaStream_t stream);
// tokens of a group of such a call, heads of V counted (not part of the ABI: the tests ask for it)
extern "C" int pevlm_rope_group_size(int64_t n_tokens, int heads, int head_dim);
cudaError_t launch_copy_segments(const CopySegments& s, cudaStream_t stream);
// Tensor maps of one attention launch.
//   q[0]: [rows, Hq, d] with a 128-token box; q[1 + kind]: the same tensor with the box of the segment kind's packed ragged
//   tail (heads x tail rows); q[4]: the question rows (box: one kv group's heads x the tokens of a tile)
//   k, v[0]: the context blocks of the call (base at the first block's row); [1]: the sink, rows [0, S), so that a ragged
//   last key tile of either range reads zeros past its end instead of a neighbour's rows; [2]: the whole cache.  The
//   sequences of a batch are the maps' last dimension, so that the end of the range is the end of the map in each of them
struct AttnMaps {
    CUtensorMap q[5], k[3], v[3];
};
cudaError_t launch_attn(const AttnParams& p, int head_dim, const AttnMaps& m, cudaStream_t stream);
cudaError_t launch_wait_selftest(WorkspaceHeader* hdr, uint32_t limit_ns, cudaStream_t stream);
// device address of the built-in scratch array of pevlm_query_attn_noalloc on the current device
int noalloc_scratch_for_current_device(void** out);
size_t query_workspace_bytes(const pevlm_shape_t* s);  // of pevlm_query_attn
int check_query_args(const pevlm_shape_t* s, const void* q_question, const void* k_cache, const void* v_cache,
                     const void* o, const float* lse);
cudaError_t launch_decode(const DecodeParams& p, int head_dim, cudaStream_t stream);
cudaError_t launch_merge(const MergeParams& p, cudaStream_t stream);
// error reporting shared by the host-side translation units: both record a text that
// pevlm_last_cuda_error returns on the calling thread
int cuda_fail(cudaError_t e, const char* what);      // returns PEVLM_ECUDA
int fail_with_text(int code, const char* text);      // returns code

}  // namespace pevlm
