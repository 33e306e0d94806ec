// C ABI of the library: argument checking, TMA tensor-map encoding and kernel launches.
// Everything here runs on the host; no device memory is allocated and nothing synchronises
// except pevlm_read_status.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

static thread_local char g_cuda_error[256] = "";

int cuda_fail(cudaError_t e, const char* what) {
    snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", what, cudaGetErrorString(e));
    return PEVLM_ECUDA;
}

int fail_with_text(int code, const char* text) {
    snprintf(g_cuda_error, sizeof(g_cuda_error), "%s", text);
    return code;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }
static bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

static int check_shape(const pevlm_shape_t* s) {
    if (!s) return PEVLM_EINVAL;
    if (s->batch < 1 || s->sink_len < 0 || s->num_blocks < 0 || s->query_len < 0) return PEVLM_EINVAL;
    if (s->num_blocks > 0 && s->block_len < 1) return PEVLM_EINVAL;
    if (s->block_len < 0) return PEVLM_EINVAL;
    if (s->num_q_heads < 1 || s->num_kv_heads < 1 || s->num_q_heads % s->num_kv_heads != 0) return PEVLM_EINVAL;
    if (s->mask_mode != PEVLM_MASK_PEVLM && s->mask_mode != PEVLM_MASK_FULL_CAUSAL) return PEVLM_EINVAL;
    if (!(s->rope_theta > 0.f) || !(s->softmax_scale >= 0.f)) return PEVLM_EINVAL;
    const int64_t L = static_cast<int64_t>(s->sink_len) + static_cast<int64_t>(s->num_blocks) * s->block_len + s->query_len;
    if (L < 1 || L > (1ll << 30)) return PEVLM_EINVAL;
    if (s->head_dim != 64 && s->head_dim != 128) return PEVLM_EUNSUPPORTED;
    if (s->num_q_heads / s->num_kv_heads > kTile) return PEVLM_EUNSUPPORTED;
    return PEVLM_OK;
}

// Video tokens; last_len > 0: the last of the blocks has that many tokens.
static int64_t n_video(const pevlm_shape_t* s, int last_len = 0) {
    return static_cast<int64_t>(s->sink_len) + static_cast<int64_t>(s->num_blocks) * s->block_len - (last_len > 0 ? s->block_len - last_len : 0);
}

// What a device is does not change: looked up once for each.
static int check_device() {
    static std::atomic<uint64_t> good{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 64 && (good.load(std::memory_order_relaxed) >> dev & 1)) return PEVLM_OK;
    int major = 0;
    e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    if (major != 10) return PEVLM_EUNSUPPORTED;
    if (dev < 64) good.fetch_or(1ull << dev, std::memory_order_relaxed);
    return PEVLM_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <typename Fn>
static Fn driver_entry(const char* name) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool found = cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess;
    return found ? reinterpret_cast<Fn>(p) : nullptr;
}

static EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = driver_entry<EncodeTiledFn>("cuTensorMapEncodeTiled");
    return fn;
}

uint64_t context_id() {
    typedef CUresult (*CurrentFn)(CUcontext*);
    typedef CUresult (*IdFn)(CUcontext, unsigned long long*);
    static const CurrentFn current = driver_entry<CurrentFn>("cuCtxGetCurrent");
    static const IdFn id_of = driver_entry<IdFn>("cuCtxGetId");
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (!current || !id_of || current(&c) != CUDA_SUCCESS || !c || id_of(c, &id) != CUDA_SUCCESS) return 0;
    return id + 1;
}

// Tensor map over a [tokens, heads, d] bf16 tensor (d contiguous) with a box of box_elems (64 or 32) elements x
// box_heads x box_tokens and the swizzle of the box's row (128 or 64 bytes) that the MMA descriptors expect; with
// batch > 0 over that many such tensors, seq_tokens rows apart, as a fourth dimension.  Rows past the end of the tensor read as zero.
static int make_tmap(CUtensorMap* m, const void* base, int64_t tokens, int heads, int d, int box_heads, int box_tokens,
                     int box_elems = 64, int batch = 0, int64_t seq_tokens = 0) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled entry point not found");
        return PEVLM_ECUDA;
    }
    const cuuint64_t row = static_cast<cuuint64_t>(d) * 2 * heads;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(tokens), static_cast<cuuint64_t>(batch)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(d) * 2, row, row * static_cast<cuuint64_t>(batch > 1 ? seq_tokens : 1)};
    cuuint32_t box[4] = {static_cast<cuuint32_t>(box_elems), static_cast<cuuint32_t>(box_heads), static_cast<cuuint32_t>(box_tokens), 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, batch > 0 ? 4 : 3, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE,
                     box_elems == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled failed with CUresult %d", static_cast<int>(r));
        return PEVLM_ECUDA;
    }
    return PEVLM_OK;
}

static float resolve_scale(const pevlm_shape_t* s) {
    return s->softmax_scale > 0.f ? s->softmax_scale : 1.0f / sqrtf(static_cast<float>(s->head_dim));
}

// ---- query tiles of one prefill segment (sink or context block) per kv head, shared by the launch and
// the stats.  A segment of `len` tokens has ceil(len/128) tile positions.  The rows of a ragged last one are packed into
// fewer than G tiles where that is possible: all its tokens of as many q heads of the kv group as fit, or all heads and as
// many tokens, whichever takes fewer tiles (80 rows of 7 heads: 5 tiles of 18 tokens; 48 rows: 3, by heads 4), by tokens only
// where that makes a pair of tiles less (3 tiles for 4 of 96 rows and 4 heads were 2 % slower).  28/4 heads, blocks of 80: 49.1 ->
// 42.4 us for 41 of them, of 208: 128 -> 115 us for 51.
struct SegPlan {
    int tiles, tail_tiles, full_tiles, entries, pairs;
    QTile tail;
};

static SegPlan plan_segment(int len, int G) {
    SegPlan s{};
    s.tiles = (len + kTile - 1) / kTile;
    const int rem = len % kTile;
    if (rem > 0 && G > 1) {
        const int heads = kTile / rem < G ? kTile / rem : G, toks = kTile / G < rem ? kTile / G : rem;
        const auto pairs = [&](int tail_tiles) { return (tail_tiles + G * (s.tiles - 1) + 1) / 2; };
        const int by_heads = (G + heads - 1) / heads, by_toks = (rem + toks - 1) / toks;
        if (by_heads <= by_toks && by_heads < G) {
            s.tail_tiles = by_heads;
            s.tail = {heads, rem, heads, 0, heads * rem};
        } else if (by_toks < G && pairs(by_toks) < pairs(G)) {
            s.tail_tiles = by_toks;
            s.tail = {G, toks, 0, toks, G * toks};
        }
    }
    s.full_tiles = s.tiles - (s.tail_tiles > 0 ? 1 : 0);
    s.entries = s.tail_tiles + G * s.full_tiles;
    s.pairs = (s.entries + 1) / 2;
    return s;
}

// ---- question-attention decomposition (shared by the launch, the workspace size and the stats)
struct QueryPlan {
    int tok_per_tile, q_tiles, total_kv_tiles, n_splits, tiles_per_split;
    int pieces, pieces_per_split;  // decode kernel (at most kDecodeRows rows per kv head): 16-key pieces; 0 = tile kernel
};

// Key tiles of the prefill work items (each a pair of query tiles): of the longest one, and of all together, with two
// for the start and the end of each item.
struct PrefillSize {
    int longest;
    int64_t all;
};

static PrefillSize prefill_size(const pevlm_shape_t* s, int last_len) {
    const int G = s->num_q_heads / s->num_kv_heads;
    PrefillSize r{0, 0};
    auto add = [&](int64_t segments, int64_t shared, int64_t len) {
        if (segments <= 0 || len <= 0) return;
        const int64_t a = (shared + kTile - 1) / kTile, n = (len + kTile - 1) / kTile;
        r.all += segments * s->num_kv_heads * ((G * (n * a + n * (n + 1) / 2) + 1) / 2 + 2 * plan_segment(static_cast<int>(len), G).pairs);
        if (a + n > r.longest) r.longest = static_cast<int>(a + n);
    };
    if (s->mask_mode == PEVLM_MASK_FULL_CAUSAL) {
        add(1, 0, n_video(s, last_len));
    } else {
        add(1, 0, s->sink_len);
        add(s->num_blocks - (last_len > 0 ? 1 : 0), s->sink_len, s->block_len);
        add(last_len > 0 ? 1 : 0, s->sink_len, last_len);
    }
    return r;
}

// Most key splits of a question beside a prefill part: a question long enough to be many waves of items by itself gains
// nothing from more of them, and its partials (an fp32 row for each row and split) would outgrow its cache: 256K tokens of
// 28/4 heads against 1M keys asked for 485 GB of workspace with splits of 64 key tiles.
constexpr int kMostQuestionItems = 16 * (kNumSms / 2);
static int most_splits(int groups) { return groups < kMostQuestionItems ? kMostQuestionItems / groups : 1; }

static QueryPlan plan_query(const pevlm_shape_t* s, bool beside_prefill = false, int last_len = 0) {
    QueryPlan q;
    const int G = s->num_q_heads / s->num_kv_heads;
    const int64_t L = n_video(s, last_len) + s->query_len;
    q.tok_per_tile = kTile / G;
    q.q_tiles = (s->query_len + q.tok_per_tile - 1) / q.tok_per_tile;
    q.total_kv_tiles = static_cast<int>((L + kTile - 1) / kTile);
    // Work items are (kv head, pair of query tiles, key split), one for each pair of CTAs, so the split count is chosen
    // to give one full wave of the 74 CTA pairs of a B200: as many splits as fit, never more than there are key tiles.
    const int pairs = (q.q_tiles + 1) / 2;
    const int groups = s->num_kv_heads * (pairs > 0 ? pairs : 1);
    int want = kNumSms / 2 / groups;
    // Keys up to `whole` tiles are not split, and there is nothing to merge.  Measured, whole against split: alone, 4/2 heads
    // and 50 tokens, 4 tiles 6.9 / 7.7 us, 5 tiles 7.7 / 7.8, 6 tiles 8.6 / 8.2; 28/4 heads and 60 tokens, whose merge is one of many
    // rows, 8 tiles 10.3 / 12.7.  Behind prefill items: 5 tiles more than the longest of them 16.6 / 17.5, 7 more 18.2 / 18.6,
    // 9 more 21.0 / 19.2; 200 tokens of 28/4 heads, 8 more 22.0 / 25.3.
    const bool many_rows = static_cast<int64_t>(s->batch) * s->query_len * s->num_q_heads > kMergeRows;
    int whole = many_rows ? 8 : 5;
    if (beside_prefill) {
        // In one launch with the prefill items, which fill in behind them.  Enough items for every pair of CTAs, none
        // longer than 64 key tiles, none shorter than 4; but where the question is the smaller part of the launch, an item
        // may take as long as the launch takes anyway, since it starts first: as a rule no split at all (12.6K tokens
        // 282 -> 277 us, 74K 2,222 -> 2,191; 1.8K tokens 35.2 -> 29.4).
        const PrefillSize pre = prefill_size(s, last_len);
        const int64_t own = static_cast<int64_t>(groups) * q.total_kv_tiles, most = (own + pre.all) / (kNumSms / 2);
        const int per_pair = static_cast<int>((own + kNumSms / 2 - 1) / (kNumSms / 2));
        int tiles = per_pair < 4 ? 4 : per_pair > 64 ? 64 : per_pair;
        if (own <= pre.all && most > tiles) tiles = most < q.total_kv_tiles ? static_cast<int>(most) : q.total_kv_tiles;
        want = (q.total_kv_tiles + tiles - 1) / tiles;
        if (want > most_splits(groups)) want = most_splits(groups);
        whole = pre.longest + (many_rows ? 9 : 7);
    }
    if (q.total_kv_tiles <= whole) want = 1;
    if (want < 1) want = 1;
    if (want > q.total_kv_tiles) want = q.total_kv_tiles;
    q.pieces = q.pieces_per_split = 0;
    if (!beside_prefill && s->query_len * G <= kDecodeRows) {
        // one CTA for every SM, no range shorter than the eight pieces its warps take at a time
        q.pieces = static_cast<int>((L + 15) / 16);
        int64_t splits = kNumSms / (static_cast<int64_t>(s->num_kv_heads) * s->batch);
        if (splits > (q.pieces + 7) / 8) splits = (q.pieces + 7) / 8;
        if (splits < 1) splits = 1;
        q.pieces_per_split = static_cast<int>((q.pieces + splits - 1) / splits);
        q.tiles_per_split = 0;
        q.n_splits = (q.pieces + q.pieces_per_split - 1) / q.pieces_per_split;
        return q;
    }
    if (!beside_prefill && q.total_kv_tiles > whole) {
        // Where one wave of items leaves pairs idle, two waves of shorter ones may be done earlier: as many splits as take
        // the fewest key tiles one after another (and three for the start and the end of each item, four for the merge), if that
        // is a tenth fewer.  20K keys, 28/4 heads: 356 tokens (40 items unsplit, three splits now) 160 -> 118 us, 420 tokens
        // 149 -> 114; 32/8 heads, 300 tokens 162 -> 121; 3K keys stay as they were (26.5, split 28.6).
        const auto steps = [&](int n) {
            return (static_cast<int64_t>(groups) * s->batch * n + kNumSms / 2 - 1) / (kNumSms / 2) * ((q.total_kv_tiles + n - 1) / n + 3) + (n > 1 ? 4 : 0);
        };
        int best = want;
        for (int n = want + 1; n <= kNumSms / groups && n <= q.total_kv_tiles; ++n)
            if (steps(n) < steps(best)) best = n;
        if (10 * steps(best) <= 9 * steps(want)) want = best;
    }
    q.tiles_per_split = (q.total_kv_tiles + want - 1) / want;
    q.n_splits = (q.total_kv_tiles + q.tiles_per_split - 1) / q.tiles_per_split;
    return q;
}

static size_t query_partial_floats(const pevlm_shape_t* s, const QueryPlan& q) {
    return static_cast<size_t>(q.n_splits) * s->query_len * s->num_q_heads * (s->head_dim + 1);
}

// Bytes of the question attention's workspace: the status header and the partials of every sequence.
static size_t query_bytes(const pevlm_shape_t* s, const QueryPlan& q) {
    return kStatusBytes + static_cast<size_t>(s->batch) * ((query_partial_floats(s, q) * sizeof(float) + 255) / 256 * 256);
}
size_t query_workspace_bytes(const pevlm_shape_t* s) { return query_bytes(s, plan_query(s)); }

// Host-side argument checks of the question attention, shared by its two entry points.
int check_query_args(const pevlm_shape_t* s, const void* q_question, const void* k_cache, const void* v_cache,
                     const void* o, const float* lse) {
    const int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if (!q_question || !k_cache || !v_cache || !o) return PEVLM_EINVAL;
    if (!aligned16(q_question) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned32(o) || !aligned16(lse))
        return PEVLM_EALIGN;
    return PEVLM_OK;
}

}  // namespace pevlm

using namespace pevlm;

extern "C" {

const char* pevlm_strerror(int code) {
    switch (code) {
        case PEVLM_OK: return "ok";
        case PEVLM_EINVAL: return "invalid shape or NULL pointer";
        case PEVLM_EALIGN: return "pointer not 16-byte aligned (attention outputs: 32-byte, workspace: 256-byte)";
        case PEVLM_EUNSUPPORTED: return "unsupported head_dim / group size, or device is not sm_100";
        case PEVLM_EWORKSPACE: return "workspace missing or too small";
        case PEVLM_ECUDA: return "CUDA error (see pevlm_last_cuda_error)";
        case PEVLM_ETIMEOUT: return "a bounded device-side wait expired";
        default: return "unknown pevlm status";
    }
}

const char* pevlm_last_cuda_error(void) { return g_cuda_error; }

size_t pevlm_workspace_bytes(const pevlm_shape_t* s, int which) {
    if (check_shape(s) != PEVLM_OK) return 0;
    if (which == PEVLM_WS_PREFILL) return kStatusBytes;
    if (which == PEVLM_WS_QUERY) {
        // The most partial rows that plan_query can ask for: pevlm_layer_forward (of one sequence) with a last block of any length,
        // pevlm_query_attn with this question and cache or shorter ones (a window that is still filling; neither the
        // splits nor splits times rows grow steadily with the lengths).
        const QueryPlan q = plan_query(s);
        const int G = s->num_q_heads / s->num_kv_heads, Q = s->query_len, T = q.total_kv_tiles;
        auto at_most = [](int64_t a, int64_t b) { return a < b ? a : b; };
        auto at_least = [](int64_t a, int64_t b) { return a > b ? a : b; };
        int64_t rows = 0;
        for (int pairs = 1; pairs == 1 || pairs <= (q.q_tiles + 1) / 2; ++pairs) {
            const int groups = s->num_kv_heads * pairs;
            int64_t splits = at_least((kNumSms / 2 + groups - 1) / groups, kNumSms / groups);
            if (s->batch == 1) splits = at_least(splits, at_most((T + 63) / 64, most_splits(groups)));
            rows = at_least(rows, at_most(splits, T) * at_most(Q, 2ll * q.tok_per_tile * pairs));
        }
        const int64_t pieces = (n_video(s) + Q + 15) / 16;
        const int64_t decode_splits = at_least(1, at_most(kNumSms / (static_cast<int64_t>(s->num_kv_heads) * s->batch), (pieces + 7) / 8));
        rows = at_least(rows, decode_splits * at_most(Q, kDecodeRows / G));
        const size_t seq = static_cast<size_t>(rows) * s->num_q_heads * (s->head_dim + 1) * sizeof(float);
        return kStatusBytes + static_cast<size_t>(s->batch) * ((seq + 255) / 256 * 256);
    }
    return 0;
}

// theta^(-2i/d) in fp64; the last ones asked for by this thread are kept (64 calls of pow cost as much as a launch).
static const double* inverse_frequencies(float theta, int d) {
    static thread_local float of_theta = 0.f;
    static thread_local int of_d = 0;
    static thread_local double f[64];
    if (theta != of_theta || d != of_d) {
        for (int i = 0; i < 64; ++i) f[i] = i < d / 2 ? pow(static_cast<double>(theta), -2.0 * i / d) : 0.0;
        of_theta = theta;
        of_d = d;
    }
    return f;
}

// Sequences of one launch: the most (at least one) whose rows can be counted in 30 bits.
static int launch_batch(int batch, int64_t rows) {
    const int64_t most = rows > 0 ? (1ll << 30) / rows : batch;
    const int64_t n = most < 1 ? 1 : most < 32768 ? most : 32768;
    return static_cast<int>(n < batch ? n : batch);
}

// RoPE of q and k (NULL pairs skipped) and a copy of v's rows (NULL = none).  q rows of tokens from `split` on go to
// q_out2 (counted from its first row).
static int rope_common(const pevlm_shape_t* s, const void* q_in, const void* k_in, const void* v_in, void* q_out, void* q_out2,
                       int64_t split, void* k_out, void* v_out, int64_t first_token, int64_t n_tokens, const int32_t* pos_ids,
                       const int32_t* pos3, const int32_t* sections, void* stream) {
    int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if (n_tokens < 0 || first_token < 0 || first_token + n_tokens > (1ll << 31)) return PEVLM_EINVAL;
    if ((q_in == nullptr) != (q_out == nullptr) || (k_in == nullptr) != (k_out == nullptr) || (v_in == nullptr) != (v_out == nullptr))
        return PEVLM_EINVAL;
    if (!q_in && !k_in) return PEVLM_EINVAL;
    if (!aligned16(q_in) || !aligned16(k_in) || !aligned16(v_in) || !aligned16(q_out) || !aligned16(q_out2) || !aligned16(k_out) ||
        !aligned16(v_out))
        return PEVLM_EALIGN;
    if (pos_ids && (reinterpret_cast<uintptr_t>(pos_ids) & 3u)) return PEVLM_EALIGN;
    if (pos3 && (reinterpret_cast<uintptr_t>(pos3) & 3u)) return PEVLM_EALIGN;
    const int d = s->head_dim;
    if (sections) {
        if (sections[0] < 0 || sections[1] < 0 || sections[2] < 0 || sections[0] + sections[1] + sections[2] != d / 2)
            return PEVLM_EINVAL;
    }
    if (n_tokens == 0) return PEVLM_OK;
    RopeParams p;
    memcpy(p.inv_freq, inverse_frequencies(s->rope_theta, d), sizeof(p.inv_freq));
    p.first_token = first_token;
    p.seq_len = static_cast<int32_t>(n_tokens < INT32_MAX ? n_tokens : INT32_MAX);
    p.Hq = q_in ? s->num_q_heads : 0;
    p.Hkv = k_in ? s->num_kv_heads : 0;
    p.Hv = v_in ? s->num_kv_heads : 0;
    p.sec_end0 = sections ? sections[0] : 0;
    p.sec_end1 = sections ? sections[0] + sections[1] : 0;
    const int step = launch_batch(s->batch, n_tokens);
    for (int b = 0; b < s->batch; b += step) {
        const int64_t t0 = static_cast<int64_t>(b) * n_tokens;
        const int64_t qo = t0 * s->num_q_heads * d, ko = t0 * s->num_kv_heads * d;
        auto at = [](const void* base, int64_t off) { return base ? static_cast<const __nv_bfloat16*>(base) + off : nullptr; };
        p.n_tokens = n_tokens * (s->batch - b < step ? s->batch - b : step);
        p.q_in = at(q_in, qo);
        p.q_out = const_cast<__nv_bfloat16*>(at(q_out, qo));
        p.split_token = q_out2 ? split : p.n_tokens;
        // the kernel counts rows from the first token
        p.q_out2 = q_out2 ? static_cast<__nv_bfloat16*>(q_out2) - split * s->num_q_heads * d : nullptr;
        p.k_in = at(k_in, ko);
        p.k_out = const_cast<__nv_bfloat16*>(at(k_out, ko));
        p.v_in = at(v_in, ko);
        p.v_out = const_cast<__nv_bfloat16*>(at(v_out, ko));
        p.pos_ids = pos_ids ? pos_ids + t0 : nullptr;
        p.pos3 = pos3 ? pos3 + 3 * t0 : nullptr;
        cudaError_t e = launch_rope(p, d, static_cast<cudaStream_t>(stream));
        if (e != cudaSuccess) return cuda_fail(e, "rope launch");
    }
    return PEVLM_OK;
}

int pevlm_rope_qk(const pevlm_shape_t* s, const void* q_in, const void* k_in, void* q_out, void* k_out,
                  int64_t first_token, int64_t n_tokens, const int32_t* pos_ids, void* stream) {
    return rope_common(s, q_in, k_in, nullptr, q_out, nullptr, 0, k_out, nullptr, first_token, n_tokens, pos_ids, nullptr, nullptr, stream);
}

int pevlm_rope_qk_mrope(const pevlm_shape_t* s, const void* q_in, const void* k_in, void* q_out, void* k_out,
                        int64_t n_tokens, const int32_t* pos_ids3, const int32_t* sections, void* stream) {
    if (!pos_ids3 || !sections) return PEVLM_EINVAL;
    return rope_common(s, q_in, k_in, nullptr, q_out, nullptr, 0, k_out, nullptr, 0, n_tokens, nullptr, pos_ids3, sections, stream);
}

int pevlm_rope_qkv(const pevlm_shape_t* s, const void* q_in, const void* k_in, const void* v_in, void* q_out, void* k_out, void* v_out,
                   int64_t first_token, int64_t n_tokens, const int32_t* pos_ids, void* stream) {
    return rope_common(s, q_in, k_in, v_in, q_out, nullptr, 0, k_out, v_out, first_token, n_tokens, pos_ids, nullptr, nullptr, stream);
}

int pevlm_assemble_kv(const pevlm_shape_t* s, const void* k_video, const void* v_video, const void* k_question,
                      const void* v_question, void* k_cache, void* v_cache, void* stream) {
    int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if ((k_video || k_question) && !k_cache) return PEVLM_EINVAL;
    if ((v_video || v_question) && !v_cache) return PEVLM_EINVAL;
    if (!aligned16(k_video) || !aligned16(v_video) || !aligned16(k_question) || !aligned16(v_question) ||
        !aligned16(k_cache) || !aligned16(v_cache))
        return PEVLM_EALIGN;
    const int64_t nv = n_video(s);
    const int64_t row_vec = static_cast<int64_t>(s->num_kv_heads) * s->head_dim * 2 / 16;  // 16-byte vectors per token
    const int64_t L = nv + s->query_len;
    CopySegments seg;
    const void* srcs[4] = {k_video, k_question, v_video, v_question};
    void* dsts[4] = {k_cache, k_cache, v_cache, v_cache};
    const int64_t rows[4] = {nv, s->query_len, nv, s->query_len};
    const int64_t dst_row0[4] = {0, nv, 0, nv};
    seg.dst_stride = L * row_vec;
    for (int b = 0; b < s->batch; b += 32768) {
        seg.batch = s->batch - b < 32768 ? s->batch - b : 32768;
        seg.total = 0;
        for (int i = 0; i < 4; ++i) {
            const int64_t n = srcs[i] ? rows[i] * row_vec : 0;
            seg.n_vec[i] = n;
            seg.src_stride[i] = n;
            seg.src[i] = srcs[i] ? static_cast<const uint4*>(srcs[i]) + b * n : nullptr;
            seg.dst[i] = dsts[i] ? static_cast<uint4*>(dsts[i]) + (static_cast<int64_t>(b) * L + dst_row0[i]) * row_vec : nullptr;
            seg.total += n;
        }
        cudaError_t e = launch_copy_segments(seg, static_cast<cudaStream_t>(stream));
        if (e != cudaSuccess) return cuda_fail(e, "assemble launch");
    }
    return PEVLM_OK;
}

// ---- parameters of an attention launch
static AttnParams common_params(const pevlm_shape_t* s, int last_len = 0) {
    AttnParams p;
    memset(&p, 0, sizeof(p));
    p.n_video = static_cast<int>(n_video(s, last_len));
    p.Q = s->query_len;
    p.L = p.n_video + s->query_len;
    p.Hq = s->num_q_heads; p.Hkv = s->num_kv_heads; p.G = p.Hq / p.Hkv;
    p.scale = resolve_scale(s);
    p.scale_log2 = p.scale * 1.4426950408889634f;
    p.wait_tries = kDefaultWaitTries;
    return p;
}

// Prefill rows.  blocks_only = false: the whole video stream [sink | N blocks] (or full causal).  blocks_only = true: N
// blocks whose K/V sit at rows [first_key_row, first_key_row + N*B) of a cache of cache_rows rows whose first S rows are
// the sink; q / o / lse cover the N*B block rows only and the sink rows are not computed.
static void add_prefill(AttnParams& p, const pevlm_shape_t* s, bool blocks_only, int64_t first_key_row, int64_t cache_rows, int last_len = 0) {
    const int64_t nv = p.n_video;
    p.mode |= 1;
    int S = s->sink_len, B = s->num_blocks > 0 ? s->block_len : 0, N = s->num_blocks - (last_len > 0 ? 1 : 0);
    if (s->mask_mode == PEVLM_MASK_FULL_CAUSAL) {
        S = 0; B = static_cast<int>(nv); N = 1;
        last_len = 0;
    }
    p.sink_len = S;
    p.block_rows = N * B + last_len;
    p.blk_key0 = blocks_only ? static_cast<int>(first_key_row) : S;
    const int blk_q0 = blocks_only ? 0 : S;
    p.q_rows = static_cast<int>(blocks_only ? static_cast<int64_t>(s->num_blocks) * s->block_len : nv);
    p.kv_rows = static_cast<int>(blocks_only ? cache_rows : nv);
    p.div_hkv = make_divisor(p.Hkv);
    p.div_g = make_divisor(p.G);
    auto fill = [&](Segment& g, int n, int len, int q0, int key0, int a_end, int own_map, bool blocks) {
        const SegPlan sp = plan_segment(n > 0 ? len : 0, p.G);
        g.len = len; g.q0 = q0; g.key0 = key0; g.a_end = a_end; g.own_map = own_map;
        g.full_tiles = sp.full_tiles; g.entries = sp.entries;
        g.tail_tiles = sp.tail_tiles;
        g.form[0] = {1, kTile, 1, 0, kTile};
        g.form[1] = sp.tail;
        // How many pairs of one (block, kv head) are handed out together (decode_item): the whole list keeps the CTAs
        // that run at the same time on few K/V tiles (best for long blocks); short blocks (at most 4 query tiles)
        // run faster when pairs of equal length are handed out together across all blocks, and a segment with few
        // items per SM balances best with single pairs, heaviest first, the sink and a shorter last block too where they are not
        // short (28/4 heads, whole list of the sink against single pairs, medians in one process: 7 times 784 tokens 111.5 / 108.6 us, a sink of
        // 1,980 before 272 49.3 / 46.2, of 999 before 80 24.0 / 21.8; of 42 shapes, batches among them, none slower beyond noise).  Thresholds
        // from measurements on B200.
        int want_pc = sp.pairs;
        if (blocks && sp.tiles <= 4) want_pc = p.G / 2 > 0 ? p.G / 2 : 1;
        else if (sp.tiles > 4 && static_cast<int64_t>(n) * p.Hkv * sp.pairs < 16 * kNumSms) want_pc = 1;
        g.pair_chunk = sp.pairs > 0 ? (want_pc < sp.pairs ? want_pc : sp.pairs) : 1;
        const int n_chunks = sp.pairs > 0 ? (sp.pairs + g.pair_chunk - 1) / g.pair_chunk : 0;
        g.per_chunk = n * p.Hkv * g.pair_chunk;
        g.items = g.per_chunk * n_chunks;
        g.div_per_chunk = make_divisor(g.per_chunk);
        g.div_pair_chunk = make_divisor(g.pair_chunk);
        p.n_items += g.items;
    };
    fill(p.seg[0], N, B, blk_q0, 0, S, 0, true);
    fill(p.seg[1], last_len > 0, last_len, blk_q0 + N * B, N * B, S, 0, false);
    fill(p.seg[2], S > 0 && !blocks_only, S, 0, 0, 0, 1, false);
}

static void add_question(AttnParams& p, const QueryPlan& qp) {
    p.mode |= 2;
    p.tok_per_tile = qp.tok_per_tile;
    p.q_tiles = qp.q_tiles;
    p.n_splits = qp.n_splits;
    p.tiles_per_split = qp.tiles_per_split;
    p.items_question = p.Hkv * ((p.q_tiles + 1) / 2) * p.n_splits;
    p.n_items += p.items_question;
    p.div_splits = make_divisor(p.n_splits);
    p.div_q_pairs = make_divisor((p.q_tiles + 1) / 2);
}

// K and V of one range of each of p.batch sequences: `rows` rows from the base on, the sequences seq_rows apart.  (A map needs at
// least one row; an empty range is never read.)
static int kv_maps(AttnMaps& m, int i, const AttnParams& p, int d, const __nv_bfloat16* k, const __nv_bfloat16* v, int64_t rows, int64_t seq_rows) {
    const int64_t n = rows > 0 ? rows : 1;
    const int rc = make_tmap(&m.k[i], k, n, p.Hkv, d, 1, kTile / 2, 64, p.batch, seq_rows);
    return rc != PEVLM_OK ? rc : make_tmap(&m.v[i], v, n, p.Hkv, d, 1, kTile, d / 2, p.batch, seq_rows);
}

static int prefill_maps(AttnMaps& m, const AttnParams& p, int d, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v) {
    int rc;
    const int64_t q_rows = static_cast<int64_t>(p.batch) * p.q_rows;
    if ((rc = make_tmap(&m.q[0], q, q_rows, p.Hq, d, 1, kTile)) != PEVLM_OK) return rc;
    for (int i = 0; i < 3; ++i) {
        const Segment& g = p.seg[i];
        if (g.items > 0 && g.tail_tiles > 0 && (rc = make_tmap(&m.q[1 + i], q, q_rows, p.Hq, d, g.form[1].heads, g.form[1].toks)) != PEVLM_OK) return rc;
    }
    const int64_t blk_off = static_cast<int64_t>(p.blk_key0) * p.Hkv * d;
    if ((rc = kv_maps(m, 0, p, d, k + blk_off, v + blk_off, p.block_rows, p.kv_rows)) != PEVLM_OK) return rc;
    return kv_maps(m, 1, p, d, k, v, p.sink_len, p.kv_rows);
}

static int question_maps(AttnMaps& m, const AttnParams& p, int d, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v) {
    const int rc = make_tmap(&m.q[4], q, static_cast<int64_t>(p.batch) * p.Q, p.Hq, d, p.G, p.tok_per_tile);
    return rc != PEVLM_OK ? rc : kv_maps(m, 2, p, d, k, v, p.L, p.L);
}

static int merge_question(const AttnParams& p, int d, __nv_bfloat16* o, float* lse, cudaStream_t st) {
    MergeParams m;
    m.batch = p.batch; m.Q = p.Q; m.Hq = p.Hq; m.d = d; m.n_splits = p.n_splits;
    m.part_o = p.part_o; m.part_lse = p.part_lse;
    m.o = o;
    m.lse = lse;
    const cudaError_t e = launch_merge(m, st);
    return e == cudaSuccess ? PEVLM_OK : cuda_fail(e, "merge launch");
}

static const __nv_bfloat16* rows_of(const void* base, int64_t rows, int heads, int d) {
    return static_cast<const __nv_bfloat16*>(base) + rows * heads * d;
}

static int prefill_common(const pevlm_shape_t* s, const void* q, const void* k, const void* v, void* o, float* lse,
                          void* workspace, size_t workspace_bytes, void* stream, bool blocks_only,
                          int64_t first_key_row, int64_t cache_rows) {
    int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if (!q || !k || !v || !o) return PEVLM_EINVAL;
    // the output rows are written with 32-byte vector stores
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned32(o) || !aligned16(lse)) return PEVLM_EALIGN;
    if (!workspace || workspace_bytes < pevlm_workspace_bytes(s, PEVLM_WS_PREFILL)) return PEVLM_EWORKSPACE;
    if (!aligned256(workspace)) return PEVLM_EALIGN;
    const int64_t block_rows = static_cast<int64_t>(s->num_blocks) * s->block_len;
    if (blocks_only) {
        if (s->mask_mode != PEVLM_MASK_PEVLM) return PEVLM_EINVAL;
        if (first_key_row < s->sink_len || first_key_row + block_rows > cache_rows || cache_rows > (1ll << 30))
            return PEVLM_EINVAL;
        if (block_rows == 0) return PEVLM_OK;
    } else if (n_video(s) == 0) {
        return PEVLM_OK;
    }
    rc = check_device();
    if (rc != PEVLM_OK) return rc;
    const int d = s->head_dim;
    AttnParams p = common_params(s);
    add_prefill(p, s, blocks_only, first_key_row, cache_rows);
    p.div_items = make_divisor(p.n_items);
    p.hdr = static_cast<WorkspaceHeader*>(workspace);
    const int step = blocks_only ? 1 : launch_batch(s->batch, p.kv_rows > p.n_items ? p.kv_rows : p.n_items);
    for (int b = 0; b < s->batch; b += step) {
        p.batch = s->batch - b < step ? s->batch - b : step;
        p.keep_status = b > 0;
        const int64_t q0 = static_cast<int64_t>(b) * p.q_rows, k0 = static_cast<int64_t>(b) * p.kv_rows;
        AttnMaps m;
        if ((rc = prefill_maps(m, p, d, rows_of(q, q0, p.Hq, d), rows_of(k, k0, p.Hkv, d), rows_of(v, k0, p.Hkv, d))) != PEVLM_OK) return rc;
        p.o = const_cast<__nv_bfloat16*>(rows_of(o, q0, p.Hq, d));
        p.lse = lse ? lse + static_cast<int64_t>(p.Hq) * q0 : nullptr;
        const cudaError_t e = launch_attn(p, d, m, static_cast<cudaStream_t>(stream));
        if (e != cudaSuccess) return cuda_fail(e, "prefill attention launch");
    }
    return PEVLM_OK;
}

int pevlm_parallel_prefill_attn(const pevlm_shape_t* s, const void* q, const void* k, const void* v, void* o, float* lse,
                                void* workspace, size_t workspace_bytes, void* stream) {
    return prefill_common(s, q, k, v, o, lse, workspace, workspace_bytes, stream, false, 0, 0);
}

int pevlm_block_attn(const pevlm_shape_t* s, const void* q_blocks, const void* k_cache, const void* v_cache,
                     int64_t first_key_row, int64_t cache_rows, void* o, float* lse, void* workspace,
                     size_t workspace_bytes, void* stream) {
    return prefill_common(s, q_blocks, k_cache, v_cache, o, lse, workspace, workspace_bytes, stream, true,
                          first_key_row, cache_rows);
}

static int decode(const pevlm_shape_t* s, const QueryPlan& qp, const void* q, const void* k, const void* v, void* o, float* lse,
                  void* workspace, cudaStream_t st) {
    const int d = s->head_dim;
    AttnParams a = common_params(s);
    a.n_splits = qp.n_splits;
    DecodeParams p;
    p.Q = a.Q; p.L = a.L; p.n_video = a.n_video; p.Hq = a.Hq; p.Hkv = a.Hkv; p.G = a.G;
    p.pieces = qp.pieces; p.pieces_per_split = qp.pieces_per_split; p.n_splits = qp.n_splits;
    p.scale = a.scale; p.scale_log2 = a.scale_log2;
    p.hdr = static_cast<WorkspaceHeader*>(workspace);
    for (int b = 0; b < s->batch; b += 32768) {
        a.batch = p.batch = s->batch - b < 32768 ? s->batch - b : 32768;
        a.part_o = p.part_o = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + kStatusBytes);
        a.part_lse = p.part_lse = p.part_o + static_cast<size_t>(p.batch) * p.n_splits * p.Q * p.Hq * d;
        const int64_t q0 = static_cast<int64_t>(b) * p.Q, k0 = static_cast<int64_t>(b) * p.L;
        p.q = rows_of(q, q0, p.Hq, d);
        p.k = rows_of(k, k0, p.Hkv, d);
        p.v = rows_of(v, k0, p.Hkv, d);
        const cudaError_t e = launch_decode(p, d, st);
        if (e != cudaSuccess) return cuda_fail(e, "decode launch");
        const int rc = merge_question(a, d, const_cast<__nv_bfloat16*>(rows_of(o, q0, p.Hq, d)), lse ? lse + p.Hq * q0 : nullptr, st);
        if (rc != PEVLM_OK) return rc;
    }
    return PEVLM_OK;
}

int pevlm_query_attn(const pevlm_shape_t* s, const void* q_question, const void* k_cache, const void* v_cache, void* o,
                     float* lse, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_query_args(s, q_question, k_cache, v_cache, o, lse);
    if (rc != PEVLM_OK) return rc;
    if (!workspace || workspace_bytes < query_workspace_bytes(s)) return PEVLM_EWORKSPACE;
    if (!aligned256(workspace)) return PEVLM_EALIGN;
    if (s->query_len == 0) return PEVLM_OK;
    rc = check_device();
    if (rc != PEVLM_OK) return rc;
    const int d = s->head_dim;
    const QueryPlan qp = plan_query(s);
    if (qp.pieces > 0) return decode(s, qp, q_question, k_cache, v_cache, o, lse, workspace, static_cast<cudaStream_t>(stream));
    AttnParams p = common_params(s);
    add_question(p, qp);
    p.div_items = make_divisor(p.n_items);
    p.hdr = static_cast<WorkspaceHeader*>(workspace);
    const int step = launch_batch(s->batch, p.L > p.n_items ? p.L : p.n_items);
    const size_t seq_floats = static_cast<size_t>(p.n_splits) * p.Q * p.Hq;
    for (int b = 0; b < s->batch; b += step) {
        p.batch = s->batch - b < step ? s->batch - b : step;
        p.keep_status = b > 0;
        p.part_o = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + kStatusBytes);
        p.part_lse = p.part_o + seq_floats * d * p.batch;
        const int64_t q0 = static_cast<int64_t>(b) * p.Q, k0 = static_cast<int64_t>(b) * p.L;
        AttnMaps m;
        if ((rc = question_maps(m, p, d, rows_of(q_question, q0, p.Hq, d), rows_of(k_cache, k0, p.Hkv, d), rows_of(v_cache, k0, p.Hkv, d))) != PEVLM_OK) return rc;
        p.o_question = const_cast<__nv_bfloat16*>(rows_of(o, q0, p.Hq, d));
        p.lse_question = lse ? lse + p.Hq * q0 : nullptr;
        const cudaError_t e = launch_attn(p, d, m, static_cast<cudaStream_t>(stream));
        if (e != cudaSuccess) return cuda_fail(e, "question attention launch");
        if (p.n_splits > 1) rc = merge_question(p, d, p.o_question, p.lse_question, static_cast<cudaStream_t>(stream));
        if (rc != PEVLM_OK) return rc;
    }
    return PEVLM_OK;
}

int pevlm_layer_forward(const pevlm_shape_t* s, int32_t last_len, const void* q, const void* k, const void* v, void* q_video, void* q_question,
                        void* k_cache, void* v_cache, void* o_video, float* lse_video, void* o_question, float* lse_question,
                        void* ws_prefill, size_t ws_prefill_bytes, void* ws_query, size_t ws_query_bytes, void* stream) {
    int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if (s->batch != 1) return PEVLM_EUNSUPPORTED;
    if (last_len < 0 || (last_len > 0 && (s->num_blocks < 1 || last_len > s->block_len))) return PEVLM_EINVAL;
    if (last_len == s->block_len) last_len = 0;
    const int64_t nv = n_video(s, last_len);
    const int Q = s->query_len, d = s->head_dim, Hq = s->num_q_heads;
    if (!q || !k || !v || !k_cache || !v_cache) return PEVLM_EINVAL;
    if (nv > 0 && (!q_video || !o_video)) return PEVLM_EINVAL;
    if (Q > 0 && (!q_question || !o_question)) return PEVLM_EINVAL;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(q_video) || !aligned16(q_question) || !aligned16(k_cache) ||
        !aligned16(v_cache) || !aligned32(o_video) || !aligned16(lse_video) || !aligned32(o_question) || !aligned16(lse_question))
        return PEVLM_EALIGN;
    const QueryPlan qp = plan_query(s, true, last_len);
    if (nv > 0 && (!ws_prefill || ws_prefill_bytes < pevlm_workspace_bytes(s, PEVLM_WS_PREFILL))) return PEVLM_EWORKSPACE;
    if (Q > 0 && (!ws_query || ws_query_bytes < query_bytes(s, qp))) return PEVLM_EWORKSPACE;
    if (!aligned256(ws_prefill) || !aligned256(ws_query)) return PEVLM_EALIGN;
    rc = check_device();
    if (rc != PEVLM_OK) return rc;
    // every token's Q and K roped, K and V into the cache
    rc = nv > 0 ? rope_common(s, q, k, v, q_video, Q > 0 ? q_question : nullptr, nv, k_cache, v_cache, 0, nv + Q, nullptr, nullptr, nullptr, stream)
                : rope_common(s, q, k, v, q_question, nullptr, 0, k_cache, v_cache, 0, Q, nullptr, nullptr, nullptr, stream);
    if (rc != PEVLM_OK) return rc;
    AttnParams p = common_params(s, last_len);
    AttnMaps m;
    p.batch = 1;
    if (nv > 0) {
        add_prefill(p, s, false, 0, 0, last_len);
        rc = prefill_maps(m, p, d, static_cast<const __nv_bfloat16*>(q_video), static_cast<const __nv_bfloat16*>(k_cache), static_cast<const __nv_bfloat16*>(v_cache));
        if (rc != PEVLM_OK) return rc;
        p.o = static_cast<__nv_bfloat16*>(o_video);
        p.lse = lse_video;
        p.hdr = static_cast<WorkspaceHeader*>(ws_prefill);
    }
    if (Q > 0) {
        add_question(p, qp);
        rc = question_maps(m, p, d, static_cast<const __nv_bfloat16*>(q_question), static_cast<const __nv_bfloat16*>(k_cache), static_cast<const __nv_bfloat16*>(v_cache));
        if (rc != PEVLM_OK) return rc;
        p.o_question = static_cast<__nv_bfloat16*>(o_question);
        p.lse_question = lse_question;
        p.hdr_question = static_cast<WorkspaceHeader*>(ws_query);
        if (nv == 0) p.hdr = p.hdr_question;
        p.part_o = reinterpret_cast<float*>(static_cast<uint8_t*>(ws_query) + kStatusBytes);
        p.part_lse = p.part_o + static_cast<size_t>(p.n_splits) * Q * Hq * d;
    }
    const cudaError_t e = launch_attn(p, d, m, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "attention launch");
    return Q > 0 && p.n_splits > 1 ? merge_question(p, d, p.o_question, p.lse_question, static_cast<cudaStream_t>(stream)) : PEVLM_OK;
}

int pevlm_selftest_wait_expiry(void* workspace, size_t workspace_bytes, int64_t limit_ns, void* stream) {
    if (!workspace || workspace_bytes < kStatusBytes) return PEVLM_EWORKSPACE;
    if (!aligned256(workspace)) return PEVLM_EALIGN;
    if (limit_ns < 1000 || limit_ns > 100ll * 1000 * 1000) return PEVLM_EINVAL;  // 1 us .. 100 ms
    int rc = check_device();
    if (rc != PEVLM_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(workspace, 0, kStatusBytes, st);
    if (e != cudaSuccess) return cuda_fail(e, "workspace memset");
    e = launch_wait_selftest(static_cast<WorkspaceHeader*>(workspace), static_cast<uint32_t>(limit_ns), st);
    if (e != cudaSuccess) return cuda_fail(e, "wait self-test launch");
    return PEVLM_OK;
}

int pevlm_read_status(const void* workspace, void* stream, int32_t* status, int32_t* detail) {
    if (!status) return PEVLM_EINVAL;
    if (!workspace) {  // the built-in array of pevlm_query_attn_noalloc on the current device
        void* scratch = nullptr;
        const int rc = noalloc_scratch_for_current_device(&scratch);
        if (rc != PEVLM_OK) return rc;
        workspace = scratch;
    }
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    int32_t words[2] = {0, 0};
    e = cudaMemcpy(words, workspace, sizeof(words), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(status)");
    *status = words[0];
    if (detail) *detail = words[1];
    return PEVLM_OK;
}

int pevlm_tile_stats(const pevlm_shape_t* s, int which, int64_t* tiles, double* flops) {
    int rc = check_shape(s);
    if (rc != PEVLM_OK) return rc;
    if (!tiles || !flops) return PEVLM_EINVAL;
    const int d = s->head_dim;
    int64_t n_tiles = 0;
    double cols = 0.0;  // sum over visited tiles of issued key columns (each over 128 query rows)
    auto add_range = [&](int64_t len) {  // a key range visited from its start in 128-key tiles
        for (int64_t j = 0; j < len; j += kTile) {
            const int64_t valid = len - j < kTile ? len - j : kTile;
            n_tiles += 1;
            cols += static_cast<double>((valid + 15) / 16 * 16);
        }
    };
    const int64_t nv = n_video(s);
    if (which == PEVLM_WS_PREFILL) {
        int64_t S = s->sink_len, B = s->num_blocks > 0 ? s->block_len : 0, N = s->num_blocks;
        if (s->mask_mode == PEVLM_MASK_FULL_CAUSAL) { S = 0; B = nv; N = nv > 0 ? 1 : 0; }
        const int G = s->num_q_heads / s->num_kv_heads;
        // query tiles of one segment per kv head: G per full tile position, tail_tiles for a packed ragged tail
        auto add_segment = [&](int64_t len, int64_t shared) {
            const SegPlan sp = plan_segment(static_cast<int>(len), G);
            for (int qt = 0; qt < sp.tiles; ++qt) {
                const int64_t q0 = static_cast<int64_t>(qt) * kTile;
                const bool tail = sp.tail_tiles > 0 && qt == sp.tiles - 1;
                const bool by_toks = tail && sp.tail.tok_step > 0;  // then the tiles of the tail see ever more keys
                for (int e = 0; e < (by_toks ? sp.tail_tiles : 1); ++e) {
                    const int64_t t0 = n_tiles; const double c0 = cols;
                    const int64_t end = by_toks ? q0 + (e + 1) * sp.tail.tok_step : q0 + kTile;
                    add_range(shared);
                    add_range(end < len ? end : len);
                    const int q_tiles = by_toks ? 1 : tail ? sp.tail_tiles : G;
                    n_tiles = t0 + (n_tiles - t0) * q_tiles;
                    cols = c0 + (cols - c0) * q_tiles;
                }
            }
        };
        add_segment(S, 0);
        const int64_t t0 = n_tiles; const double c0 = cols;
        add_segment(B, S);
        n_tiles = t0 + (n_tiles - t0) * N;   // the block part repeats for each of the N blocks
        cols = c0 + (cols - c0) * static_cast<double>(N);
        n_tiles *= s->num_kv_heads;
        cols *= s->num_kv_heads;
    } else if (which == PEVLM_WS_QUERY) {
        const QueryPlan qp = plan_query(s);
        if (qp.pieces > 0) {  // decode kernel: 16 or 32 rows against 16 keys at a time, counted in key tiles of 128
            n_tiles = (qp.pieces + 7) / 8 * static_cast<int64_t>(s->num_kv_heads);
            *tiles = n_tiles * s->batch;
            const int rows = s->query_len * (s->num_q_heads / s->num_kv_heads);
            *flops = 4.0 * d * (rows > 16 ? 32 : 16) * 16.0 * qp.pieces * s->num_kv_heads * s->batch;
            return PEVLM_OK;
        }
        for (int qt = 0; qt < qp.q_tiles; ++qt) {
            const int tok0 = qt * qp.tok_per_tile;
            const int ntok = s->query_len - tok0 < qp.tok_per_tile ? s->query_len - tok0 : qp.tok_per_tile;
            const int64_t kv_end = nv + tok0 + ntok;
            for (int sp = 0; sp < qp.n_splits; ++sp) {
                int64_t a = static_cast<int64_t>(sp) * qp.tiles_per_split * kTile, e = a + static_cast<int64_t>(qp.tiles_per_split) * kTile;
                if (a > kv_end) a = kv_end;
                if (e > kv_end) e = kv_end;
                add_range(e - a);
            }
        }
        n_tiles *= s->num_kv_heads;
        cols *= s->num_kv_heads;
    } else {
        return PEVLM_EINVAL;
    }
    *tiles = n_tiles * s->batch;
    *flops = 4.0 * d * kTile * cols * s->batch;
    return PEVLM_OK;
}

}  // extern "C"
