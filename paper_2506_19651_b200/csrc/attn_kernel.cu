// Warp-specialised block-masked flash attention for sm_100a (Eq. 1 under the masks of Eq. 3-5), on CTA pairs.
//
// A pair of CTAs (a cluster of 2, cta_group::2) owns a work item = TWO query tiles of 128 rows that share a kv head and
// a key-tile list (two q heads of one GQA group at the same block position, or two neighbouring positions); CTA r of the
// pair owns tile r.  The MMAs span the pair (M = 256): each CTA stages half of every K tile (64 keys) and half of every
// V tile (D/2 columns), so a pair reads each K/V tile from L2 once and an SM's shared memory holds and delivers half.
// Per CTA, 16 warps:
//   warps 0-3, 4-7  two softmax warpgroups, one thread per row, taking the key tiles of the CTA's query tile in turn.
//               The 128 scores of a key tile are read from TMEM once, the probabilities written back as bf16.  The
//               running reference maximum of a row passes from one warpgroup to the other through shared memory
//               (warp to warp); it moves only when the row's maximum grows by more than 2^8, and then the thread
//               rescales its row of the output accumulator in place (rare).  Each warpgroup keeps the row sum of its
//               own tiles; the epilogue adds the two
//   warps 8-11  epilogue: reads the finished accumulator, releases it, writes the normalised output and the LSE
//   warps 12, 14 (first CTA of the pair) issue the tcgen05 MMAs of both CTAs: warp 12 S = Q K^T (operands from shared
//               memory), warp 14 O += P V (P from TMEM, V from shared memory).  Neither has to know of the other
//   warp 13     TMA producer of Q, K and V
//   warp 15     scheduler: takes work items from the hardware's queue of unlaunched clusters, decodes each once into
//               shared memory for the other roles (the decode is a dozen integer divisions)
// TMEM (512 columns): score buffers S0 S1 of 128 columns, probability buffers P0 P1 of 64, accumulator O of D.
// Probabilities and scores do not share columns, so QK(t + 2) needs nothing but that tile t's scores have been read
// into registers, which is the first thing its softmax does: the scores of a softmax warpgroup's next tile are ready
// long before it has finished this one, and neither the tensor pipe's latency nor the hand-offs between the warps are
// on its path.  QK runs three tiles ahead of PV, over the boundaries of work items too.
// What bounds it: back to back, the 1 kW cap (all sizes from 12K tokens on run at 1.4 to 1.6 GHz): what a tile costs in
// energy, for which idle cycles count too.  At a given clock, the softmax: two warpgroups that never wait take 2,390
// cycles for two key tiles beside running MMAs, the MMAs 1,024 a tile (both measured free-running).  Reached are 1,460
// cycles a tile on long work items (1,741 before, with two query tiles and two softmax warpgroups per CTA) and 1,830 with
// four tiles an item (2,710 before).  Back to back: 50K tokens 1.708 -> 1.49 ms, 12.6K 0.249 -> 0.213, 256-token blocks
// 0.322 -> 0.257, 8,192-token blocks 4.97 -> 4.5.  Two things took more than the schedule itself:
//   - the two softmax warps that share a scheduler take turns on its special-function unit (left alone they fall into
//     step, form their exponentials at the same time and leave the unit idle at the same time: 1,741 cycles a tile);
//   - instruction fetch.  What a work item runs (all roles, masks and item ends included) has to stay near the size of
//     the SM's instruction cache: at 73 KB of code four-tile items lost more time to missing instructions than to
//     anything else (26 % of the fetches missed, 0.348 ms), at 55 KB they took 0.296 ms, at 50 KB 0.257.  Hence one
//     instantiation per mode, loops that stay loops wherever the registers' indices allow it, waits that expand to
//     little, no divisions, and warp-uniform values that the compiler knows to be uniform (the MMA warps' descriptors
//     then live in uniform registers instead of being moved there for every MMA: 10 KB of code).
// Every wait on an mbarrier is bounded; an expired wait records PEVLM_ETIMEOUT and the CTA still runs to its
// normal end (waits become short) and stays until what is in flight has landed, so TMEM is always released and nothing
// writes to shared memory that has a new owner.
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

constexpr int kAttnThreads = 512;
constexpr int kRing = 4;      // K tiles and V tiles in flight
constexpr int kQkAhead = 3;   // tiles by which QK runs ahead of PV
constexpr int kItems = 8;     // decoded work items in flight
constexpr int kSums = 8;      // items whose row sums may be in flight between softmax and epilogue
constexpr int kDrainUs = 64;
constexpr unsigned kNoMore = 1u << 31;
constexpr int kClaimAhead = 6;  // tiles before the end of an item's loads at which the next item is claimed
// pair of exponentials (of 64) after which a softmax warp passes the turn on: the rest overlaps the other warp's start
// (measured: 16 to 40 within 1 % of each other, 52 and later 4 % slower)
constexpr int kTurn = 40;
constexpr float kRescaleThresholdLog2 = 8.0f;  // rescale O only when the row maximum grew by > 2^8
constexpr uint32_t kTmemP = 2 * kTile;          // first TMEM column of the probability buffers
constexpr uint32_t kTmemO = kTmemP + kTile;     // of the accumulator

enum WaitId : int {
    kWaitQ = 11, kWaitK = 12, kWaitV = 13, kWaitS = 14, kWaitP = 15, kWaitSRead = 16, kWaitPV = 17, kWaitPFree = 18, kWaitItem = 19,
    kWaitItemFree = 20, kWaitQFree = 21, kWaitOFree = 22, kWaitKvFree = 23, kWaitSum = 25, kWaitODone = 26,
    kWaitGo = 27, kWaitClc = 28
};

template <int D>
struct AttnSmem {
    static constexpr int kPanels = D / 64;
    static constexpr int kQPanelBytes = kTile * 128;     // 128 rows of 64 elements
    static constexpr int kKPanelBytes = kTile / 2 * 128; // this CTA's 64 keys of 64 elements
    static constexpr int kQBytes = kPanels * kQPanelBytes;
    static constexpr int kKBytes = kPanels * kKPanelBytes;
    static constexpr int kVBytes = kTile * D;            // 128 keys of this CTA's D/2 columns
    static constexpr int kQ = 0;                         // two buffers
    static constexpr int kK = 2 * kQBytes;
    static constexpr int kV = kK + kRing * kKBytes;
    static constexpr int kTotal = kV + kRing * kVBytes;
};

static size_t attn_smem_bytes(int head_dim) {
    return 1024 + (head_dim == 128 ? AttnSmem<128>::kTotal : AttnSmem<64>::kTotal);
}

// One query tile.  Row r of the tile is token q_tok0 + r / row_div, head q_head0 + r % row_div; it
// exists iff r / row_div < ntok and r % row_div < nheads.  Full prefill tiles have row_div = 1; the
// ragged last tile of a segment packs the tails of several q heads of the kv group (row_div heads,
// ntok = the tail's rows, or some of them and all heads); question tiles pack all G heads of the group.
struct QSlot {
    int valid;
    int q_tok0, q_head0, row_div, ntok, nheads, qmap, box_rows;
    int per_div;  // ceil(2^16 / row_div): r / row_div = r * per_div >> 16 for r < 128
    int limit0;  // last visible key of row token 0, counted from the first key of the own range
    int end;     // keys of the own range that the tile's rows can see at all
};
// Key tiles of an item: first the na tiles of the shared range [0, a_end) (the sink), then the tiles of the own
// range, nt tiles in all (what the longer of the two query tiles needs; the other one masks its surplus tile).
// The own range is fetched at row b_coord0 of the block tensor map (own_map = 0), for the sink's own items of the sink map
// (1), for question items of the map of the whole cache (2).  seq: sequence of the batch, a dimension of those maps of its own.
// n_a, n_b: MMA columns of tile na - 1 and of the last tile; the others have 128.
struct WorkItem {
    int kv_head, a_end, na, nt, n_a, n_b, split, b_coord0, own_map, seq;
    QSlot s[2];
};

// Optional accounting (-DPEVLM_TRACE): for the first CTA pair of a launch, the cycles every warp spent in each kind of
// wait and between the start and the end of its role, read back through pevlm_debug_waits (see timeline.py).
#ifdef PEVLM_TRACE
constexpr int kTraceIds = 32;  // wait ids are below this; index 0 = whole role, 1 = key tiles handled
__device__ unsigned g_waits[2][16][kTraceIds];
extern "C" int pevlm_debug_waits(unsigned* host_out) {
    return cudaMemcpyFromSymbol(host_out, g_waits, sizeof(g_waits)) == cudaSuccess ? 0 : -1;
}
#endif

// A value that is the same in all lanes of a warp, told to the compiler, so that what depends on it stays in uniform registers.
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }
__device__ __forceinline__ int cdiv(int a, int b) { return (a + b - 1) / b; }

// MODE: bit 0 = the launch has prefill items, bit 1 = it has question items (handed out first: they are the longest).
// Items of a sequence follow one another, w counts over the whole batch.
template <int MODE>
__device__ __forceinline__ void decode_item(const AttnParams& p, int w, WorkItem& it) {
    it.split = 0;
    it.seq = 0;
    if (p.batch > 1) {
        it.seq = quotient(w, p.div_items);
        w -= it.seq * p.n_items;
    }
    const bool question = MODE == 2 || (MODE == 3 && w < p.items_question);
    if (MODE == 3) w -= question ? 0 : p.items_question;
    int own_keys = 0;  // keys of the own range that the longer query tile sees
    if (!question) {
        // Which kind of segment: the full blocks, a shorter last block, the sink.
        int kind = 0;
#pragma unroll 1
        while (kind < 2 && w >= p.seg[kind].items) w -= p.seg[kind++].items;
        const Segment& sg = p.seg[kind];
        // Order of the items: the pair list of a (block, kv head), heaviest first, is cut into chunks of
        // pair_chunk pairs; chunk-major, then (block, kv head), then the pairs of the chunk.  CTAs that run
        // at the same time then share few K/V tiles' worth of L2 traffic, and the launch ends on the
        // lightest chunk of every (block, kv head) rather than on the last block's whole list.  A pair
        // index past the end of the list (padding of the last chunk) is an empty item.
        const int chunk = quotient(w, sg.div_per_chunk), r = w - chunk * sg.per_chunk;
        const int combo = quotient(r, sg.div_pair_chunk);
        const int pi = chunk * sg.pair_chunk + r - combo * sg.pair_chunk;
        const int blk = quotient(combo, p.div_hkv), g = combo - blk * p.Hkv;
        it.kv_head = g;
        it.a_end = sg.a_end;
        it.b_coord0 = sg.key0 + blk * sg.len;
        it.own_map = sg.own_map;
        // entries of this (segment, kv head), heaviest first: the packed tail tiles (last tile position of
        // the segment), then (tile position, q head) for the full positions
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
            const int e = 2 * pi + x;
            QSlot& s = it.s[x];
            s.valid = e < sg.entries;
            const bool tail = e < sg.tail_tiles;
            const int e2 = e - sg.tail_tiles, up = quotient(max(e2, 0), p.div_g);
            const int qt = tail ? sg.full_tiles : sg.full_tiles - 1 - up;
            const int n = tail ? e : e2 - up * p.G;  // of the tiles at this position
            const QTile& form = sg.form[tail];
            const int head = n * form.head_step, tok = qt * kTile + n * form.tok_step;
            s.q_head0 = g * p.G + head;
            s.row_div = form.heads;
            s.ntok = min(form.toks, sg.len - tok);
            s.nheads = min(form.heads, p.G - head);
            s.qmap = tail ? 1 + kind : 0;
            s.box_rows = form.box_rows;
            s.q_tok0 = it.seq * p.q_rows + sg.q0 + blk * sg.len + tok;
            s.limit0 = tok;
            s.end = tok + s.ntok;
            if (s.valid) own_keys = max(own_keys, s.end);
        }
    } else {
        const int rest = quotient(w, p.div_splits);
        it.split = w - rest * p.n_splits;
        const int q_pairs = cdiv(p.q_tiles, 2);
        const int g = quotient(rest, p.div_q_pairs);
        const int pi = rest - g * q_pairs;
        it.kv_head = g;
        it.a_end = 0;
        const int split_lo = it.split * p.tiles_per_split * kTile;
        it.b_coord0 = split_lo;
        it.own_map = 2;
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
            const int qt = 2 * pi + x;
            QSlot& s = it.s[x];
            s.valid = qt < p.q_tiles;
            const int tok0 = qt * p.tok_per_tile;
            const int ntok = max(0, min(p.tok_per_tile, p.Q - tok0));
            s.q_tok0 = it.seq * p.Q + tok0;
            s.q_head0 = g * p.G;
            s.row_div = p.G;
            s.ntok = ntok;
            s.nheads = p.G;
            s.qmap = 4;
            s.box_rows = p.G * p.tok_per_tile;
            s.limit0 = p.n_video + tok0 - split_lo;
            // keys past the last row's limit are never visible; a split that lies past it altogether still takes
            // one (wholly masked) tile and leaves the neutral partial
            s.end = max(0, min(p.n_video + tok0 + ntok - split_lo, p.tiles_per_split * kTile));
            if (s.valid) own_keys = max(own_keys, max(1, s.end));
        }
    }
#pragma unroll 1
    for (int x = 0; x < 2; ++x) it.s[x].per_div = static_cast<int>(ceilf(__fdiv_rn(65536.f, static_cast<float>(it.s[x].row_div))));
    it.na = cdiv(it.a_end, kTile);
    it.nt = own_keys > 0 ? it.na + cdiv(own_keys, kTile) : 0;
    it.n_a = (it.a_end - (it.na - 1) * kTile + 15) & ~15;
    it.n_b = (own_keys - (it.nt - it.na - 1) * kTile + 15) & ~15;
}

// Between the two softmax warps that share a scheduler (warp `quarter` of each warpgroup), hardware barriers of 64
// threads, one id per direction, all sixteen in use (the kernel has no __syncthreads: the cluster barrier stands at its
// start and end).  These have no limit: both warps go through the same tiles whatever happens, a timeout included, because
// they see the same work items (item_ready), so every pass meets its wait.  What the passing warp wrote to shared memory
// before is seen after the wait.  kPassMax: the row maxima of a tile; kPassTurn: the turn on
// the scheduler's special-function unit.
constexpr int kPassMax = 0, kPassTurn = 8;
__device__ __forceinline__ void pass_wait(int what, int wg, int quarter) {
    asm volatile("bar.sync %0, 64;" ::"r"(what + wg * 4 + quarter) : "memory");
}
__device__ __forceinline__ void pass_on(int what, int wg, int quarter) {
    asm volatile("bar.arrive %0, 64;" ::"r"(what + (wg ^ 1) * 4 + quarter) : "memory");
}

template <int D, int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ AttnMaps maps) {
    using L = AttnSmem<D>;
    constexpr int NP = L::kPanels;
    extern __shared__ uint8_t smem_raw[];
    // Barriers.  "first": the copy of the pair's first CTA is the one that is used (the MMA warps wait there and both
    // CTAs arrive); "both": each CTA has its own.
    struct Bars {
        uint64_t item_full[kItems], item_free[kItems];  // both: decoded items
        uint64_t clc;                                   // both: answer of the hardware queue
        uint64_t clc_read;                              // first: the second CTA has read it
        uint64_t q_full[2];                             // first
        uint64_t q_free[2];                             // both
        uint64_t k_full[kRing], v_full[kRing];          // first: a tile has landed in both CTAs
        uint64_t s_full[kRing];                         // both: QK(t) is complete: scores there, K tile consumed
        uint64_t s_read[2];                             // first: scores are in registers
        uint64_t p_full[2];                             // first: probabilities are written
        uint64_t pv_done[kRing];                        // both: PV(t) is complete: P and V tile consumed, O up to date
        uint64_t o_free;                                // first: both CTAs have read it
        uint64_t sums_full[kSums];                      // both: row sums of an item are in shared memory
        uint64_t go;                                    // first: the next item may be claimed
    };
    __shared__ Bars bars;
    __shared__ __align__(16) uint4 s_clc;
    __shared__ uint32_t tmem_base_slot;
    __shared__ WaitState wait_state;
    __shared__ unsigned s_published;     // work items so far; kNoMore added: there will be no others
    __shared__ WorkItem s_decoded[kItems];
    __shared__ float s_max[2][kTile];
    __shared__ float2 s_sums[kSums][2][kTile];  // (row sum, reference maximum) of the even and of the odd tiles:
                                              // added in this order, whichever warpgroup had them

    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // the same in all lanes, and known to be
    const int lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    constexpr int kConsumerWarps = 1 + 8 + 4;  // producer, softmax, epilogue; in the first CTA also the MMA warps

    if (tid == 0) {
        wait_state.tries = p.wait_tries;
        wait_state.expired = 0;
        s_published = 0;
        for (int i = 0; i < kItems; ++i) {
            mbar_init(smem_u32(&bars.item_full[i]), 1);
            mbar_init(smem_u32(&bars.item_free[i]), kConsumerWarps + (rank == 0 ? 2 : 0));
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars.q_full[i]), 1);
            mbar_init(smem_u32(&bars.q_free[i]), 1);
            mbar_init(smem_u32(&bars.s_read[i]), 8);  // 4 warps of each CTA
            mbar_init(smem_u32(&bars.p_full[i]), 8);
        }
        for (int i = 0; i < kRing; ++i) {
            mbar_init(smem_u32(&bars.k_full[i]), 1);
            mbar_init(smem_u32(&bars.v_full[i]), 1);
            mbar_init(smem_u32(&bars.s_full[i]), 1);
            mbar_init(smem_u32(&bars.pv_done[i]), 1);
        }
        for (int i = 0; i < kSums; ++i) mbar_init(smem_u32(&bars.sums_full[i]), 8);
        mbar_init(smem_u32(&bars.o_free), 8);
        mbar_init(smem_u32(&bars.go), 1);
        mbar_init(smem_u32(&bars.clc), 1);
        mbar_init(smem_u32(&bars.clc_read), 1);
        fence_mbar_init();
        if (MODE & 1) {
            tma_prefetch_desc(&maps.q[0]);
#pragma unroll 1
            for (int i = 0; i < 2; ++i) {
                tma_prefetch_desc(&maps.k[i]);
                tma_prefetch_desc(&maps.v[i]);
            }
        }
        if (MODE & 2) {
            tma_prefetch_desc(&maps.q[4]);
            tma_prefetch_desc(&maps.k[2]);
            tma_prefetch_desc(&maps.v[2]);
        }
    }
    if (warp == 12) {
        __syncwarp();
        tmem_alloc_pair(smem_u32(&tmem_base_slot), 512);
    }
    tc_fence_before_sync();
    cluster_sync_all();  // also: the other CTA's barriers are initialised before anything arrives on them
    tc_fence_after_sync();
    const uint32_t tmem_base = uniform(tmem_base_slot);
    // Every role reads its first item while the kernels before this one finish and then calls grid_wait(), before it touches
    // global memory or waits for what others fetch from there: the kernels before do not count towards the limit of a wait,
    // however many they are.  (All of them waiting before the first item is decoded: 0.45 us a launch.)
    grid_launch_dependents();

#ifdef PEVLM_TRACE
    __shared__ unsigned s_waits[16][kTraceIds];
    for (int i = lane; i < kTraceIds; i += 32) s_waits[warp][i] = 0;
    __syncwarp();
    const unsigned role_start = static_cast<unsigned>(clock64());
#define PEVLM_WAIT_ACCOUNT(which, call)                                                              \
    const unsigned before = static_cast<unsigned>(clock64());                                        \
    call;                                                                                            \
    if (lane == 0) s_waits[warp][which] += static_cast<unsigned>(clock64()) - before
#else
#define PEVLM_WAIT_ACCOUNT(which, call) call
#endif
    auto wait = [&](const uint64_t& bar, uint32_t parity, int which) {
        PEVLM_WAIT_ACCOUNT(which, mbar_wait(smem_u32(&bar), parity, wait_state, which));
    };
    auto wait_asleep = [&](const uint64_t& bar, uint32_t parity, int which) {
        PEVLM_WAIT_ACCOUNT(which, mbar_wait<100>(smem_u32(&bar), parity, wait_state, which));
    };
    // k-th item of the pair: wait for it, read from s_decoded[k % kItems], then give the slot back (once per warp).
    // Whether there is a k-th item has the same answer in every warp, a timeout included: it is decided in one word, where
    // the scheduler counts item k in before it lets anyone have it and a wait that runs out says that there are no more,
    // whichever comes first.  (Warps that disagreed would wait for one another in pass_wait, without a limit.)
    auto item_ready = [&](int k) {
        wait(bars.item_full[k % kItems], (k / kItems) & 1, kWaitItem);
        if (static_cast<int>(*static_cast<volatile unsigned*>(&s_published) & ~kNoMore) > k) return true;
        return static_cast<int>(atomicOr(&s_published, kNoMore) & ~kNoMore) > k;
    };
    auto item_release = [&](int k) { mbar_arrive(smem_u32(&bars.item_free[k % kItems])); };
    auto wait_s_full = [&](uint32_t t, int which) { wait(bars.s_full[t % kRing], (t / kRing) & 1, which); };
    auto wait_pv_done = [&](uint32_t t, int which) { wait(bars.pv_done[t % kRing], (t / kRing) & 1, which); };

    // register budget per warpgroup: 2 x 184 (softmax) + 96 (epilogue) + 48 (the rest) = 4 x 128
    if (warp >= 12) {
        reg_dealloc<48>();
        if (warp == 15) {
            // --------------------------------------------------------- scheduler
            if (lane == 0) {
                int w = static_cast<int>(blockIdx.x >> 1);
                int published = 0, asked = 0;
                // After a timeout the clusters that are still to be launched do nothing (those of the first wave may find
                // an older call's status, so they do not look).
                if (w >= kNumSms / 2) {
                    grid_wait();
                    if (*reinterpret_cast<volatile int32_t*>(&p.hdr->status) != 0) w = -1;
                }
                while (true) {
                    const int slot = published % kItems;
                    if (published >= kItems) {
                        wait_asleep(bars.item_free[slot], (published / kItems - 1) & 1, kWaitItemFree);
                        if (!mbar_try_wait(smem_u32(&bars.item_free[slot]), (published / kItems - 1) & 1)) w = -2;  // may still be read
                    }
                    bool some = false;
                    if (w >= 0) {
                        decode_item<MODE>(p, w, s_decoded[slot]);
                        some = s_decoded[slot].nt > 0;  // padding of the item list is skipped
                    }
                    if (w < 0 || some) {
                        __threadfence_block();
                        if (w < 0) atomicOr(&s_published, kNoMore);
                        else if (atomicCAS(&s_published, published, published + 1) != static_cast<unsigned>(published)) w = -1;
                        if (w != -2) mbar_arrive(smem_u32(&bars.item_full[slot]));  // release: the decoded item is visible
                        if (w < 0) break;
                        ++published;
                        if (published == 1) grid_wait();
                        // the next item is claimed when the loads of this one near their end, so that a pair never
                        // sits on work another one could take
                        if (rank == 0) wait_asleep(bars.go, (published - 1) & 1, kWaitGo);
                    }
                    mbar_arrive_expect_tx(smem_u32(&bars.clc), 16);
                    if (rank == 0) {
                        if (asked > 0) wait_asleep(bars.clc_read, (asked - 1) & 1, kWaitClc);
                        clc_try_cancel(smem_u32(&s_clc), smem_u32(&bars.clc));
                    }
                    wait_asleep(bars.clc, asked & 1, kWaitClc);
                    const int first = clc_first_block(smem_u32(&s_clc));
                    fence_proxy_async_smem();  // the answer is written again by the asynchronous proxy
                    if (rank == 1) mbar_arrive_cluster(map_to_cta(smem_u32(&bars.clc_read), 0));
                    w = (first < 0 || *static_cast<volatile int*>(&wait_state.expired) != 0) ? -1 : first >> 1;
                    ++asked;
                }
            }
        } else if (warp == 13) {
            // --------------------------------------------------------- TMA producer: K(s), then V(s - kQkAhead)
            // (The whole warp runs this with uniform values; single lanes issue.)
            {
                // The K cursor's item, and where V has to come from: the rows of the last kQkAhead K tiles (base row of the
                // tile, kv head and map, sequence), the V tile of a step being that of kQkAhead steps ago.
                int k = -1, j = 0, nt = 0, na = 0, n_a = 0, n_b = 0, kv_head = 0, b_coord0 = 0, own_map = 0, seq = 0;
                int v_row[kQkAhead], v_from[kQkAhead], v_seq[kQkAhead];
                uint32_t tiles = 0;  // K tiles loaded so far
                bool more = true;
#pragma unroll 1
                for (uint32_t s = 0; more || s < tiles + kQkAhead; ++s) {
                    if (more && j == nt) {
                        more = uniform(item_ready(++k));
                        if (more) {
                            const WorkItem& it = s_decoded[k % kItems];
                            const QSlot& q = it.s[rank];
                            j = 0;
                            nt = uniform(it.nt); na = uniform(it.na); n_a = uniform(it.n_a); n_b = uniform(it.n_b);
                            kv_head = uniform(it.kv_head); b_coord0 = uniform(it.b_coord0); own_map = uniform(it.own_map);
                            seq = uniform(it.seq);
                            const int qm = uniform(q.qmap), q_head0 = uniform(q.q_head0), q_tok0 = uniform(q.q_tok0);
                            const int valid = uniform(q.valid);
                            const int rows = uniform((it.s[0].valid ? it.s[0].box_rows : 0) + (it.s[1].valid ? it.s[1].box_rows : 0));
                            __syncwarp();
                            if (lane == 0) item_release(k);
                            if (k == 0) grid_wait();
                            const int qb = k & 1;
                            if (k >= 2) wait(bars.q_free[qb], ((k >> 1) - 1) & 1, kWaitQFree);
                            if (rank == 0 && lane == 0) mbar_arrive_expect_tx(smem_u32(&bars.q_full[qb]), static_cast<uint32_t>(NP * 128 * rows));
                            if (valid) {
                                const uint32_t bar = map_to_cta(smem_u32(&bars.q_full[qb]), 0);
#pragma unroll 1
                                for (int h = 0; h < NP; ++h)
                                    tma_load_3d_pair(smem_base + L::kQ + qb * L::kQBytes + h * L::kQPanelBytes, &maps.q[MODE == 2 ? 4 : qm],
                                                     h * 64, q_head0, q_tok0, bar, l2_evict_first());
                            }
                        }
                    }
                    // Rows past the end of the sink, and past the end of the block range, are outside their tensor map, in
                    // every sequence of a batch, and arrive as zeros: a ragged last tile brings in no rows of the range or
                    // the sequence behind it, whatever those hold (a probability of 0 times a NaN in V would be one).
                    int row = 0, from = 0;
                    if (more) {
                        if (rank == 0 && lane == 0 && j == max(0, nt - kClaimAhead)) mbar_arrive(smem_u32(&bars.go));
                        const int map = MODE == 2 ? 2 : j < na ? 1 : own_map;
                        const int n = j == na - 1 ? n_a : j == nt - 1 ? n_b : kTile;  // this CTA's keys: half of them
                        row = j < na ? j * kTile : b_coord0 + (j - na) * kTile;
                        from = kv_head * 4 + map;
                        const uint32_t slot = tiles % kRing;
                        if (tiles >= kRing) wait_s_full(tiles - kRing, kWaitKvFree);
                        if (rank == 0 && lane == 0) mbar_arrive_expect_tx(smem_u32(&bars.k_full[slot]), 2 * L::kKBytes);
                        const uint32_t bar = map_to_cta(smem_u32(&bars.k_full[slot]), 0);
#pragma unroll 1
                        for (int h = 0; h < NP; ++h)
                            tma_load_4d_pair(smem_base + L::kK + slot * L::kKBytes + h * L::kKPanelBytes, &maps.k[map], h * 64, kv_head,
                                             row + static_cast<int>(rank) * (n >> 1), seq, bar);
                        ++j;
                        ++tiles;
                    }
                    if (s >= kQkAhead && s - kQkAhead < tiles) {
                        const uint32_t u = s - kQkAhead, slot = u % kRing;
                        if (u >= kRing) wait_pv_done(u - kRing, kWaitKvFree);
                        if (rank == 0 && lane == 0) mbar_arrive_expect_tx(smem_u32(&bars.v_full[slot]), 2 * L::kVBytes);
                        tma_load_4d_pair(smem_base + L::kV + slot * L::kVBytes, &maps.v[v_from[0] & 3], static_cast<int>(rank) * (D / 2),
                                         v_from[0] >> 2, v_row[0], v_seq[0], map_to_cta(smem_u32(&bars.v_full[slot]), 0));
                    }
#pragma unroll
                    for (int i = 0; i < kQkAhead - 1; ++i) {
                        v_row[i] = v_row[i + 1];
                        v_from[i] = v_from[i + 1];
                        v_seq[i] = v_seq[i + 1];
                    }
                    v_row[kQkAhead - 1] = row;
                    v_from[kQkAhead - 1] = from;
                    v_seq[kQkAhead - 1] = seq;
                }
            }
        } else if (rank == 0 && warp == 12) {
            // --------------------------------------------------------- S = Q K^T of the pair
            // All 32 lanes run this loop with warp-uniform values (descriptors and addresses stay in
            // uniform registers); the MMA and commit instructions themselves go out from one elected lane.
            uint32_t t = 0;
#pragma unroll 1
            for (int k = 0; uniform(item_ready(k)); ++k) {
                const WorkItem& it = s_decoded[k % kItems];
                const int nt = uniform(it.nt), na = uniform(it.na), n_a = uniform(it.n_a), n_b = uniform(it.n_b);
                __syncwarp();
                if (lane == 0) item_release(k);
                const uint32_t q_lo = desc_lo(smem_base + L::kQ + (k & 1) * L::kQBytes, 16);
                if (k == 0) grid_wait();
                wait(bars.q_full[k & 1], (k >> 1) & 1, kWaitQ);
#pragma unroll 1
                for (int j = 0; j < nt; ++j, ++t) {
                    const int n = j == na - 1 ? n_a : j == nt - 1 ? n_b : kTile;
                    const uint32_t slot = t % kRing;
                    wait(bars.k_full[slot], (t / kRing) & 1, kWaitK);
                    if (t >= 2) wait(bars.s_read[t & 1], ((t >> 1) - 1) & 1, kWaitSRead);
                    tc_fence_after_sync();
                    mma_ss_batch<D / 16>(tmem_base + (t & 1) * kTile, q_lo, desc_lo(smem_base + L::kK + slot * L::kKBytes, 16),
                                         make_idesc_bf16(2 * kTile, n, false));
                    mma_commit_pair(smem_u32(&bars.s_full[slot]));
                }
                mma_commit_pair(smem_u32(&bars.q_free[k & 1]));
            }
        } else if (rank == 0 && warp == 14) {
            // --------------------------------------------------------- O += P V of the pair
            constexpr uint32_t kIdescPv = make_idesc_bf16(2 * kTile, D, true);
            const uint32_t d_tmem = tmem_base + kTmemO;
            uint32_t t = 0;
#pragma unroll 1
            for (int k = 0; uniform(item_ready(k)); ++k) {
                const WorkItem& it = s_decoded[k % kItems];
                const int nt = uniform(it.nt), na = uniform(it.na), n_a = uniform(it.n_a), n_b = uniform(it.n_b);
                __syncwarp();
                if (lane == 0) item_release(k);
                // the previous item's output must have left TMEM before O is overwritten
                if (k > 0) wait(bars.o_free, (k - 1) & 1, kWaitOFree);
                else grid_wait();
#pragma unroll 1
                for (int j = 0; j < nt; ++j, ++t) {
                    const int n = j == na - 1 ? n_a : j == nt - 1 ? n_b : kTile;
                    const uint32_t slot = t % kRing;
                    const uint32_t v_lo = desc_lo(smem_base + L::kV + slot * L::kVBytes, 0);
                    const uint32_t a_tmem = tmem_base + kTmemP + (t & 1) * (kTile / 2);
                    wait(bars.v_full[slot], (t / kRing) & 1, kWaitV);
                    wait(bars.p_full[t & 1], (t >> 1) & 1, kWaitP);
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int ks = 0; ks < (n >> 4); ++ks)
                        mma_ts_step<D>(d_tmem, a_tmem + ks * 8, v_lo + ks * kVDescStep<D>, kIdescPv, j + ks);
                    mma_commit_pair(smem_u32(&bars.pv_done[slot]));
                }
            }
        }
    } else if (warp >= 8) {
        // ------------------------------------------------------------- epilogue
        reg_dealloc<96>();
        grid_wait();
        // The status word of the previous call on this workspace is cleared by the launch's first block, long before any
        // wait of this launch can have run out.
        if (blockIdx.x == 0 && tid == 256 && !p.keep_status) {
            p.hdr->detail = 0;
            *reinterpret_cast<volatile int32_t*>(&p.hdr->status) = 0;
            if (MODE == 3) p.hdr_question->status = p.hdr_question->detail = 0;
        }
        const int row = tid & 127;
        const uint32_t tO = tmem_base + kTmemO + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t o_free_bar = map_to_cta(smem_u32(&bars.o_free), 0);
        uint32_t t_end = 0;  // tiles up to the end of this item
#pragma unroll 1
        for (int k = 0; uniform(item_ready(k)); ++k) {
            const WorkItem& it = s_decoded[k % kItems];
            const QSlot& qs = it.s[rank];
            t_end += it.nt;
            const int row_tok = row * qs.per_div >> 16, row_head = row - row_tok * qs.row_div;
            const bool row_ok = qs.valid && (row_tok < qs.ntok) && (row_head < qs.nheads);
            const int tok = qs.q_tok0 + row_tok;
            const int head = qs.q_head0 + row_head;
            const int split = it.split, seq = it.seq;
            const bool question = MODE == 2 || (MODE == 3 && it.own_map == 2);
            const bool partial = question && p.n_splits > 1;  // left to the merge
            __syncwarp();
            if (lane == 0) item_release(k);
            wait_asleep(bars.sums_full[k % kSums], (k / kSums) & 1, kWaitSum);
            const float2 sa = s_sums[k % kSums][0][row], sb = s_sums[k % kSums][1][row];
            const float m = fmaxf(sa.y, sb.y);
            const float l = m == -INFINITY ? 0.f
                                           : sa.x * fast_exp2((sa.y - m) * p.scale_log2) + sb.x * fast_exp2((sb.y - m) * p.scale_log2);
            const float inv_l = (l > 0.f) ? 1.f / l : 0.f;
            const float lse_val = (l > 0.f) ? m * p.scale + logf(l) : -INFINITY;
            wait_pv_done(t_end - 1, kWaitODone);
            tc_fence_after_sync();
            // 32 columns at a time, in a loop that stays one; 32 bytes per store: every lane writes whole sectors of
            // its own row
            // (tok counts over the batch; the partials are ordered sequence, split, token, head)
            const size_t r = !partial ? static_cast<size_t>(tok) * p.Hq + head
                                      : (static_cast<size_t>(seq * (p.n_splits - 1) + split) * p.Q + tok) * p.Hq + head;
            __nv_bfloat16* const out = question ? p.o_question : p.o;
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
                uint32_t o[32];
                tmem_ld32(tO + c * 32, o);
                tmem_wait_ld();
                if (c == D / 32 - 1) {  // the accumulator may be written again
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(o_free_bar);
                }
                if (!partial) {
                    uint32_t wd[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float x, y;
                        unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1])), pack_f32x2(inv_l, inv_l)), x, y);
                        wd[e] = pack_bf16x2(x, y);
                    }
                    if (row_ok) {
#pragma unroll
                        for (int v = 0; v < 2; ++v)
                            st_global_v8(out + r * D + c * 32 + v * 16, *reinterpret_cast<uint32_t(*)[8]>(&wd[8 * v]));
                    }
                } else if (row_ok) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * inv_l);
#pragma unroll
                    for (int v = 0; v < 4; ++v) st_global_v8(p.part_o + r * D + c * 32 + v * 8, *reinterpret_cast<uint32_t(*)[8]>(&o[8 * v]));
                }
            }
            float* const lse = partial ? p.part_lse : question ? p.lse_question : p.lse;
            const int rows = question ? p.Q : p.q_rows;  // of a sequence
            const size_t at = partial ? r : static_cast<size_t>(seq * p.Hq + head) * rows + (tok - seq * rows);
            if (row_ok && lse) st_global_stream_f32(lse + at, lse_val);
        }
    } else {
        // ------------------------------------------------------------- softmax, every other key tile
        reg_alloc<184>();
        const int wg = warp >> 2, quarter = warp & 3;
        const int row = tid & 127;
        const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
        const uint32_t p_bar = map_to_cta(smem_u32(&bars.p_full[wg]), 0), s_read_bar = map_to_cta(smem_u32(&bars.s_read[wg]), 0);
        const uint32_t tS = tmem_base + wg * kTile + lane_off, tP = tmem_base + kTmemP + wg * (kTile / 2) + lane_off;
        const uint32_t tO = tmem_base + kTmemO + lane_off;
        uint32_t t0 = 0;                // tiles of all items so far
#pragma unroll 1
        for (int k = 0; uniform(item_ready(k)); ++k) {
            const WorkItem& it = s_decoded[k % kItems];
            const QSlot& qs = it.s[rank];
            const int nt = uniform(it.nt), na = uniform(it.na), a_end = uniform(qs.valid ? it.a_end : 0);  // a slot without a tile sees nothing
            const int row_tok = row * qs.per_div >> 16;
            // this row's last visible key and the smallest such key of the tile, counted from the own range's start
            const int end = uniform(qs.valid ? qs.end : 0), first_limit = uniform(qs.limit0);
            const int my_limit = min(first_limit + row_tok, end - 1), limit0 = min(first_limit, end - 1);
            __syncwarp();
            if (lane == 0) item_release(k);
            if (k == 0) grid_wait();
            float m_own = -INFINITY;  // reference maximum (raw score units) this warpgroup's row sum is scaled by
            float l_run = 0.f;
            const int first = static_cast<int>((t0 ^ static_cast<uint32_t>(wg)) & 1u);  // this warpgroup has the even or the odd tiles
#pragma unroll 1
            for (int j = first; j < nt; j += 2) {
                const uint32_t t = t0 + j;
                // keys of this tile that the row sees, and that every row of the query tile sees
                const int max_col = j < na ? a_end - j * kTile : my_limit + 1 - (j - na) * kTile;
                const bool need_mask = (j < na ? a_end - j * kTile : limit0 + 1 - (j - na) * kTile) < kTile;
                wait_s_full(t, kWaitS);
                tc_fence_after_sync();
                // all 128 scores of the row in registers: one round trip to TMEM
                uint32_t r[kTile];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32 * c]));
                tmem_wait_ld();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(s_read_bar);
                if (need_mask) {
                    // by 32 columns: on the diagonal the rows of a warp differ within one such part only, the others are
                    // visible or hidden as a whole (a compare for each of the 128 columns took 1,200 cycles a tile)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int cols = max_col - c * 32;  // visible ones of this part
                        if (__all_sync(0xffffffffu, cols >= 32)) continue;
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (i >= cols) r[c * 32 + i] = 0xff800000u;  // -inf
                    }
                }
                float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int i = 0; i < kTile; i += 8) {
#pragma unroll
                    for (int a = 0; a < 4; ++a)
                        mx[a] = fmax3(mx[a], __uint_as_float(r[i + 2 * a]), __uint_as_float(r[i + 2 * a + 1]));
                }
                const float m_tile = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                // the row's reference maximum after tile t - 1 comes from the other warpgroup
                float m_prev = -INFINITY;
                if (t > 0) {
                    pass_wait(kPassMax, wg, quarter);
                    if (j > 0) m_prev = s_max[wg ^ 1][row];
                }
                float m_ref = m_prev;
                if ((m_tile - m_prev) * p.scale_log2 > kRescaleThresholdLog2 || m_prev == -INFINITY) m_ref = fmaxf(m_prev, m_tile);
                s_max[wg][row] = m_ref;
                pass_on(kPassMax, wg, quarter);
                if (j > 0 && __any_sync(0xffffffffu, m_ref != m_prev)) {
                    // rare: rescale this row of the O accumulator in place, once PV(t - 1) has landed
                    const float alpha = m_ref == m_prev ? 1.f : fast_exp2((m_prev - m_ref) * p.scale_log2);
                    wait_pv_done(t - 1, kWaitPV);
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int c = 0; c < D / 16; ++c) {
                        uint32_t o[16];
                        tmem_ld16(tO + c * 16, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st16(tO + c * 16, o);
                    }
                }
                if (t >= 2) wait_pv_done(t - 2, kWaitPFree);  // this probability buffer has been read
                if (t > 0) pass_wait(kPassTurn, wg, quarter);
                const float neg_ms = (m_ref == -INFINITY) ? 0.f : -m_ref * p.scale_log2;
                // probabilities as bf16 pairs; scale-and-shift and the row sum run as packed fp32 pairs
                const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
                const uint64_t shift2 = pack_f32x2(neg_ms, neg_ms);
                uint64_t sm2[4] = {0ull, 0ull, 0ull, 0ull};
                uint32_t pk[kTile / 2];
#pragma unroll
                for (int i = 0; i < kTile / 2; ++i) {
                    const uint64_t t2 = fma_f32x2(pack_f32x2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])), scale2, shift2);
                    float e0, e1;
                    unpack_f32x2(t2, e0, e1);
                    const float p0 = fast_exp2(e0), p1 = fast_exp2(e1);
                    sm2[i & 3] = add_f32x2(sm2[i & 3], pack_f32x2(p0, p1));
                    pk[i] = pack_bf16x2(p0, p1);
                    if (i % 16 == 15) tmem_st16(tP + i - 15, &pk[i - 15]);
                    if (i == kTurn) pass_on(kPassTurn, wg, quarter);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(p_bar);
                float a0, a1, b0, b1;
                unpack_f32x2(add_f32x2(sm2[0], sm2[1]), a0, a1);
                unpack_f32x2(add_f32x2(sm2[2], sm2[3]), b0, b1);
                const float sum = (a0 + a1) + (b0 + b1);
                l_run = (m_own == m_ref ? l_run : l_run * fast_exp2((m_own - m_ref) * p.scale_log2)) + sum;
                m_own = m_ref;
#ifdef PEVLM_TRACE
                if (lane == 0) ++s_waits[warp][1];
#endif
            }
            t0 += nt;
            s_sums[k % kSums][first][row] = make_float2(l_run, m_own);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.sums_full[k % kSums]));
        }
        if (t0 > 0 && static_cast<uint32_t>(wg) == (t0 & 1u)) {  // the last tile's passes
            pass_wait(kPassMax, wg, quarter);
            pass_wait(kPassTurn, wg, quarter);
        }
    }
#ifdef PEVLM_TRACE
    __syncwarp();
    if (lane == 0) s_waits[warp][0] = static_cast<unsigned>(clock64()) - role_start;
    __syncwarp();
    if (blockIdx.x < 2)
        for (int i = lane; i < kTraceIds; i += 32) g_waits[blockIdx.x][warp][i] = s_waits[warp][i];
#endif
    // A wait that ran out may have left loads, MMAs or an answer of the hardware queue on their way into this pair's memory.
    // They take microseconds; the pair stays until they have had tens of them.
    if (*static_cast<volatile int*>(&wait_state.expired) != 0) {
#pragma unroll 1
        for (int i = 0; i < kDrainUs; ++i) __nanosleep(1000);
    }
    tc_fence_before_sync();
    __syncwarp();
    cluster_sync_all();  // neither CTA leaves, or frees TMEM, while the other may still reach it
    if (warp == 12) {
        __syncwarp();
        tmem_dealloc_pair(tmem_base, 512);
    }
    if (tid == 0 && wait_state.expired != 0) {
        const int detail = wait_state.expired * 1000000 + blockIdx.x;
        if (atomicCAS(&p.hdr->status, 0, PEVLM_ETIMEOUT) == 0) p.hdr->detail = detail;
        if (MODE == 3 && atomicCAS(&p.hdr_question->status, 0, PEVLM_ETIMEOUT) == 0) p.hdr_question->detail = detail;
    }
}

cudaError_t launch_attn(const AttnParams& p, int head_dim, const AttnMaps& m, cudaStream_t stream) {
    const int64_t items = static_cast<int64_t>(p.n_items) * p.batch;
    if (items <= 0) return cudaSuccess;
    const size_t smem = attn_smem_bytes(head_dim);
    // one cluster per work item; those that run take the rest from the hardware's queue
    const unsigned grid = 2u * static_cast<unsigned>(items);
#define PEVLM_GO(D_, M_) launch_chained<attn_kernel<D_, M_>>(grid, kAttnThreads, smem, stream, p, m)
    if (head_dim == 128) return p.mode == 1 ? PEVLM_GO(128, 1) : p.mode == 2 ? PEVLM_GO(128, 2) : PEVLM_GO(128, 3);
    return p.mode == 1 ? PEVLM_GO(64, 1) : p.mode == 2 ? PEVLM_GO(64, 2) : PEVLM_GO(64, 3);
#undef PEVLM_GO
}

}  // namespace pevlm
