// RoPE at global positions (Sec. 3.2.2): every token keeps its original sequential position.
// HBM-bound elementwise kernel.  The result is that of the fp64 definition: angle, sine/cosine and rotation in fp64 (no
// fused multiply-add in the rotation, so every fp64 operation rounds exactly once), then one rounding fp64 -> fp32 ->
// bf16 (round to nearest even).
//
// The CTAs share the tokens out in groups of up to 4 neighbours (8 with few heads).  A CTA evaluates a group's angles once (fp64 sincos)
// into shared memory, one group ahead, and its threads walk over the group's head vectors of Q and K: d/16 threads a
// vector, 16 bytes of either half each; the vectors of a group are one contiguous range per tensor.  What bounds it: DRAM
// traffic.  Two things used to stand in the way (numbers for B200, 28/4 heads of 128):
//   - the fp64 <-> fp32 conversion unit (16 values per clock and SM, 70 % busy at 50K tokens).  The rotation therefore
//     runs in fp32, with the sine and cosine rounded to fp32, and takes its result r only where it cannot differ: where
//     r - E and r + E, E = 2^-23 (|a| + |b|), round to the same bf16 (see rotate2 for why that is enough).  Elsewhere
//     (about one head vector of a warp in sixteen) the thread repeats its eight pairs in fp64;
//   - the bytes in flight, above all in ranges that do not fill the GPU many times over (12.5K tokens took 73 us where
//     50K took 148).  The loads go through a ring in shared memory, kRing vectors ahead, over the ends of groups
//     too, which costs no registers.  A thread reads only what it has fetched itself, so the ring needs no barrier.
// The V rows of the same tokens can be copied along (V needs no rotation): a third range of vectors.
#include "internal.h"
#include "ptx.cuh"

namespace pevlm {

// Threads of a CTA, CTAs of an SM, most tokens of a group and vectors a thread has in flight.  With V copied along, 50K tokens of
// 28/4 heads take 171 us with groups of 8 and a ring of 6, 151 with 4 and 6, 150 with 4 and 5, 164 with 2 and 6; two CTAs per SM
// with longer rings are faster at 32/8 heads only (130 against 148 us for 33K tokens), slower everywhere else.
// FEW: calls with few heads (launch_rope).  There is little to rotate for each angle then: the fp64 evaluations, some 240 cycles
// for a warp on its scheduler, are the larger part, and with groups of four tokens in large CTAs the warps wait for one another's
// (33K tokens of 8/2 heads of 128 with V 45.7 us, 38.9 in this form; 1/1 heads 26.9, 17.2; rings of 5 and five CTAs 39.5, 17.6; 64
// registers and eight CTAs 41.7 for 8/2 heads without V where this form takes 36.7).
template <bool FEW>
struct RopeForm {
    static constexpr int kThreads = FEW ? 128 : 256;
    static constexpr int kCtasPerSm = FEW ? 6 : 3;
    static constexpr int kTokens = FEW ? 8 : 4;
    static constexpr int kRing = FEW ? 3 : 5;
};

// 16-byte accesses that do not allocate in L1 (every byte is touched once)
__device__ __forceinline__ void fetch16(uint32_t dst, const __nv_bfloat16* src, uint64_t l2_policy) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(l2_policy) : "memory");
}
__device__ __forceinline__ void st_stream(__nv_bfloat16* p, const uint4& v) {
    asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// bf16 -> fp64 is exact (widen through fp32).
__device__ __forceinline__ double bf16_bits_to_f64(uint32_t bits16) {
    return static_cast<double>(__uint_as_float(bits16 << 16));
}

// Two rotation pairs (a0, b0), (a1, b1), packed as bf16 words: outputs of both halves, and whether any of the four could
// round differently from the exact value.  cs = (cos0, cos1, sin0, sin1).  least: the smallest |a| + |b| - 1 as bits, so
// that zero counts as the largest.
//
// Why r = fl(a C - fl(b S)) may be taken where lo = fl(r - E) and hi = fl(r + E) round to the same bf16.  Let x be the
// fp64 result and t = fl(x), M = |a| + |b| in [2^k, 2^(k+1)), u = 2^(k-23) (fp32's spacing there); E >= u, as fl(M) >= 2^k.
// Rounding is monotone, so lo <= t <= hi is enough.  |x - r| is at most 2^-25 M (C and S, of magnitude <= 1) + half a
// spacing at b S + half a spacing at r, and fp64's own 2^-51 M.
//   - r >= 2^k (magnitudes), M >= 1.34 * 2^k: at most 2^-25 M + u <= 3.99 * 2^-25 M < E (fl(M) is off by 2^-24 M).
//   - r >= 2^k, M < 1.34 * 2^k: at most 1.34 u, so t is less than 2 u off.  Both lie on the grid of u: t is r or its
//     neighbour, and lo and hi reach the neighbours.  (t below 2^k: then everything is within 4 u of 2^k, which is
//     itself a bf16, and rounds to it.)  This is the one case where |x - r| does exceed E, by up to a third.
//   - r < 2^k: half a spacing at r is u / 4, in all at most 2^-25 M + 3/4 u <= 3.98 * 2^-25 M < E from M = 1.01 * 2^k on, and
//     below that at most 1.003 u with t and r on the grid of u / 2 (or finer, with smaller terms): t is at most u off, as above.
// The second output is the same with a and b exchanged.  M >= 2^-126 is needed: below, the spacing stays 2^-149, E is less than
// that and t may be r's neighbour unnoticed (5 of 10^7 outputs differed).  Such pairs, both subnormal and not both zero, count
// as unsure; M = 0 gives an exact zero (with the sign checked by lo and hi).  (The check is
// nine instructions: 12.6K tokens 267.7 -> 268.8 us a layer, 50K tokens 1,741 -> 1,744.)
__device__ __forceinline__ uint32_t rotate2(uint32_t a, uint32_t b, const float4& cs, uint32_t& out_a, uint32_t& out_b, uint32_t& least) {
    const float a0 = __uint_as_float(a << 16), a1 = __uint_as_float(a & 0xffff0000u);
    const float b0 = __uint_as_float(b << 16), b1 = __uint_as_float(b & 0xffff0000u);
    const uint64_t A = pack_f32x2(a0, a1), B = pack_f32x2(b0, b1);
    const uint64_t C = pack_f32x2(cs.x, cs.y), S = pack_f32x2(cs.z, cs.w), nS = pack_f32x2(-cs.z, -cs.w);
    const uint64_t ra = fma_f32x2(A, C, mul_f32x2(B, nS)), rb = fma_f32x2(B, C, mul_f32x2(A, S));
    const float m0 = fabsf(a0) + fabsf(b0), m1 = fabsf(a1) + fabsf(b1);
    least = __viaddmin_u32(__float_as_uint(m0), ~0u, __viaddmin_u32(__float_as_uint(m1), ~0u, least));
    const uint64_t m = pack_f32x2(m0, m1);
    const float e = 1.0f / 8388608.0f;  // 2^-23
    const uint64_t up = pack_f32x2(e, e), down = pack_f32x2(-e, -e);
    float x0, x1, y0, y1;
    unpack_f32x2(fma_f32x2(m, up, ra), x0, x1);
    unpack_f32x2(fma_f32x2(m, down, ra), y0, y1);
    out_a = pack_bf16x2(x0, x1);
    const uint32_t other_a = pack_bf16x2(y0, y1);
    unpack_f32x2(fma_f32x2(m, up, rb), x0, x1);
    unpack_f32x2(fma_f32x2(m, down, rb), y0, y1);
    out_b = pack_bf16x2(x0, x1);
    return (out_a ^ other_a) | (out_b ^ pack_bf16x2(y0, y1));
}

template <int D, bool FEW>
struct RopeSmem {
    using F = RopeForm<FEW>;
    static constexpr int kHalf = D / 2;
    // per token: [pair / 2 of the thread][thread of the vector], so that the threads of a vector read 16 contiguous bytes each
    float4 cs32[2][F::kTokens * kHalf / 2];   // (cos0, cos1, sin0, sin1) of two pairs
    double2 cs64[2][F::kTokens * kHalf];      // (cos, sin), [pair of the thread][thread of the vector]
    uint4 ring[F::kRing][2][F::kThreads];    // [half of the vector][thread]
};

template <int D, bool FEW>
__global__ void __launch_bounds__(RopeForm<FEW>::kThreads, RopeForm<FEW>::kCtasPerSm) rope_kernel(const __grid_constant__ RopeParams p) {
    constexpr int kRopeThreads = RopeForm<FEW>::kThreads, kRopeRing = RopeForm<FEW>::kRing;
    constexpr int HALF = D / 2;
    constexpr int TPV = HALF / 8;                // threads per head vector: 8 rotation pairs each
    constexpr int SLOTS = kRopeThreads / TPV;    // vectors the CTA has in hand at a time
    extern __shared__ __align__(16) uint8_t raw[];
    RopeSmem<D, FEW>& sm = *reinterpret_cast<RopeSmem<D, FEW>*>(raw);
    const int v = threadIdx.x % TPV, slot = threadIdx.x / TPV;
    const int i0 = v * 8;
    const int heads = p.Hq + p.Hkv + p.Hv;

    // groups of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ... of p.group tokens each
    const int64_t stride = static_cast<int64_t>(gridDim.x) * p.group;
    auto size_of = [&](int64_t tok0) { return static_cast<int>(p.n_tokens - tok0 < p.group ? p.n_tokens - tok0 : p.group); };
    // The pair that this thread forms angles of: always the same one, so its frequency is read once (the lanes of a warp read
    // different words of constant memory, one after another).  One position per token, or, multimodal, the component that the
    // pair's section picks.
    static_assert(kRopeThreads % HALF == 0, "a thread keeps its pair");
    const int pair = threadIdx.x % HALF;
    const double freq = p.inv_freq[pair];
    const int comp = pair < p.sec_end0 ? 0 : pair < p.sec_end1 ? 1 : 2;
    auto angles = [&](int64_t tok0, int buf) {
        if (tok0 >= p.n_tokens) return;
        for (int t = threadIdx.x / HALF; t < size_of(tok0); t += kRopeThreads / HALF) {
            const int64_t tok = tok0 + t;
            const int64_t seq = p.n_tokens == p.seq_len ? 0 : quotient(static_cast<int>(tok), p.div_seq);
            const int64_t pos = p.pos3 ? p.pos3[(2 * seq + comp) * p.seq_len + tok]
                              : p.pos_ids ? p.pos_ids[tok]
                                          : p.first_token + tok - seq * p.seq_len;
            double sn, cn;
            sincos(__dmul_rn(static_cast<double>(pos), freq), &sn, &cn);
            const int e = pair % 8, w = pair / 8;
            sm.cs64[buf][t * HALF + e * TPV + w] = make_double2(cn, sn);
            float* f = reinterpret_cast<float*>(&sm.cs32[buf][t * (HALF / 2) + (e / 2) * TPV + w]);
            f[e % 2] = __double2float_rn(cn);
            f[2 + e % 2] = __double2float_rn(sn);
        }
    };
    const uint64_t once = l2_evict_first();
    // fetch cursor: kRopeRing vectors ahead of the one that is rotated
    int64_t f_tok0 = static_cast<int64_t>(blockIdx.x) * p.group;
    int f_u = slot, f_total = f_tok0 < p.n_tokens ? size_of(f_tok0) * heads : 0, f_ring = 0;
    auto fetch = [&]() {
        if (f_tok0 < p.n_tokens) {
            if (f_u < f_total) {
                const int nt = size_of(f_tok0), nq = nt * p.Hq, nqk = nq + nt * p.Hkv;
                const __nv_bfloat16* src = f_u < nq ? p.q_in + (f_tok0 * p.Hq + f_u) * D
                                         : f_u < nqk ? p.k_in + (f_tok0 * p.Hkv + (f_u - nq)) * D
                                                     : p.v_in + (f_tok0 * p.Hv + (f_u - nqk)) * D;
                fetch16(smem_u32(&sm.ring[f_ring][0][threadIdx.x]), src + i0, once);
                fetch16(smem_u32(&sm.ring[f_ring][1][threadIdx.x]), src + i0 + HALF, once);
            }
            f_u += SLOTS;
            if (f_u - slot >= f_total) {  // the same for all threads: every thread takes the same number of steps
                f_tok0 += stride;
                f_u = slot;
                f_total = f_tok0 < p.n_tokens ? size_of(f_tok0) * heads : 0;
            }
        }
        f_ring = f_ring + 1 == kRopeRing ? 0 : f_ring + 1;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    grid_launch_dependents();
    // The first group's angles need nothing from the kernels before this one unless positions are given: they are formed
    // while those finish (a layer of 608 tokens 12.1 -> 11.7 us, a streaming step 45.9 -> 44.8).
    const bool given = p.pos3 || p.pos_ids;
#pragma unroll 1
    for (int step = 0; step < 2; ++step) {
        if ((step == 0) == given) {
            grid_wait();
#pragma unroll 1
            for (int i = 0; i < kRopeRing - 1; ++i) fetch();
        } else {
            angles(static_cast<int64_t>(blockIdx.x) * p.group, 0);
        }
    }
    int buf = 0, ring = 0;
    for (int64_t tok0 = static_cast<int64_t>(blockIdx.x) * p.group; tok0 < p.n_tokens; tok0 += stride, buf ^= 1) {
        __syncthreads();  // this group's angles are there, and nobody reads the previous group's any more
        angles(tok0 + stride, buf ^ 1);
        const int nt = size_of(tok0), nq = nt * p.Hq, nqk = nq + nt * p.Hkv, total = nt * heads;
#pragma unroll 1
        for (int base = 0; base < total; base += SLOTS) {
            fetch();
            asm volatile("cp.async.wait_group %0;" ::"n"(kRopeRing - 1) : "memory");
            const int u = base + slot;
            if (u < total) {
                const uint4 lo = sm.ring[ring][0][threadIdx.x], hi = sm.ring[ring][1][threadIdx.x];
                uint4 out_lo = lo, out_hi = hi;
                __nv_bfloat16* dst;
                if (u < nqk) {
                    const bool is_q = u < nq;
                    const int t = is_q ? quotient(u, p.div_hq) : quotient(u - nq, p.div_hkv);
                    if (is_q) dst = (tok0 + t < p.split_token ? p.q_out : p.q_out2) + (tok0 * p.Hq + u) * D;
                    else dst = p.k_out + (tok0 * p.Hkv + (u - nq)) * D;
                    const uint32_t lw[4] = {lo.x, lo.y, lo.z, lo.w}, hw[4] = {hi.x, hi.y, hi.z, hi.w};
                    uint32_t ol[4], oh[4], unsure = 0, least = ~0u;
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        unsure |= rotate2(lw[w], hw[w], sm.cs32[buf][t * (HALF / 2) + w * TPV + v], ol[w], oh[w], least);
                    if (__builtin_expect(unsure != 0 || least < 0x007fffffu, 0)) {
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            float ra[2], rb[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const double a = bf16_bits_to_f64((lw[w] >> (16 * e)) & 0xFFFFu);
                                const double b = bf16_bits_to_f64((hw[w] >> (16 * e)) & 0xFFFFu);
                                const double2 cs = sm.cs64[buf][t * HALF + (2 * w + e) * TPV + v];
                                ra[e] = __double2float_rn(__dsub_rn(__dmul_rn(a, cs.x), __dmul_rn(b, cs.y)));
                                rb[e] = __double2float_rn(__dadd_rn(__dmul_rn(b, cs.x), __dmul_rn(a, cs.y)));
                            }
                            ol[w] = pack_bf16x2(ra[0], ra[1]);
                            oh[w] = pack_bf16x2(rb[0], rb[1]);
                        }
                    }
                    out_lo = make_uint4(ol[0], ol[1], ol[2], ol[3]);
                    out_hi = make_uint4(oh[0], oh[1], oh[2], oh[3]);
                } else {
                    dst = p.v_out + (tok0 * p.Hv + (u - nqk)) * D;
                }
                st_stream(dst + i0, out_lo);
                st_stream(dst + i0 + HALF, out_hi);
            }
            ring = ring + 1 == kRopeRing ? 0 : ring + 1;
        }
    }
}

// Tokens of a group.  The call takes as many rounds as the resident CTAs need for its groups; in a round a CTA forms its group's
// angles, kStep tokens at a time, and walks over the group's vectors, kSlots at a time.  Taken is the group for which the rounds come to
// the least of both, counted in vectors (a step of angles, a chain of fp64 operations, is as long as a turn of the slots; with few heads
// a turn counts whole), the larger of two that are alike.  Heads of 64 in the small form take whole steps of tokens or one:
// 1,695 tokens of 8/1 heads, a layer, are 10 % slower with groups of two than with four.
// Layers, us, groups such that every CTA has four (three with few heads) of them, as it was at first / this rule: 28/4 heads of 128, 1,300
// tokens 22.3 / 21.8, 2,500 38.4 / 36.2, 3,500 57.4 / 53.5; 32/8, 3,500 tokens 75.4 / 70.2; 14/2, 4,300 tokens 44.0 / 41.5; 4/2 heads of 64,
// 900 tokens 14.2 / 12.4.  Counting elements instead of turns and steps, and few groups in a last round as less than one, took
// the wrong group in between: 14/2 heads of 64, 1,776 tokens 24.4 / 25.3 so / 22.9, 16/2 heads of 128, 3,700 tokens 37.3 / 38.7 / 36.2,
// 14/2, 7,755 tokens 79.9 / 83.2 / 79.2.  Over 2,176 layers of 300 to 21,000 tokens of 17 forms of heads, every group timed, the rule is
// on average within 0.5 % of the best group, 1.0 % with few heads (the first one 3.8 and 3.5 %); 43 of them are 1.2 to 10 % slower than with the first one.
// Calls that are long enough take the most tokens: no rounds to be won, though not always the best (RoPE alone, 28/4 heads, 10,000
// tokens 33.1 us, 31.1 with groups of three; 14/2 heads, 33,000 tokens 54.7, 52.0 with six).
template <int D, bool FEW>
static int group_size(int64_t n_tokens, int heads) {
    using F = RopeForm<FEW>;
    const int64_t resident = static_cast<int64_t>(kNumSms) * F::kCtasPerSm;
    if (n_tokens >= (FEW ? 3 : 4) * resident * F::kTokens) return F::kTokens;
    constexpr int kSlots = F::kThreads / (D / 16), kStep = F::kThreads / (D / 2);
    constexpr int kMore = FEW && D == 64 ? kStep : 1;
    int best = 0;
    int64_t least = 0;
    for (int g = 1; g <= F::kTokens; g = g < kMore ? kMore : g + kMore) {
        const int64_t rounds = ((n_tokens + g - 1) / g + resident - 1) / resident;
        const int64_t walked = static_cast<int64_t>(heads) * g, vectors = FEW ? (walked + kSlots - 1) / kSlots * kSlots : walked;
        const int64_t cost = rounds * ((g + kStep - 1) / kStep * kSlots + vectors);
        if (best == 0 || cost <= least) {
            best = g;
            least = cost;
        }
    }
    return best;
}

template <int D, bool FEW>
static cudaError_t launch_form(const RopeParams& params, cudaStream_t stream) {
    using F = RopeForm<FEW>;
    RopeParams p = params;
    const int64_t resident = static_cast<int64_t>(kNumSms) * F::kCtasPerSm;
    p.group = group_size<D, FEW>(p.n_tokens, p.Hq + p.Hkv + p.Hv);
    p.div_hq = make_divisor(p.Hq);
    p.div_hkv = make_divisor(p.Hkv);
    p.div_seq = make_divisor(p.seq_len);
    const int64_t groups = (p.n_tokens + p.group - 1) / p.group;
    const unsigned grid = static_cast<unsigned>(groups < resident ? groups : resident);
    return launch_chained<rope_kernel<D, FEW>>(grid, F::kThreads, sizeof(RopeSmem<D, FEW>), stream, p);
}

// Most heads, V's counted, of the form for few.  The small form against the large one, 12.6K / 33K / 74K tokens: heads of 128, 18 of
// them 0.97 / 0.95 / 0.87, 20 0.97 / 0.93 / 0.87, 24 1.04 / 1.06 / 1.02, 28 1.00 / 1.08 / 1.02; heads of 64, 20 of them
// 0.92 / 0.81 / 0.77, 24 0.92 / 1.03 / 1.06, 28 0.99 / 0.94 / 0.87.
constexpr int kFewHeads = 20;

cudaError_t launch_rope(const RopeParams& p, int head_dim, cudaStream_t stream) {
    const int heads = p.Hq + p.Hkv + p.Hv;
    if (p.n_tokens <= 0 || heads == 0) return cudaSuccess;
    if (head_dim == 128) return heads <= kFewHeads ? launch_form<128, true>(p, stream) : launch_form<128, false>(p, stream);
    return heads <= kFewHeads ? launch_form<64, true>(p, stream) : launch_form<64, false>(p, stream);
}

extern "C" int pevlm_rope_group_size(int64_t n_tokens, int heads, int head_dim) {
    if (head_dim == 128) return heads <= kFewHeads ? group_size<128, true>(n_tokens, heads) : group_size<128, false>(n_tokens, heads);
    return heads <= kFewHeads ? group_size<64, true>(n_tokens, heads) : group_size<64, false>(n_tokens, heads);
}

}  // namespace pevlm
