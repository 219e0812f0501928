// The two operations on whole score vectors that need an order: Spearman's rho and the budgeted oracle rule.
//
// Spearman's rho (the rank correlation the paper reports between router scores and the oracle advantage,
// Section 4.2 "Evaluation" and Tables 1-3): ranks with ties sharing the mean of the ranks they span, then the
// Pearson formula over the ranks.  Budgeted oracle (Appendix B, Theorem): escalate the min(budget, #{Delta > 0}) steps
// with the largest positive Delta, equal advantages to the lower index.
//
// Both take at most 65536 values, which is what one cluster of eight CTAs holds on chip: 8192 keys per CTA.  What
// bounds them is latency, a chain of passes with a cluster barrier each, not bytes (8 per value) or arithmetic.
//   - Spearman: one cluster per sample sorts it (least significant digit first, 8 bits per pass, four passes; the
//     scatter of a pass goes straight into the other CTAs' shared memory), finds the runs of equal keys by a scan from
//     either side, and leaves twice the rank of every value; the cluster that finishes second adds up the products.
//     Twice the centred ranks are whole numbers, so the three sums are exact in 64-bit integers.
//   - Budget: radix selection, four histograms of 8 bits from the top digit down give the smallest advantage that
//     still fits the budget and how many of its equals do; a count in index order picks those.
// 20,000 steps: rho 345 us -> 38 us, budgeted rule 240 us -> 14 us, against the same ranks found by counting (every value
// against every other); 300 steps: 18 and 10 us, the passes' latency.  Sorting on a single CTA would quadruple the rounds of every pass; more CTAs than a
// portable cluster would have to meet in global memory.
#include <climits>

#include <cooperative_groups.h>

#include "arb_common.cuh"

namespace arb {

namespace {

namespace cg = cooperative_groups;

constexpr int kCtas = 8;
constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxPer = 8;                        // values per thread: 8 * 1024 * 8 = 65536
constexpr int kMaxPerCta = kThreads * kMaxPer;
constexpr int kDigits = 256;
constexpr int kPasses = 4;

struct SortSmem {
    uint2 val[2][kMaxPerCta];          // (key, index): one store moves both to the CTA they belong to
    uint32_t whist[kWarps][kDigits];   // a warp's count of every digit, then the count in the warps before it
    uint32_t tot[kDigits];             // the CTA's count of every digit
    uint32_t offs[kDigits];            // where the CTA's values with a digit go
    int wmax[kWarps], wmin[kWarps];
    int cta_max, cta_min, last;
    long long sum[3];
};

struct SelectSmem {
    uint32_t hist[kPasses][kDigits];
    uint32_t cnt[kWarps * kMaxPer];
    uint32_t wsum[kWarps];
    uint32_t digit, above, all;
    uint32_t esc, wst;
    double real, gain;
    uint32_t wesc[kWarps], wwst[kWarps];
    double wreal[kWarps], wgain[kWarps];
};

// unsigned keys in the order of the floats; the two zeros are one value
__device__ __forceinline__ uint32_t order_key(float f) {
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}

// The lanes whose digit is this lane's: a vote per bit.  For the low digits of a sort, nearly all distinct in a warp, this
// beats match.any (rho over 20,000: 43 -> 38.7 us); for the top digits of the selection, nearly all alike, match.any
// wins (19.6 -> 14.4 us).
__device__ __forceinline__ uint32_t same_digit(uint32_t d) {
    uint32_t mask = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const uint32_t set = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        mask &= ((d >> b) & 1u) ? set : ~set;
    }
    return mask;
}

// Inclusive sum over the first 256 threads (8 warps), every thread of the block calling; ws: 8 words of shared memory.
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t *ws) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += t;
    }
    if (warp < 8 && lane == 31) ws[warp] = v;
    __syncthreads();
    if (warp < 8)
        for (int w = 0; w < warp; ++w) v += ws[w];
    return v;
}

__device__ __forceinline__ long long block_sum(long long v, long long *scratch) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    long long t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kWarps; ++w) t += scratch[w];
    __syncthreads();
    return t;
}

// values per CTA, a power of two (positions split into CTA and slot by shift and mask), at least one per thread
inline int log_per_cta(int n) {
    int lg = 10;
    while ((kCtas << lg) < n) ++lg;
    return lg;
}

// ranks: [2][65536], twice the rank of every value; done: clusters that have finished, zero between calls
__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kThreads, 1)
spearman_kernel(int n, int lg, const float *__restrict__ x, const float *__restrict__ y, uint32_t *ranks, int *done, double *rho) {
    extern __shared__ __align__(16) char smem[];
    SortSmem &s = *reinterpret_cast<SortSmem *>(smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int me = (int)cluster.block_rank(), sample = blockIdx.x / kCtas;
    const int m = 1 << lg, per = m / kThreads;
    const float *src = sample ? y : x;
    const uint32_t below = (1u << lane) - 1u;

    for (int i = tid; i < m; i += kThreads) {
        const int g = me * m + i;
        s.val[0][i] = make_uint2(g < n ? order_key(src[g]) : 0xffffffffu, (uint32_t)g);   // (padding sorts behind everything)
    }
    __syncthreads();

    // ---- stable sort, least significant digit first; a warp owns per * 32 consecutive slots -------------------------
    for (int pass = 0; pass < kPasses; ++pass) {
        const int cur = pass & 1, shift = 8 * pass;
        for (int d = lane; d < kDigits; d += 32) s.whist[warp][d] = 0;
        __syncwarp();
        uint2 k[kMaxPer];
        uint32_t rank[kMaxPer];
#pragma unroll
        for (int j = 0; j < kMaxPer; ++j) {
            if (j < per) {
                k[j] = s.val[cur][(warp * per + j) * 32 + lane];
                const uint32_t d = (k[j].x >> shift) & (kDigits - 1);
                const uint32_t same = same_digit(d), before = s.whist[warp][d];
                __syncwarp();
                rank[j] = before + __popc(same & below);
                if ((same & below) == 0) s.whist[warp][d] = before + __popc(same);
                __syncwarp();
            }
        }
        __syncthreads();
        if (tid < kDigits) {
            uint32_t c[kWarps], run = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) c[w] = s.whist[w][tid];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                s.whist[w][tid] = run;
                run += c[w];
            }
            s.tot[tid] = run;
        }
        cluster.sync();
        uint32_t before = 0, total = 0;
        if (tid < kDigits) {
#pragma unroll
            for (int c = 0; c < kCtas; ++c) {
                const uint32_t v = *cluster.map_shared_rank(&s.tot[tid], c);
                if (c < me) before += v;
                total += v;
            }
        }
        const uint32_t incl = scan256(total, reinterpret_cast<uint32_t *>(s.wmax));
        if (tid < kDigits) s.offs[tid] = incl - total + before;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kMaxPer; ++j) {
            if (j < per) {
                const uint32_t d = (k[j].x >> shift) & (kDigits - 1);
                const uint32_t pos = s.offs[d] + s.whist[warp][d] + rank[j];
                *cluster.map_shared_rank(&s.val[cur ^ 1][pos & (uint32_t)(m - 1)], (int)(pos >> lg)) = k[j];
            }
        }
        cluster.sync();
    }

    // ---- runs of equal keys: first position by a max-scan of the run starts, last by a min-scan of the run ends ------
    // (a thread has `per` consecutive positions; after four passes the sorted keys are in buffer 0)
    int first[kMaxPer], lastp[kMaxPer];
    int lo = -1, hi = INT_MAX;   // the last run start and the first run end among this thread's positions
    {
        const int slot0 = tid * per;
        uint32_t prev = 0;
        bool have_prev = true;
        if (slot0 > 0) prev = s.val[0][slot0 - 1].x;
        else if (me > 0) prev = *cluster.map_shared_rank(&s.val[0][m - 1].x, me - 1);
        else have_prev = false;
#pragma unroll
        for (int j = 0; j < kMaxPer; ++j) {
            if (j < per) {
                const int slot = slot0 + j, p = me * m + slot;
                const uint32_t k = s.val[0][slot].x;
                uint32_t next = 0;
                bool have_next = true;
                if (slot + 1 < m) next = s.val[0][slot + 1].x;
                else if (me + 1 < kCtas) next = *cluster.map_shared_rank(&s.val[0][0].x, me + 1);
                else have_next = false;
                const bool start = !have_prev || k != prev, end = !have_next || k != next;
                first[j] = start ? p : -1;
                lastp[j] = end ? p : INT_MAX;
                if (start) lo = p;
                if (end && hi == INT_MAX) hi = p;
                prev = k;
                have_prev = true;
            }
        }
    }
    int in_lo = lo, in_hi = hi;   // inclusive scans over the threads below / above
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, in_lo, off), b = __shfl_down_sync(0xffffffffu, in_hi, off);
        if (lane >= off) in_lo = max(in_lo, a);
        if (lane + off < 32) in_hi = min(in_hi, b);
    }
    if (lane == 31) s.wmax[warp] = in_lo;
    if (lane == 0) s.wmin[warp] = in_hi;
    int carry_lo = __shfl_up_sync(0xffffffffu, in_lo, 1), carry_hi = __shfl_down_sync(0xffffffffu, in_hi, 1);
    if (lane == 0) carry_lo = -1;
    if (lane == 31) carry_hi = INT_MAX;
    __syncthreads();
    {   // the warps' results: lane w of every warp looks at warp w
        const int a = s.wmax[lane], b = s.wmin[lane];
        carry_lo = max(carry_lo, __reduce_max_sync(0xffffffffu, lane < warp ? a : -1));
        carry_hi = min(carry_hi, __reduce_min_sync(0xffffffffu, lane > warp ? b : INT_MAX));
        const int all_lo = __reduce_max_sync(0xffffffffu, a), all_hi = __reduce_min_sync(0xffffffffu, b);
        if (tid == 0) { s.cta_max = all_lo; s.cta_min = all_hi; }
    }
    cluster.sync();
    {   // the CTAs' results: lane c looks at CTA c
        const int c = lane & (kCtas - 1);
        const int a = *cluster.map_shared_rank(&s.cta_max, c), b = *cluster.map_shared_rank(&s.cta_min, c);
        carry_lo = max(carry_lo, __reduce_max_sync(0xffffffffu, c < me ? a : -1));
        carry_hi = min(carry_hi, __reduce_min_sync(0xffffffffu, c > me ? b : INT_MAX));
    }
#pragma unroll
    for (int j = 0; j < kMaxPer; ++j)
        if (j < per) { if (first[j] < 0) first[j] = carry_lo; carry_lo = first[j]; }
#pragma unroll
    for (int j = kMaxPer - 1; j >= 0; --j)
        if (j < per) { if (lastp[j] == INT_MAX) lastp[j] = carry_hi; carry_hi = lastp[j]; }
#pragma unroll
    for (int j = 0; j < kMaxPer; ++j) {
        if (j < per) {
            const int id = (int)s.val[0][tid * per + j].y;
            if (id < n) __stcg(ranks + sample * (kCtas * kMaxPerCta) + id, (uint32_t)(first[j] + lastp[j] + 2));
        }
    }

    // ---- the cluster that finishes second takes the sums ------------------------------------------------------------
    __threadfence();
    cluster.sync();
    if (me == 0 && tid == 0) {
        const int last = atomicAdd(done, 1) == 1;
        __threadfence();
        for (int c = 0; c < kCtas; ++c) *cluster.map_shared_rank(&s.last, c) = last;
    }
    cluster.sync();
    if (!s.last) return;   // (uniform over the cluster; nobody reads this CTA's shared memory any more)
    __threadfence();
    long long v[3] = {0, 0, 0};
    for (int i = me * m + tid; i < min((me + 1) * m, n); i += kThreads) {
        const long long a = (long long)__ldcg(ranks + i) - (n + 1), b = (long long)__ldcg(ranks + kCtas * kMaxPerCta + i) - (n + 1);
        v[0] += a * b;
        v[1] += a * a;
        v[2] += b * b;
    }
    long long *scratch = reinterpret_cast<long long *>(s.whist);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const long long t = block_sum(v[q], scratch);
        if (tid == 0) s.sum[q] = t;
    }
    cluster.sync();
    if (me == 0 && tid == 0) {
        long long t[3] = {0, 0, 0};
        for (int c = 0; c < kCtas; ++c)
            for (int q = 0; q < 3; ++q) t[q] += *cluster.map_shared_rank(&s.sum[q], c);
        const double sxx = (double)t[1], syy = (double)t[2];
        *rho = (n < 2 || t[1] == 0 || t[2] == 0) ? __longlong_as_double(0x7ff8000000000000ll) : (double)t[0] / sqrt(sxx * syy);
        *done = 0;
    }
    cluster.sync();
}

__device__ __forceinline__ float sub_ieee(float a, float b) {
    float r;
    asm("sub.rn.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kThreads, 1)
policy_budget_kernel(int n, int lg, const float *__restrict__ s_d, const float *__restrict__ s_t, int budget,
                     uint8_t *__restrict__ decisions, arb_policy_stats *stats) {
    __shared__ SelectSmem s;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, me = (int)cluster.block_rank();
    const int m = 1 << lg, per = m / kThreads, base = me * m;
    const uint32_t below = (1u << lane) - 1u;

    // the bits of a positive float order as the float does, infinity last; 0: not worth a call (a NaN advantage is not)
    uint32_t key[kMaxPer];
#pragma unroll
    for (int j = 0; j < kMaxPer; ++j) {
        key[j] = 0;
        const int i = base + j * kThreads + tid;
        if (j < per && i < n) {
            const uint32_t d = __float_as_uint(sub_ieee(s_t[i], s_d[i]));
            if ((int)d > 0 && d <= 0x7f800000u) key[j] = d;
        }
    }
    for (int i = tid; i < kPasses * kDigits; i += kThreads) (&s.hist[0][0])[i] = 0;
    __syncthreads();

    uint32_t prefix = 0, need = (uint32_t)max(budget, 0);
    bool all = false;
    for (int pass = 0; pass < kPasses; ++pass) {
        const int shift = 24 - 8 * pass;
#pragma unroll
        for (int j = 0; j < kMaxPer; ++j) {
            if (j < per) {
                // (a shift by 32 is not defined: the top digit has no prefix to match)
                const bool in = key[j] != 0 && (pass == 0 || (key[j] >> (shift + 8)) == prefix);
                const uint32_t d = (key[j] >> shift) & (kDigits - 1);
                // one addition per digit and warp: the top digits are nearly all alike
                const uint32_t same = __match_any_sync(0xffffffffu, in ? d : kDigits);
                if (in && (same & below) == 0) atomicAdd(&s.hist[pass][d], (uint32_t)__popc(same));
            }
        }
        cluster.sync();
        uint32_t total = 0;
        const int d = kDigits - 1 - tid;   // from the largest digit down
        if (tid < kDigits)
#pragma unroll
            for (int c = 0; c < kCtas; ++c) total += *cluster.map_shared_rank(&s.hist[pass][d], c);
        const uint32_t upto = scan256(total, s.wsum);   // values with this digit or a larger one
        if (tid == 0) { s.digit = 0; s.above = 0; }
        if (tid == kDigits - 1) s.all = upto;
        __syncthreads();
        if (tid < kDigits && upto >= need && upto - total < need) { s.digit = (uint32_t)d; s.above = upto - total; }
        __syncthreads();
        if (pass == 0 && s.all <= need) { all = true; break; }   // every positive advantage fits (uniform over the cluster)
        prefix = (prefix << 8) | s.digit;
        need -= s.above;
        __syncthreads();
    }
    // the equals of the smallest advantage that fits, in index order: CTA by CTA, round by round, thread by thread
    uint32_t eq_base = 0;
    if (!all) {
        for (int c = 0; c < me; ++c) eq_base += *cluster.map_shared_rank(&s.hist[kPasses - 1][prefix & (kDigits - 1)], c);
    }
    uint32_t ballots[kMaxPer];
#pragma unroll
    for (int j = 0; j < kMaxPer; ++j) {
        ballots[j] = __ballot_sync(0xffffffffu, !all && j < per && key[j] == prefix && key[j] != 0);
        if (lane == 0) s.cnt[j * kWarps + warp] = __popc(ballots[j]);
    }
    __syncthreads();
    const uint32_t mine = tid < kWarps * kMaxPer ? s.cnt[tid] : 0u;
    const uint32_t incl = scan256(mine, s.wsum);
    __syncthreads();
    if (tid < kWarps * kMaxPer) s.cnt[tid] = incl - mine;
    __syncthreads();

    uint32_t esc = 0, wst = 0;
    double real = 0.0, gain = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxPer; ++j) {
        const int i = base + j * kThreads + tid;
        if (j < per && i < n) {
            const bool a = key[j] != 0 && need > 0 &&
                           (all || key[j] > prefix || (key[j] == prefix && eq_base + s.cnt[j * kWarps + warp] + __popc(ballots[j] & below) < need));
            decisions[i] = a ? 1 : 0;
            if (stats != nullptr) {
                const float sd = s_d[i], st = s_t[i];
                esc += a;
                wst += a && !(st > sd);
                real += (double)(a ? st : sd);
                gain += a ? (double)st - (double)sd : 0.0;
            }
        }
    }
    if (stats != nullptr) {
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            esc += __shfl_xor_sync(0xffffffffu, esc, off);
            wst += __shfl_xor_sync(0xffffffffu, wst, off);
            real += __shfl_xor_sync(0xffffffffu, real, off);
            gain += __shfl_xor_sync(0xffffffffu, gain, off);
        }
        if (lane == 0) { s.wesc[warp] = esc; s.wwst[warp] = wst; s.wreal[warp] = real; s.wgain[warp] = gain; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < kWarps; ++w) { esc += s.wesc[w]; wst += s.wwst[w]; real += s.wreal[w]; gain += s.wgain[w]; }
            s.esc = esc; s.wst = wst; s.real = real; s.gain = gain;
        }
    }
    cluster.sync();   // (also: nobody leaves while its histograms may be read)
    if (stats != nullptr && me == 0 && tid == 0) {
        for (int c = 1; c < kCtas; ++c) {
            esc += *cluster.map_shared_rank(&s.esc, c);
            wst += *cluster.map_shared_rank(&s.wst, c);
            real += *cluster.map_shared_rank(&s.real, c);
            gain += *cluster.map_shared_rank(&s.gain, c);
        }
        stats->escalated = esc;
        stats->wasted = wst;
        stats->realised = real;
        stats->gain = gain;
    }
    cluster.sync();
}

}  // namespace

size_t rank_ws_bytes() { return kRankCounterBytes + kPolicyPartBytes + sizeof(uint32_t) * 2 * kCtas * kMaxPerCta; }

arb_status launch_spearman(Ctx *ctx, int n, const float *x, const float *y, double *rho, cudaStream_t stream) {
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device & 63]) {
        if (cudaFuncSetAttribute(spearman_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)) != cudaSuccess)
            return ARB_ERR_CUDA;
        attr_set[ctx->device & 63] = true;
    }
    spearman_kernel<<<2 * kCtas, kThreads, sizeof(SortSmem), stream>>>(
        n, log_per_cta(n), x, y, reinterpret_cast<uint32_t *>(ctx->rank_ws + kRankCounterBytes + kPolicyPartBytes), reinterpret_cast<int *>(ctx->rank_ws), rho);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? ARB_OK : ARB_ERR_CUDA;
}

arb_status launch_policy_budget(Ctx *ctx, int n, const float *s_d, const float *s_t, int budget, uint8_t *decisions,
                                arb_policy_stats *stats, cudaStream_t stream) {
    policy_budget_kernel<<<kCtas, kThreads, 0, stream>>>(n, log_per_cta(n), s_d, s_t, budget, decisions, stats);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? ARB_OK : ARB_ERR_CUDA;
}

}  // namespace arb
