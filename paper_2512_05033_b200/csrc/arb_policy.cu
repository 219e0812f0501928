// Escalation policies on PRM scores, and C-way router heads.
//
// Policies (decision 1 = escalate the step to the target, 0 = keep the draft step):
//   RSD baseline (Section 3.1 of the paper): the step is accepted iff s_d > tau, so escalated iff s_d <= tau.
//   Oracle threshold (Section 4.1): escalate iff Delta = s_t - s_d > tau.
//   Oracle arg max (Section 4.1): keep the higher-scoring step; escalate iff s_t > s_d.
//   Budgeted oracle (Appendix B, Theorem): needs an order over the steps, see arb_rank.cu.
// Each kernel also accumulates the escalation count, the wasted escalations of Section 3.2 (escalated
// although s_t <= s_d), the realised score sum_i (a_i ? s_t : s_d) and the gain sum_i a_i (s_t - s_d).
// Delta is one fp32 subtraction, not flushed to zero for subnormal results, so that the decision is
// the one an IEEE fp32 subtraction gives.
//
// C-way heads (Section 6.1, ablation): one warp per step computes the C logits (softmax head) or one
// logit against C - 1 ordered cut points (ordinal head), the class probabilities, the expected class
// level scaled to [0, 1] as the routing score, and the threshold decision (a tie accepts).
#include "arb_common.cuh"

namespace arb {

namespace {

constexpr int kPolicyThreads = 256;
constexpr int kPolicyMaxCtas = 256;

__device__ __forceinline__ float sub_ieee(float a, float b) {
    float r;
    asm("sub.rn.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// block-wide sums of the four statistics, in thread 0
__device__ __forceinline__ void block_stats(arb_policy_stats &v) {
    __shared__ arb_policy_stats part[kPolicyThreads / 32];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        v.escalated += __shfl_xor_sync(0xffffffffu, v.escalated, off);
        v.wasted += __shfl_xor_sync(0xffffffffu, v.wasted, off);
        v.realised += __shfl_xor_sync(0xffffffffu, v.realised, off);
        v.gain += __shfl_xor_sync(0xffffffffu, v.gain, off);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kPolicyThreads / 32; ++w) {
            v.escalated += part[w].escalated;
            v.wasted += part[w].wasted;
            v.realised += part[w].realised;
            v.gain += part[w].gain;
        }
    }
}

// One launch, statistics included: every CTA leaves its sums, the last to finish adds them up in CTA order (so the
// same scores give the same bits).  Launch-bound at the sizes of a split; with the statistics zeroed by a copy engine
// and added by fp64 atomics it was two stream operations, and the sums came out in any order.
__global__ void __launch_bounds__(kPolicyThreads)
policy_kernel(int kind, int n, const float *__restrict__ s_d, const float *__restrict__ s_t, float tau,
              uint8_t *__restrict__ decisions, arb_policy_stats *stats, arb_policy_stats *part, int *done) {
    __shared__ int last;
    arb_policy_stats v = {0u, 0u, 0.0, 0.0};
    for (int i = blockIdx.x * kPolicyThreads + threadIdx.x; i < n; i += (int)gridDim.x * kPolicyThreads) {
        const float sd = s_d[i];
        const float st = s_t != nullptr ? s_t[i] : sd;
        bool a;
        if (kind == ARB_POLICY_RSD) a = !(sd > tau);
        else if (kind == ARB_POLICY_ORACLE_THRESHOLD) a = sub_ieee(st, sd) > tau;
        else a = st > sd;
        decisions[i] = a ? 1 : 0;
        v.escalated += a;
        v.wasted += a && !(st > sd);
        v.realised += (double)(a ? st : sd);
        v.gain += a ? (double)st - (double)sd : 0.0;
    }
    if (stats == nullptr) return;
    block_stats(v);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = v;
        __threadfence();
        last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    v = {0u, 0u, 0.0, 0.0};
    if (threadIdx.x < gridDim.x) {   // kPolicyMaxCtas == kPolicyThreads: at most one record per thread
        const arb_policy_stats *p = part + threadIdx.x;
        v.escalated = __ldcg(&p->escalated);
        v.wasted = __ldcg(&p->wasted);
        v.realised = __ldcg(&p->realised);
        v.gain = __ldcg(&p->gain);
    }
    block_stats(v);
    if (threadIdx.x == 0) {
        *stats = v;
        *done = 0;
    }
}
static_assert(kPolicyMaxCtas <= kPolicyThreads, "one record per thread of the last CTA");
static_assert(kPolicyMaxCtas * sizeof(arb_policy_stats) <= kPolicyPartBytes, "the records of a call");

constexpr int kHeadWarps = 4;

struct HeadArgs {
    const char *hidden;
    const char *w;
    float b[ARB_MAX_CLASSES];
    int n_steps, hidden_dim, n_classes, mode;
    float tau;
    float *probs, *scores;
    uint8_t *decisions;
};

template <typename T>
__global__ void __launch_bounds__(kHeadWarps * 32)
route_classes_kernel(const HeadArgs a) {
    constexpr int EPL = Elt<T>::kPerVec;
    // one CTA per step: its warps share the row (a single warp per step would walk the row in 14 dependent
    // round trips at the router's hidden size), partial sums meet in shared memory
    __shared__ float part[kHeadWarps][ARB_MAX_CLASSES];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int step = blockIdx.x;
    const int C = a.n_classes;
    const int nlog = a.mode == ARB_HEAD_SOFTMAX ? C : 1;   // dot products to take
    const int nvec = a.hidden_dim / EPL;
    const uint4 *hrow = reinterpret_cast<const uint4 *>(a.hidden + (size_t)step * a.hidden_dim * sizeof(T));
    float acc[ARB_MAX_CLASSES];
#pragma unroll
    for (int c = 0; c < ARB_MAX_CLASSES; ++c) acc[c] = 0.f;
    for (int v = threadIdx.x; v < nvec; v += kHeadWarps * 32) {
        float hf[EPL];
        Elt<T>::unpack(__ldg(hrow + v), hf);
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c) {
            if (c < nlog) {
                float wf[EPL];
                Elt<T>::unpack(__ldg(reinterpret_cast<const uint4 *>(a.w + (size_t)c * a.hidden_dim * sizeof(T)) + v), wf);
#pragma unroll
                for (int e = 0; e < EPL; ++e) acc[c] = fmaf(hf[e], wf[e], acc[c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < ARB_MAX_CLASSES; ++c) {
        if (c < nlog) {
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], off);
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c)
            if (c < nlog) part[warp][c] = acc[c];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int c = 0; c < ARB_MAX_CLASSES; ++c) {
        if (c < nlog) {
            float t = part[0][c];
            for (int w2 = 1; w2 < kHeadWarps; ++w2) t += part[w2][c];
            acc[c] = t;
        }
    }
    float p[ARB_MAX_CLASSES];
    if (a.mode == ARB_HEAD_SOFTMAX) {
        float mx = -INFINITY, z = 0.f;
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c)
            if (c < C) { acc[c] += a.b[c]; mx = fmaxf(mx, acc[c]); }
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c)
            if (c < C) { p[c] = expf(acc[c] - mx); z += p[c]; }
        const float inv = 1.0f / z;
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c)
            if (c < C) p[c] *= inv;
    } else {
        const float z = acc[0] + a.b[0];
        float ge_prev = 1.0f;   // P(y >= 0)
#pragma unroll
        for (int c = 0; c < ARB_MAX_CLASSES; ++c) {
            if (c < C) {
                const float ge_next = c + 1 < C ? 1.0f / (1.0f + expf(-(z - a.b[c + 1]))) : 0.f;   // P(y >= c + 1)
                p[c] = ge_prev - ge_next;
                ge_prev = ge_next;
            }
        }
    }
    float score = 0.f;
    const float step_level = 1.0f / (float)(C - 1);
#pragma unroll
    for (int c = 0; c < ARB_MAX_CLASSES; ++c) {
        if (c < C) {
            score = fmaf(p[c], (float)c * step_level, score);
            if (a.probs != nullptr) a.probs[(size_t)step * C + c] = p[c];
        }
    }
    a.scores[step] = score;
    a.decisions[step] = score > a.tau ? 1 : 0;   // a tie accepts the draft step
}

}  // namespace

arb_status launch_policy(Ctx *ctx, int kind, int n_steps, const float *s_d, const float *s_t, float tau, int budget,
                         uint8_t *decisions, arb_policy_stats *stats, cudaStream_t stream) {
    if (kind == ARB_POLICY_ORACLE_BUDGET) return launch_policy_budget(ctx, n_steps, s_d, s_t, budget, decisions, stats, stream);
    const int need = (n_steps + kPolicyThreads - 1) / kPolicyThreads;
    const int grid = need < kPolicyMaxCtas ? need : kPolicyMaxCtas;
    policy_kernel<<<grid, kPolicyThreads, 0, stream>>>(kind, n_steps, s_d, s_t, tau, decisions, stats,
                                                       reinterpret_cast<arb_policy_stats *>(ctx->rank_ws + kRankCounterBytes),
                                                       reinterpret_cast<int *>(ctx->rank_ws) + 1);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? ARB_OK : ARB_ERR_CUDA;
}

arb_status launch_route_classes(Ctx *ctx, int dtype, int mode, int n_steps, int hidden_dim, int n_classes,
                                const void *hidden, const void *w, const float *b_host, float tau, float *probs,
                                float *scores, uint8_t *decisions, cudaStream_t stream) {
    HeadArgs a;
    a.hidden = static_cast<const char *>(hidden);
    a.w = static_cast<const char *>(w);
    for (int c = 0; c < ARB_MAX_CLASSES; ++c) a.b[c] = c < n_classes ? b_host[c] : 0.f;
    a.n_steps = n_steps;
    a.hidden_dim = hidden_dim;
    a.n_classes = n_classes;
    a.mode = mode;
    a.tau = tau;
    a.probs = probs;
    a.scores = scores;
    a.decisions = decisions;
    const int grid = n_steps;
    if (dtype == ARB_BF16)
        route_classes_kernel<__nv_bfloat16><<<grid, kHeadWarps * 32, 0, stream>>>(a);
    else if (dtype == ARB_F32)
        route_classes_kernel<float><<<grid, kHeadWarps * 32, 0, stream>>>(a);
    else
        return ARB_ERR_UNSUPPORTED;
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? ARB_OK : ARB_ERR_CUDA;
}

}  // namespace arb
