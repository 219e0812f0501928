// Step-chunk attention over an fp32 cache (whose 1e-5 tolerance rules out tf32), on the CUDA cores.
//
// A chunk of n query tokens against one KV head is rows = n * group query rows (token-major) over the same keys.  A CTA of
// eight warps takes a tile of 64, 32 or 16 rows (see launch_one) and walks keys in tiles of 32 (two pages, double-buffered with
// cp.async): every key that reaches shared memory is used by all rows of the tile.  A warp owns an eighth of the rows, so the online
// softmax needs no barrier.  Per key tile and lane, of 64 rows: S as 2 rows x 4 keys (32 FMA per 6 conflict-free 16-byte loads per
// 4 dimensions), of 32 as 1 x 4, of 16 as 1 x 2; P through the warp's own corner of shared memory; O += P V as 8, 4 or 2 rows x 4
// dimensions (half the rows at head_dim 64).
// What bounds it is shared-memory loads and FMA issue on large calls, latency on small ones, so the flat list of (sequence, kv head, row tile,
// key tile) units is cut evenly over two CTAs per SM; a row tile that is cut leaves partials, and the CTA that arrives last
// at the tile's counter merges them.  A CTA per (query row, kv head), which this replaces, re-read the keys for every
// row and ran 528 keys as one chain: a 16-token step over 528 keys (8 / 2 heads of 64) 41.6 -> 17.3 us (in row tiles of 16 and with
// the loads of a merge in flight together 13.1 us), two steps of 56 and
// 104 tokens over 1.3k and 1.8k keys (8 / 2 heads of 128) 291 -> 61 us (a quarter of the FMA rate: the shared-memory
// loads of the first product are the bound there).
#include "arb_common.cuh"

namespace arb {

namespace {

constexpr int kKeys = 32;               // keys of a tile
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMinUnits = 2;            // fewest key tiles worth giving a CTA
constexpr int kCtasPerSm = 2;

// The kernel's template parameter R is the number of query rows of a tile: 64, 32 or 16, a warp owning R / 8 of them.
template <int D, int R>
struct Smem {
    static constexpr int kPitch = D + 4;    // neighbouring rows start 4 banks apart
    float q[R][kPitch];
    float k[2][kKeys][kPitch];
    float v[2][kKeys][kPitch];
    float p[kWarps][kKeys][R / kWarps];
    float row[kWarps][R / kWarps];           // a warp's rescale factors, then 1 / sum
    int last;
};

template <int D, int R>
__host__ __device__ constexpr size_t slot_floats() { return (size_t)R * D + 2 * R; }   // O [R][D], max [R], sum [R]

struct F32Args {
    const float *q, *k_pages, *v_pages;
    const int32_t *block_table, *seq_lens, *q_lens;
    float *out;
    uint32_t *status;
    float *partials;
    int *counters;      // arrivals per (sequence, kv head, row tile), zero between calls
    int slots, max_items;
    int batch, Hq, Hkv, num_pages, max_pages, rows;
    float scale_log2;
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool real) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(real ? 16 : 0) : "memory");
}

// Tokens of a sequence that q and out have rows for: all of them, unless the q_lens on the device add up to more than the
// caller's total_q.
__device__ __forceinline__ int rows_there(const F32Args &a, int qrow0, int n) { return qrow0 < 0 ? 0 : max(0, min(n, a.rows - qrow0)); }

// One row tile over the key tiles [t0, t1); nparts > 1: leaves partial `slot` and merges if it is the last to arrive.
template <int D, int G, int kRows>
__device__ void row_tile(const F32Args &a, Smem<D, kRows> &s, int b, int kvh, int rt, int t0, int t1, int qrow0, int nparts,
                         long long slot, long long slot_first, int item) {
    constexpr int kVecs = D / 4;
    constexpr int kWarpRows = kRows / kWarps;
    constexpr int kLaneRows = D == 128 ? kWarpRows : kWarpRows / 2;   // rows of O a lane holds, 4 dimensions each
    constexpr int kRowLanes = kWarpRows < 4 ? 16 : 8;                 // S: lanes of a row,
    constexpr int kSRows = kWarpRows < 4 ? 1 : kWarpRows / 4;         // a lane's rows, 32 / kRowLanes apart,
    constexpr int kSKeys = kKeys / kRowLanes;                         // and its keys, kRowLanes apart
    constexpr int kRowStep = 32 / kRowLanes;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = a.q_lens[b], L = a.seq_lens[b], rows = n * G, r_begin = rt * kRows;
    const int there = rows_there(a, qrow0, n) * G;   // rows that q and out have
    const int kv_len = L - n + (min(r_begin + kRows, rows) - 1) / G + 1;   // keys the tile's last row sees
    t1 = min(t1, (kv_len + kKeys - 1) / kKeys);
    auto row_of = [&](int i) -> size_t {   // first element of row i of the tile in q and out
        const int r = r_begin + i, tok = r / G;
        return ((size_t)(qrow0 + tok) * a.Hq + kvh * G + (r - tok * G)) * D;
    };
    auto limit_of = [&](int i) { return L - n + min(r_begin + i, rows - 1) / G + 1; };   // keys row i sees

    // Keys past the last visible one are zero-filled, not read: stale slots must not reach a product.
    auto load_tile = [&](int t, int st) {
#pragma unroll
        for (int i = 0; i < kKeys * kVecs / kThreads; ++i) {
            const int idx = i * kThreads + tid, r = idx / kVecs, c = idx - r * kVecs, key = t * kKeys + r;
            const bool real = key < kv_len;
            int pid = real ? __ldg(a.block_table + (size_t)b * a.max_pages + key / kPage) : 0;
            if ((unsigned)pid >= (unsigned)a.num_pages) {
                atomicOr(a.status, (uint32_t)ARB_DEV_BAD_PAGE);
                pid = 0;
            }
            const size_t at = (((size_t)pid * a.Hkv + kvh) * kPage + key % kPage) * D + c * 4;
            cp_async16(&s.k[st][r][c * 4], a.k_pages + at, real);
            cp_async16(&s.v[st][r][c * 4], a.v_pages + at, real);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    const int rg = lane / kRowLanes, kg = lane % kRowLanes;
    const int orow = D == 128 ? 0 : (lane >> 4) * kLaneRows;      // O: first row ...
    const int odim = (D == 128 ? lane : (lane & 15)) * 4;         // ... and first dimension of this lane
    const bool warp_ok = r_begin + warp * kWarpRows < rows;
    int lim[kSRows];
#pragma unroll
    for (int i = 0; i < kSRows; ++i) lim[i] = limit_of(warp * kWarpRows + rg + kRowStep * i);
    const int lim_min = limit_of(warp * kWarpRows);
    float m[kSRows], l[kSRows];
#pragma unroll
    for (int i = 0; i < kSRows; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
    float o[kLaneRows][4];
#pragma unroll
    for (int r = 0; r < kLaneRows; ++r) { o[r][0] = o[r][1] = o[r][2] = o[r][3] = 0.f; }

    __syncthreads();   // the tile before this one is done with shared memory
    if (t0 < t1) load_tile(t0, 0);   // (the keys' way is the longer one: table, then rows)
#pragma unroll
    for (int i = tid; i < kRows * kVecs; i += kThreads) {
        const int r = i / kVecs, c = i - r * kVecs;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r_begin + r < there) {
            x = __ldg(reinterpret_cast<const float4 *>(a.q + row_of(r)) + c);
            x.x *= a.scale_log2; x.y *= a.scale_log2; x.z *= a.scale_log2; x.w *= a.scale_log2;
        }
        *reinterpret_cast<float4 *>(&s.q[r][c * 4]) = x;
    }
    for (int t = t0; t < t1; ++t) {
        const int st = (t - t0) & 1;
        if (t + 1 < t1) {
            load_tile(t + 1, st ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        if (warp_ok) {
            float sc[kSRows][kSKeys] = {};
#pragma unroll 4
            for (int c = 0; c < D; c += 4) {
                float4 x[kSRows];
#pragma unroll
                for (int i = 0; i < kSRows; ++i) x[i] = *reinterpret_cast<const float4 *>(&s.q[warp * kWarpRows + rg + kRowStep * i][c]);
#pragma unroll
                for (int j = 0; j < kSKeys; ++j) {
                    const float4 kv = *reinterpret_cast<const float4 *>(&s.k[st][kg + kRowLanes * j][c]);
#pragma unroll
                    for (int i = 0; i < kSRows; ++i)
                        sc[i][j] = fmaf(x[i].x, kv.x, fmaf(x[i].y, kv.y, fmaf(x[i].z, kv.z, fmaf(x[i].w, kv.w, sc[i][j]))));
                }
            }
#pragma unroll
            for (int i = 0; i < kSRows; ++i) {
                float mx = -INFINITY;
#pragma unroll
                for (int j = 0; j < kSKeys; ++j) {
                    if (t * kKeys + kg + kRowLanes * j >= lim[i]) sc[i][j] = -INFINITY;
                    mx = fmaxf(mx, sc[i][j]);
                }
#pragma unroll
                for (int off = 1; off < kRowLanes; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                const float mn = fmaxf(m[i], mx), base = mn == -INFINITY ? 0.f : mn;   // (a part may hold no key of a row)
                const float f = fast_exp2(m[i] - base);
                m[i] = mn;
                l[i] *= f;
#pragma unroll
                for (int j = 0; j < kSKeys; ++j) {
                    const float p = fast_exp2(sc[i][j] - base);
                    l[i] += p;
                    s.p[warp][kg + kRowLanes * j][rg + kRowStep * i] = p;
                }
                if (kg == 0) s.row[warp][rg + kRowStep * i] = f;
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kLaneRows; ++r) {
                const float f = s.row[warp][orow + r];
                o[r][0] *= f; o[r][1] *= f; o[r][2] *= f; o[r][3] *= f;
            }
            if (t * kKeys + kKeys <= lim_min) {
#pragma unroll 4
                for (int key = 0; key < kKeys; ++key) {
                    const float4 v = *reinterpret_cast<const float4 *>(&s.v[st][key][odim]);
                    float p[kLaneRows];
#pragma unroll
                    for (int r = 0; r < kLaneRows; r += 4) {
                        const float *from = &s.p[warp][key][orow + r];
                        if constexpr (kLaneRows >= 4) {
                            const float4 x = *reinterpret_cast<const float4 *>(from);
                            p[r] = x.x; p[r + 1] = x.y; p[r + 2] = x.z; p[r + 3] = x.w;
                        } else if constexpr (kLaneRows == 2) {
                            const float2 x = *reinterpret_cast<const float2 *>(from);
                            p[0] = x.x; p[1] = x.y;
                        } else {
                            p[0] = *from;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < kLaneRows; ++r) {
                        o[r][0] = fmaf(p[r], v.x, o[r][0]); o[r][1] = fmaf(p[r], v.y, o[r][1]);
                        o[r][2] = fmaf(p[r], v.z, o[r][2]); o[r][3] = fmaf(p[r], v.w, o[r][3]);
                    }
                }
            } else {   // the causal edge: a value a row does not see is not used, not even times zero
                for (int key = 0; key < kKeys; ++key) {
                    const float4 v = *reinterpret_cast<const float4 *>(&s.v[st][key][odim]);
#pragma unroll
                    for (int r = 0; r < kLaneRows; ++r) {
                        if (t * kKeys + key < limit_of(warp * kWarpRows + orow + r)) {
                            const float p = s.p[warp][key][orow + r];
                            o[r][0] = fmaf(p, v.x, o[r][0]); o[r][1] = fmaf(p, v.y, o[r][1]);
                            o[r][2] = fmaf(p, v.z, o[r][2]); o[r][3] = fmaf(p, v.w, o[r][3]);
                        }
                    }
                }
            }
        }
        __syncthreads();   // the stage is free
    }

#pragma unroll
    for (int i = 0; i < kSRows; ++i) {
#pragma unroll
        for (int off = 1; off < kRowLanes; off <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
    }
    if (nparts == 1) {
        if (kg == 0) {
#pragma unroll
            for (int i = 0; i < kSRows; ++i) s.row[warp][rg + kRowStep * i] = 1.0f / l[i];
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < kLaneRows; ++r) {
            const int i = warp * kWarpRows + orow + r;
            if (r_begin + i < there && ARB_IN_RANGE(a.status, qrow0 + (r_begin + i) / G, a.rows)) {
                const float inv = s.row[warp][orow + r];
                *reinterpret_cast<float4 *>(a.out + row_of(i) + odim) =
                    make_float4(o[r][0] * inv, o[r][1] * inv, o[r][2] * inv, o[r][3] * inv);
            }
        }
        return;
    }
    float *po = a.partials + (size_t)slot * slot_floats<D, kRows>();
    if (ARB_IN_RANGE(a.status, slot, a.slots)) {
#pragma unroll
        for (int r = 0; r < kLaneRows; ++r)
            *reinterpret_cast<float4 *>(po + (warp * kWarpRows + orow + r) * D + odim) = make_float4(o[r][0], o[r][1], o[r][2], o[r][3]);
        if (kg == 0) {
#pragma unroll
            for (int i = 0; i < kSRows; ++i) {
                po[kRows * D + warp * kWarpRows + rg + kRowStep * i] = m[i];
                po[kRows * D + kRows + warp * kWarpRows + rg + kRowStep * i] = l[i];
            }
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        s.last = atomicAdd(&a.counters[item], 1) == nparts - 1;
        if (s.last) a.counters[item] = 0;   // everyone has arrived: ready for the next call
        __threadfence();
    }
    __syncthreads();
    if (!s.last) return;
    // m = max_p m_p, w_p = 2^(m_p - m), out = sum_p w_p o_p / sum_p w_p l_p; part 0 sees key 0: m is finite
    const float *p0 = a.partials + (size_t)slot_first * slot_floats<D, kRows>();
    constexpr int kRowThreads = kThreads / kRows, kPieces = kVecs / kRowThreads;   // threads of a row, and what each of them merges
    constexpr int kAtOnce = kPieces > 2 ? 4 : kPieces > 1 ? 8 : 16;   // parts whose loads are in flight together
    const int i = tid / kRowThreads, c0 = tid % kRowThreads;
    if (r_begin + i >= there || !ARB_IN_RANGE(a.status, qrow0 + (r_begin + i) / G, a.rows)) return;
    float M = -INFINITY, sum = 0.f;
    float4 acc[kPieces];
#pragma unroll
    for (int c = 0; c < kPieces; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p = 0; p < nparts; p += kAtOnce) {
        float pm[kAtOnce], pl[kAtOnce];
        float4 x[kAtOnce][kPieces];
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
            const float *pp = p0 + (size_t)(p + j) * slot_floats<D, kRows>();
            const bool in = p + j < nparts;
            pm[j] = in ? __ldcg(pp + kRows * D + i) : -INFINITY;
            pl[j] = in ? __ldcg(pp + kRows * D + kRows + i) : 0.f;
#pragma unroll
            for (int c = 0; c < kPieces; ++c)
                x[j][c] = in ? __ldcg(reinterpret_cast<const float4 *>(pp + i * D) + c0 + kRowThreads * c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float mx = M;
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) mx = fmaxf(mx, pm[j]);
        const float base = mx == -INFINITY ? 0.f : mx, f = fast_exp2(M - base);   // (the first parts may hold no key of the row)
        M = mx;
        sum *= f;
#pragma unroll
        for (int c = 0; c < kPieces; ++c) { acc[c].x *= f; acc[c].y *= f; acc[c].z *= f; acc[c].w *= f; }
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
            const float w = fast_exp2(pm[j] - base);
            sum = fmaf(w, pl[j], sum);
#pragma unroll
            for (int c = 0; c < kPieces; ++c) {
                acc[c].x = fmaf(w, x[j][c].x, acc[c].x); acc[c].y = fmaf(w, x[j][c].y, acc[c].y);
                acc[c].z = fmaf(w, x[j][c].z, acc[c].z); acc[c].w = fmaf(w, x[j][c].w, acc[c].w);
            }
        }
    }
    const float inv = 1.0f / sum;
#pragma unroll
    for (int c = 0; c < kPieces; ++c)
        reinterpret_cast<float4 *>(a.out + row_of(i))[c0 + kRowThreads * c] = make_float4(acc[c].x * inv, acc[c].y * inv, acc[c].z * inv, acc[c].w * inv);
}

template <int D, int G, int kRows>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
chunk_f32_kernel(const F32Args a) {
    extern __shared__ __align__(16) char smem[];
    using Shared = Smem<D, kRows>;
    Shared &s = *reinterpret_cast<Shared *>(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, B = a.batch, Hkv = a.Hkv;
    long long *units = reinterpret_cast<long long *>(smem + ((sizeof(Shared) + 15) & ~size_t(15)));   // [B + 1] key tiles before b
    int *items = reinterpret_cast<int *>(units + B + 1);   // [B + 1] row tiles before b (times kv heads)
    int *row0 = items + B + 1;                             // [B + 1] rows of q before b
    pdl_enter();
    auto shape = [&](int b, int &rts, int &kts) {   // row tiles and key tiles of a sequence this kernel serves
        const int n = a.q_lens[b], L = a.seq_lens[b];
        const bool ok = n >= 2 && n <= a.rows && L >= n && L <= a.max_pages * kPage;
        rts = ok ? (n * G + kRows - 1) / kRows : 0;
        kts = ok ? (L + kKeys - 1) / kKeys : 0;
        return n >= 2 && !ok;
    };
    if (tid == 0) { units[0] = 0; items[0] = 0; row0[0] = 0; }
    if (warp == 0) {
        long long cu = 0;
        int ci = 0, cr = 0;
        for (int b0 = 0; b0 < B; b0 += 32) {
            const int b = b0 + lane;
            int rts = 0, kts = 0, vr = 0;
            if (b < B) { shape(b, rts, kts); vr = max(a.q_lens[b], 0); }
            long long vu = (long long)Hkv * rts * kts;
            int vi = Hkv * rts;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const long long tu = __shfl_up_sync(0xffffffffu, vu, off);
                const int ti = __shfl_up_sync(0xffffffffu, vi, off), tr = __shfl_up_sync(0xffffffffu, vr, off);
                if (lane >= off) { vu += tu; vi += ti; vr += tr; }
            }
            if (b < B) { units[b + 1] = vu + cu; items[b + 1] = vi + ci; row0[b + 1] = vr + cr; }
            cu += __shfl_sync(0xffffffffu, vu, 31);
            ci += __shfl_sync(0xffffffffu, vi, 31);
            cr += __shfl_sync(0xffffffffu, vr, 31);
        }
    }
    __syncthreads();
    // chunk sequences whose lengths are invalid: status bit, rows of zeros
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        int rts, kts;
        if (!shape(b, rts, kts)) continue;
        if (tid == 0) atomicOr(a.status, (uint32_t)ARB_DEV_BAD_SEQ_LEN);
        for (size_t i = tid; i < (size_t)rows_there(a, row0[b], row0[b + 1] - row0[b]) * a.Hq * D; i += kThreads) a.out[(size_t)row0[b] * a.Hq * D + i] = 0.f;
    }
    const long long total = units[B];
    if (total == 0) return;
    const int grid = gridDim.x, n_items = items[B];
    // without room for partials or counters every row tile stays whole
    const bool whole = n_items > a.max_items || n_items + grid > a.slots;
    const long long chunk = max((long long)kMinUnits, (total + grid - 1) / grid);
    long long cur = whole ? blockIdx.x : blockIdx.x * chunk;
    const long long end = whole ? n_items : min(cur + chunk, total);
    while (cur < end) {
        int lo = 0, hi = B;   // the last sequence that starts at or before cur
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((whole ? (long long)items[mid] : units[mid]) <= cur) lo = mid; else hi = mid;
        }
        int rts, kts;
        shape(lo, rts, kts);
        const long long rel = cur - (whole ? (long long)items[lo] : units[lo]);
        const int in_seq = whole ? (int)rel : (int)(rel / kts), item = items[lo] + in_seq;
        const int t0 = whole ? 0 : (int)(rel - (long long)in_seq * kts);
        const int t1 = whole ? kts : (int)min((long long)kts, t0 + (end - cur));
        const long long first = units[lo] + (long long)in_seq * kts;   // the row tile's place in the list
        const int c_first = (int)(first / chunk), nparts = whole ? 1 : (int)((first + kts - 1) / chunk) - c_first + 1;
        row_tile<D, G, kRows>(a, s, lo, in_seq / rts, in_seq % rts, t0, t1, row0[lo], nparts, (long long)item + blockIdx.x,
                       (long long)item + c_first, item);
        cur += whole ? grid : t1 - t0;
    }
}

template <int D, int G, int R>
arb_status launch_rows(Ctx *ctx, F32Args a, cudaStream_t stream) {
    using Shared = Smem<D, R>;
    auto bytes = [](int batch) {
        return ((sizeof(Shared) + 15) & ~size_t(15)) + (sizeof(long long) + 2 * sizeof(int)) * ((size_t)batch + 1);
    };
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device & 63]) {
        if (cudaFuncSetAttribute(chunk_f32_kernel<D, G, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kMaxBatch)) != cudaSuccess)
            return ARB_ERR_CUDA;
        attr_set[ctx->device & 63] = true;
    }
    a.slots = (int)(ctx->chunk_ws_bytes / (slot_floats<D, R>() * sizeof(float)));
    const cudaError_t err = launch_pdl(chunk_f32_kernel<D, G, R>, dim3(kCtasPerSm * ctx->num_sms), dim3(kThreads), bytes(a.batch), stream, a);
    ctx->launches++;
    return err == cudaSuccess ? ARB_OK : ARB_ERR_CUDA;
}

// Rows of a tile: 64, or 32 or 16 where the call is so small that the CTAs cannot all have work with more.  Smaller tiles read
// the keys more often and take less time each, and so does the merge of their parts.  The host knows the rows and the most keys
// that the table can hold, not the lengths: a short sequence under a wide table keeps 64 rows.  us per call with tiles of
// 16 / 32 / 64 rows, one sequence, 8 / 2 heads of 64 (of 128), the table as long as the sequence, by `most`:
//   16 tokens over  528 keys,  68:  13.2 / 15.9 / 17.6  (18.0 / 23.6 / 25.5)
//   16 tokens over 1100 keys, 140:  12.8 / 17.6 / 21.2  (17.5 / 25.2 / 36.7)
//   64 tokens over  528 keys, 170:  13.4 / 15.7 / 18.7  (18.6 / 23.7 / 31.9)
//   16 tokens over 2300 keys, 288:  14.4 / 18.1 / 23.7  (19.5 / 28.1 / 44.4)
//   64 tokens over 1100 keys, 350:  18.7 / 18.3 / 21.7  (26.5 / 27.6 / 41.0)
//   64 tokens over 4600 keys, 1440: 55.2 / 42.0 / 37.2  (81.1 / 70.0 / 77.5)
// and two sequences of 64 tokens over 300 keys, 200: 18.1 / 16.5 / 20.5 (24.4 / 24.5 / 32.4).  At the first line (room / 4 = 148) 16 rows
// win by a quarter, at the second (296) 32 do against 64.  Both lie low: they were drawn where a CTA's share falls below kMinUnits,
// and tiles of the next smaller height still win somewhat above them, the less the more row tiles the call has.
template <int D, int G>
arb_status launch_one(Ctx *ctx, const F32Args &a, cudaStream_t stream) {
    const long long most = (long long)a.Hkv * ((long long)a.rows * G / 64 + a.batch) * ((a.max_pages * (long long)kPage + kKeys - 1) / kKeys);
    const long long room = (long long)kMinUnits * kCtasPerSm * ctx->num_sms;
    if (4 * most <= room) return launch_rows<D, G, 16>(ctx, a, stream);
    if (2 * most <= room) return launch_rows<D, G, 32>(ctx, a, stream);
    return launch_rows<D, G, 64>(ctx, a, stream);
}

template <int D>
arb_status launch_g(Ctx *ctx, int g, const F32Args &a, cudaStream_t stream) {
    switch (g) {
        case 1: return launch_one<D, 1>(ctx, a, stream);
        case 2: return launch_one<D, 2>(ctx, a, stream);
        case 3: return launch_one<D, 3>(ctx, a, stream);
        case 4: return launch_one<D, 4>(ctx, a, stream);
        case 5: return launch_one<D, 5>(ctx, a, stream);
        case 6: return launch_one<D, 6>(ctx, a, stream);
        case 7: return launch_one<D, 7>(ctx, a, stream);
        case 8: return launch_one<D, 8>(ctx, a, stream);
        default: return ARB_ERR_UNSUPPORTED;
    }
}

}  // namespace

arb_status launch_chunk_f32(Ctx *ctx, const arb_attn_params &p, const void *q, const void *k_pages, const void *v_pages,
                            const int32_t *block_table, const int32_t *seq_lens, const int32_t *q_lens, void *out,
                            cudaStream_t stream) {
    F32Args a;
    a.q = static_cast<const float *>(q);
    a.k_pages = static_cast<const float *>(k_pages);
    a.v_pages = static_cast<const float *>(v_pages);
    a.block_table = block_table;
    a.seq_lens = seq_lens;
    a.q_lens = q_lens;
    a.out = static_cast<float *>(out);
    a.status = ctx->status;
    a.partials = ctx->chunk_ws;
    a.counters = ctx->counters;
    a.max_items = ctx->counters_len;
    a.batch = p.batch;
    a.Hq = p.num_q_heads;
    a.Hkv = p.num_kv_heads;
    a.num_pages = p.num_pages;
    a.max_pages = p.max_pages_per_seq;
    a.rows = p.total_q;
    const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 1.0f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * 1.4426950408889634f;
    const int g = p.num_q_heads / p.num_kv_heads;
    return p.head_dim == 64 ? launch_g<64>(ctx, g, a, stream) : launch_g<128>(ctx, g, a, stream);
}

}  // namespace arb
