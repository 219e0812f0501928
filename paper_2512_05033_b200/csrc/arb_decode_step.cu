// One decode token in one launch (bf16, head_dim 64 or 128, group size <= 8): the cache write of the token's new
// K/V rows, split-KV attention over the paged cache, the split combine and the length update, all in one
// kernel.  This is what a token of a draft or target step costs in Algorithm 1 of the paper ("Sample draft
// step" / "Sample target step": z_i ~ q(z_i | x, z_<i), Section 3.1): every call of that chain reads what the
// call before it wrote, so nothing overlaps and a token pays the latency of every launch on its way.  Three
// launches (append, decode, combine) become one.
//
// What is shared with the two-kernel decode (arb_decode_mma.cu): the flat (sequence, kv head, page) list cut
// into equal ranges per CTA, a ring of 4 KB page tiles fed through tiled TMA copies (here by two producer warps, one for K and
// one for V), one consumer warp per page with its own online softmax.  What differs:
//   - The product is transposed.  S^T = K q^T puts the 16 keys of a page on the 16 rows of an m16n8k16 tile and
//     the group's heads (padded to 8) on its 8 columns; O^T += V^T P^T does the same for the second product.
//     A page costs 8 + 8 MMAs instead of 16 + 16, the accumulators take 32 registers instead of 64, and the
//     CTA runs eight consumer warps, two per scheduler, which hide one another's latencies.  P^T reaches the
//     second product's B fragment through two movmatrix transposes; the row maximum is a reduction over the
//     lanes that share a column pair (three shuffles).
//   - The kernel waits for its predecessor near its top (griddepcontrol.wait) and lets its successor come up at
//     once (griddepcontrol.launch_dependents; beside chunks only behind its own wait): launched as a programmatic dependent
//     it is resident when the kernel before it ends, and by then it has read lengths and table and knows its work.  What it
//     read is a guess, since the predecessor may be writing either: it is read again behind the wait, while the first
//     tiles are on their way, and where anything differs the CTA starts over (see `guess`).
//   - The combine is inside, and the partials are their own arrival signal: a CTA that holds a part of a split (sequence, kv
//     head) stores it into its slot of an exchange buffer whose words hold a value no result has, and leaves; a CTA that
//     merges reads the slots until every word has come, writes the rows and puts the value back.  It waits only for CTAs
//     that drew an earlier ticket, which have started, so every wait ends whatever else is running.  The merging CTA is one
//     with nothing else to do (the last tickets, see kMergerShare), or the one that holds the item's last part; of an item of
//     many parts the last CTA of a run of them hands on the run's sum.
//   - With k_new / v_new given, the warp that owns a sequence's last page puts the token's new row into the
//     tile in shared memory (the tile arrives with whatever the slot held) and stores it to the pool; the
//     lengths move forward once every CTA has read them (a counter in the prologue tells the last reader).
//
// The template parameter KV names the cache.  Compiled a second time (KV = E4M3) the kernel serves an E4M3 cache
// (arb_decode_step_e4m3: the token of a quantised draft).  A page tile is 2 KB of codes, widened to f16 (exact) on its way
// into the MMA fragments, f16 MMAs (q converted bf16 -> f16, P rounded to f16).  The token's new rows are
// quantised by the warp that patches them in (x * inv_scale, nearest code, saturating: the arithmetic of
// arb_kv_append_e4m3) and stored to the pool as codes.
// A third time (KV = 4-bit; arb_decode_step_i4) it serves a cache of 4-bit codes with one fp32 scale per (token, kv head)
// row: a stage is 1 KB of codes and the rows' 16 scales; codes widen to bf16 (exact), the scales of a lane's two keys
// multiply the scores and the weights, and the MMAs are the bf16 ones; the
// token's rows are quantised in the kernel (row max by shuffles, IEEE divisions, nearest with ties to even).
//
// Fragments out of codes.  The sum over dimensions may run in any order and the rows of O^T may stand for any dimensions, so a
// lane takes what lies together: for S^T the 32 dimensions 32 tq .. of key rows gq and gq + 8 (step ks: dimensions
// 32 tq + 4 ks ..; q is loaded in the same order), for O^T the 16 dimensions 16 gq .. of its four key rows, two rows' codes
// sorted into pairs by byte permutes (accumulator rows gq and gq + 8 of m-tile mt: dimensions 16 gq + 2 mt and + 1).  A page
// is 4 + 4 16-byte loads of codes and two or three instructions per fragment register.  Widened into a tile in shared
// memory and read back by ldmatrix, which this replaced, a page took a warp 1.4 us and the consumers set the pace of
// every call: tokens of the target shape (16 sequences of 4k to 32k, 8 kv heads) E4M3 199 -> 108 us (6.0 TB/s, 0.93 of the
// measured copy rate), 4-bit 192 -> 138 us (2.5 TB/s; the copies' issue and the page chain share the time: 132 us without
// the scales' copies, 118 without the products); the draft shape 16.5 -> 14.4 us, either cache
// (of the form of the call at the time; now 9.1 us over E4M3, 10.4 us over 4-bit codes).
#include "arb_decode_tc.cuh"

#include <type_traits>

namespace arb {

namespace {

constexpr int kHalfTile = kPage * 128;        // 2 KB: 64 dimensions of a (page, kv head) tile of K or of V
constexpr int kCodeTileBytes = kPage * kD;    // 2 KB: the same tile of an E4M3 cache
constexpr int kI4CodeBytes = kPage * kD / 2;  // 1 KB: the same tile of a 4-bit cache (16 rows x 64 bytes, not swizzled) ...
constexpr int kI4ScaleBytes = kPage * 4;      // ... followed by the 16 fp32 scales of its rows
constexpr int kI4StageBytes = 1152;           // both, rounded up to 128
enum { kKvBf16 = 0, kKvE4m3 = 1, kKvI4 = 2 }; // the cache a kernel instance reads
constexpr int kCW = 8;                        // consumer warps
constexpr int kCT = kCW * 32;                 // consumer threads
constexpr int kProdWarp = kCW;                // the producer warps, and behind them one for bookkeeping: length update,
                                              // rows of refused sequences
// A warp issues a tiled copy every hundred cycles or so, whatever it brings, so two warps issue, one K and one V.  Against one
// warp: rounds of the step loop 1196 -> 1137 us, a token of 8 x 8 kv heads over 1k to 8k 30.2 -> 28.9 us, draft-shaped
// tokens the same within 1 %, and where a tile is 2 KB or less more: 16 x 8 kv heads of 64 dimensions (150 MB) 38 -> 32 us,
// draft-shaped tokens over 4-bit codes 17.6 -> 16.7 us.
constexpr int kAuxWarp = kCW + 2;
constexpr int kVerifyWarp = kCW - 1;          // the consumer warp that compares the guess (see decode_step_kernel) with what is final
constexpr int kNT = 32 * (kCW + 3);
// Named barriers: the consumers', and behind the comparison of the guess one for each kind of warp, so that none waits for
// another's copies or prefetches (the consumers behind the producers' first copies: 4-bit tokens 10.8 -> 12.0 us).
enum { kBarConsumers = 1, kBarPages = 2, kBarConsumersTold = 3, kBarProducersTold = 4, kBarAuxTold = 5 };

// The exchange of a split item's parts.  A slot is what one CTA hands on: the group's outputs and (max, sum) per head, every
// 32-bit word of it kEmpty until it is stored, and kEmpty again once it has been read.  A NaN of a result never has these bits
// (see not_empty).  Against partials, a fence, an arrival counter and the last to arrive reading what the others left, a
// draft-shaped token 12.4 -> 11.6 us, one of a single sequence of 256 tokens 7.3 -> 6.6 us.
constexpr uint32_t kEmpty = 0xffffffffu;
// A call of few items gives each a CTA that streams nothing and merges it: the others leave when they have stored their parts,
// the next kernel's CTAs come up in their places, and where they would come late, behind a merge, there are the next
// kernel's mergers, which have time: draft-shaped token (16 items) 11.0 -> 10.85 us, over E4M3 codes 10.0 -> 9.6 us.  Up to a
// kMergerShare-th of the CTAs, and only where one of the others then streams at most kMergerPages more: that is a microsecond or
// so, what a merger saves (with more, 32 items of 16 sequences of 2k to 8k over E4M3 codes 14 -> 15 us, 30 of 28k 69.5 -> 70.1 us).
// Nor where there is less than a CTA's smallest range for each of the others (they would leave CTAs without work anyway, and an item's
// last part is sooner merged where it is: 36 items of 50 pages 8.8 -> 7.8 us without, 8 over 4-bit codes 7.8 -> 7.5 us), nor for items of more
// than kMergerParts parts (2 and 4 items: 0.1 us).
constexpr int kMergerShare = 4, kMergerPages = 5, kMergerParts = 32;
// What a boundary costs is time (the warps meet, a second arrival, perhaps a second merge), a few microseconds
// whatever the call's size: as pages it is the CTA's even share, but no more than this many.
constexpr int kBoundaryCap = 32;
// The first kAheadPages page tiles of a CTA's range are asked into L2 before the wait for the predecessor (the bookkeeping warp
// does, off every other warp's path): in a chain of dependent calls the bytes of call n + 1 cross from HBM while call n is in
// its latency-bound tail.
// Copies for L2 pass through the unit that brings the tiles, so many of them stand in front of the first: 0 / 4 / 8 / 16 / 24
// pages, draft-shaped token 11.3 / 10.7 / 10.6 / 10.7 / 10.9 us, 48 x 2 kv heads of 512 to 2048 tokens 16.4 / 16.2 / 15.9 / 15.8 /
// 15.3 us, 16 x 8 heads of 64 dimensions 30.5 / 30.1 / 30.0 / 29.7 / 29.8 us.  (By prefetch instructions the lines held up the
// loads behind them: 11.8 us.)
constexpr int kAheadPages = 16;
constexpr int kLensCycles = 10000;   // a few microseconds: the lengths move one or two after the predecessor's end

// The decode rows of a call with chunks stream while the chunks compute, on SMs of their own: alone an SM draws about 77 GB/s
// (65 of them 5 TB/s), beside chunks less.  Both kinds of work are known from the lengths; the decode rows get the share of
// the SMs that kBesideWeight times their work is of the whole, counted in page tiles: a page of a kv head is 1, 128 keys of a
// pair of chunk row tiles are kBesidePairTile (2.3 us against 0.106 us), of a lone row tile kBesideLoneTile.  A serving
// iteration (32 decode rows, 32 steps, lognormal lengths) 806 -> 748 us at full clock, 921 -> 871 us under the power cap (weights
// 1.33 / 1.9 / 2.6 / 3.5: 813 / 749 / 746 / 769 us); one 16-token step beside 15 decode rows of 4k to 32k 217 -> 199 us (on a
// fixed 65 SMs 271), four of 32 tokens beside 60 rows of 500 to 3000 114 -> 100 us, one of 8 beside 7 draft-shaped rows 33 -> 24 us.
// The same numbers serve E4M3 calls and 64-dimension heads, whose pages are half the bytes.  With both tile weights times
// 0.6 / 1 / 1.5 / 2 / 2.6: the serving iteration over E4M3 codes 828 / 834 / 843 / 940 / 1002 us (one after the other 828),
// with 64-dimension heads 668 / 680 / 676 / 677 / 772 us; 8 rows beside 8 steps of 16 to 32 tokens, 28 / 4 heads, E4M3 265 / 267 /
// 273 / 270 / 260 us (one after the other 297), 64 dimensions 240 / 239 / 240 / 238 / 234 us: flat around 1.
constexpr float kBesideWeight = 2.2f;
constexpr int kBesidePairTile = 22, kBesideLoneTile = 13;

struct StepArgs {
    const char *q;
    const char *k_new, *v_new;   // [rows, Hkv, D]; null: no cache write, seq_lens already count the token
    char *k_pool, *v_pool;
    const int32_t *block_table;
    int32_t *seq_lens;
    const int32_t *q_lens;
    char *out;
    float *part_o;     // [CTAs][2][G][D]  the exchange slots (see kEmpty): of an item's later parts, and of its first part
    float *part_ml;    // [CTAs][2][kMaxGroup][2]
    unsigned *ticket;  // the next CTA's number; back at zero when the last has drawn
    int *lens_counter; // CTAs that have read the lengths, zero between calls and once the lengths have moved
    int guess;         // lengths and table may be read before the predecessor has ended
    uint32_t *status;
    int batch, Hq, Hkv, num_pages, max_pages;
    int beside;        // the kernel launched next runs beside this one (see launch_decode_step)
    int whole_rows;    // the tensor maps are 3-D: one copy per page tile instead of one per half
    int rows;          // rows of q and out
    int min_chunk;     // fewest pages worth giving a CTA
    int boundary_pct;  // cost of a (sequence, kv head) boundary inside a CTA's range: percent of min(even share, kBoundaryCap) pages
    float scale_log2;  // softmax scale (times the key scale of an E4M3 cache) * log2(e)
    float v_scale;     // value scale of an E4M3 cache, 1 otherwise
    float k_inv_scale, v_inv_scale;   // E4M3 cache with a cache write: code = e4m3(x * inv_scale)
    float *k_scales, *v_scales;       // 4-bit cache: the scale pools [num_pages, Hkv, 16]
};

constexpr int kQPitch = kD * 2 + 16;   // of q in shared memory: neighbouring heads start 4 banks apart

template <int STAGES>
struct Tail {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    alignas(16) char q[kMaxGroup * kQPitch];   // the group's heads of q, of the first segment of a guess
    int pages[32];        // guessed page numbers of the CTA's first look-ups
    int differs;          // the comparing warp's finding: the guess does not hold
    int ended;            // the predecessor is known to have ended
    int abort;
    int ticket;
};

template <int G, int HD>
struct Cfg {
    static constexpr int kOStride = HD + 4;               // floats between two heads of a warp record (spreads the banks)
    static constexpr int WREC = 2 * 8 + G * kOStride;     // warp record: [m[8] | l[8] | o[G][kOStride]]
    static constexpr int OSM_BYTES = kCW * WREC * 4;
};

template <int G, int STAGES, int KV, int HD>
size_t smem_bytes(int batch) {
    using C = Cfg<G, HD>;
    constexpr int kTileBytes = HD / 64 * kHalfTile;
    const size_t tiles = (size_t)STAGES * (KV == kKvE4m3 ? kCodeTileBytes : KV == kKvI4 ? kI4StageBytes : kTileBytes);
    return 1024 + tiles + C::OSM_BYTES + sizeof(Tail<STAGES>) + sizeof(int) * (6 * (size_t)batch + 3);
}

__device__ __forceinline__ float4 load_slot4(const float4 *p) {   // not ordered among one another: each word is its own signal
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 load_slot2(const float2 *p) {
    float2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_slot4(float4 *p, float4 v) {
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void store_slot2(float2 *p, float2 v) {
    asm volatile("st.relaxed.gpu.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ int load_now(const int32_t *p) {   // from L2, whoever wrote it and whenever
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void raise_flag(int *flag) {   // in shared memory; what happened before is seen by who sees it raised
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(flag)), "r"(1) : "memory");
}
__device__ __forceinline__ bool flag_raised(const int *flag) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(flag)) : "memory");
    return v != 0;
}
__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ bool is_empty(float x) { return __float_as_uint(x) == kEmpty; }
__device__ __forceinline__ bool any_empty(float4 v) { return is_empty(v.x) || is_empty(v.y) || is_empty(v.z) || is_empty(v.w); }
// a word fit for a slot: a NaN with kEmpty's bits becomes another NaN
__device__ __forceinline__ float not_empty(float x) { return is_empty(x) ? __uint_as_float(0x7fffffffu) : x; }

__device__ __forceinline__ uint32_t tile_off(int r, int c) {   // 16-byte chunk c of row r of a swizzled bf16 tile
    return (uint32_t)((c >> 3) * kHalfTile + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float2 unpack_f16(uint32_t v) {
    float lo, hi;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tcvt.f32.f16 %0, l;\n\tcvt.f32.f16 %1, h;\n\t}" : "=f"(lo), "=f"(hi) : "r"(v));
    return make_float2(lo, hi);
}
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t v) {
    return pack_f16(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
// two E4M3 codes (a 16-bit pair) -> f16x2, exact; the low byte lands in the low half
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint16_t v) {
    uint32_t r;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"(v));
    return r;
}
// two values -> two E4M3 codes (nearest, ties to even, saturating); lo lands in the low byte
__device__ __forceinline__ uint32_t e4m3x2_from_f32(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
// 4-bit cache: a 32-bit word holds 8 dimensions as nibbles (code + 8), nibble i and nibble i + 4 being the neighbouring
// dimensions 2i and 2i + 1.  A nibble in the low bits of the bf16 128 counts in ones (128 + nibble); one exact
// subtraction of 136 leaves the code.  The codes themselves enter the products: left biased (the number 16 + nibble is an
// instruction cheaper) they make every partial sum of S = q . k carry 24 sum(q), and a q with one large component then
// lost what the other dimensions add.
__device__ __forceinline__ uint32_t i4_pair_to_bf16x2(uint32_t w, int i) {
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(((w >> (4 * i)) & 0x000F000Fu) | 0x43004300u), "r"(0x3F803F80u), "r"(0xC308C308u));
    return r;
}

// Codes of one key row for S^T -> the two registers of k-step ks: row = this lane's 32 dimensions (8 or 4 words).
template <bool E4M3>
__device__ __forceinline__ void k_fragment(const uint32_t *row, int ks, uint32_t &a0, uint32_t &a2) {
    if constexpr (E4M3) {
        a0 = e4m3x2_to_f16x2((uint16_t)row[ks]);
        a2 = e4m3x2_to_f16x2((uint16_t)(row[ks] >> 16));
    } else {
        a0 = i4_pair_to_bf16x2(row[ks >> 1], 2 * (ks & 1));
        a2 = i4_pair_to_bf16x2(row[ks >> 1], 2 * (ks & 1) + 1);
    }
}
// Codes of two neighbouring key rows for O^T, 16 dimensions each (4 or 2 words) -> the registers of m-tile mt: the two
// keys' values of dimension 2 mt (a0) and 2 mt + 1 (a1) of the 16.
template <bool E4M3>
__device__ __forceinline__ void v_fragment(const uint32_t *ra, const uint32_t *rb, int mt, uint32_t &a0, uint32_t &a1) {
    if constexpr (E4M3) {
        const uint32_t pair = __byte_perm(ra[mt >> 1], rb[mt >> 1], (mt & 1) ? 0x7362 : 0x5140);
        a0 = e4m3x2_to_f16x2((uint16_t)pair);
        a1 = e4m3x2_to_f16x2((uint16_t)(pair >> 16));
    } else {
        a0 = i4_pair_to_bf16x2(__byte_perm(ra[mt >> 2], rb[mt >> 2], 0x5410), mt & 3);
        a1 = i4_pair_to_bf16x2(__byte_perm(ra[mt >> 2], rb[mt >> 2], 0x7632), mt & 3);
    }
}

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A sequence takes part when it decodes (q_len 1) and its length after the token fits the block table.
// L0: the length the call finds in seq_lens; with a cache write the token lands at position L0.
template <bool APPEND>
__device__ __forceinline__ bool step_ok(int n, int L0, int max_pages) {
    if (n != 1) return false;
    const long long L = (long long)L0 + (APPEND ? 1 : 0);
    return L0 >= (APPEND ? 0 : 1) && L <= (long long)max_pages * kPage;
}

// a / b for 0 <= a, 0 < b: through the float reciprocal with a correction step while a is exactly representable
// (the plan sits on every CTA's path to its first copy, and an integer division is some forty dependent instructions)
__device__ __forceinline__ int fast_div(int a, int b) {
    if (a >= (1 << 24)) return a / b;
    int q = __float2int_rz(__fdividef((float)a, (float)b));
    const int r = a - q * b;
    if (r < 0) --q; else if (r >= b) ++q;
    return q;
}

// a / b where the quotient is a kv head index (small): a few subtractions beat any division.  (Whoever asks holds a page of the
// sequence, so b > 0; the loop ends for any b.)
__device__ __forceinline__ int small_div(int a, int b, int &rem) {
    int q = 0;
    while (a >= b && b > 0) { a -= b; ++q; }
    rem = a;
    return q;
}

// The cut of the flat (sequence, kv head, page) list into per-CTA ranges.  A CTA whose range crosses from one
// (sequence, kv head) into the next pays for it (the warps meet, their records are merged, the next q is
// loaded), and both items wait for it.  So a boundary counts as
// `pen` pages of work: the list is cut evenly in a padded coordinate in which every item is preceded by `pen`
// virtual pages.  Item j (in list order) with real range [s, s + n) occupies [s + j pen, s + (j + 1) pen + n) there,
// its real pages the last n of them.  Everything after the cut works in real coordinates.
struct Plan {
    const int *pref;   // [B + 1] real flat start of sequence b (pages times kv heads)
    const int *act;    // [B + 1] sequences before b that take part
    const int *slen;   // [B] length of sequence b (with the new token)
    int B, Hkv, pen, chunk, total_padded;
    int stream;        // CTAs that stream; with `mergers` those behind them have an item each to merge
    bool mergers;

    __device__ __forceinline__ int pages_of(int b) const { return pref[b + 1] != pref[b] ? (slen[b] + kPage - 1) / kPage : 0; }
    __device__ __forceinline__ int padded_start(int b) const { return pref[b] + pen * Hkv * act[b]; }
    // real flat position of padded position r inside sequence b (a virtual page maps to the first real page behind it)
    __device__ __forceinline__ int real_in(int b, long long r) const {
        const int pages = pages_of(b);
        int o2;
        const int kvh = small_div((int)r - padded_start(b), pages + pen, o2);
        return pref[b] + kvh * pages + max(0, o2 - pen);
    }
    // the CTA that holds real page `pg` of item (b, kvh)
    __device__ __forceinline__ int cta_of(int b, int kvh, int pages, int pg) const {
        return fast_div(padded_start(b) + kvh * (pages + pen) + pen + pg, chunk);
    }
    // the sequence that holds real flat position r, walking up from a sequence known to start at or before r
    __device__ __forceinline__ int seq_of(int r, int b) const {
        while (b + 1 < B && pref[b + 1] <= r) ++b;
        return b;
    }
};

// Next segment of the real flat range [cur, r1); `b` is the sequence of the segment before (or of r0) and moves along.
__device__ __forceinline__ bool next_segment(int &cur, int r1, int &b, const Plan &pl, Segment &s) {
    if (cur >= r1) return false;
    b = pl.seq_of(cur, b);
    const int pages = pl.pages_of(b);
    int pg0;
    const int kvh = small_div(cur - pl.pref[b], pages, pg0);
    const int s1 = pl.pref[b] + (kvh + 1) * pages;
    const int end = s1 < r1 ? s1 : r1;
    s.b = b;
    s.kvh = kvh;
    s.pg0 = pg0;
    s.pg1 = pg0 + (end - cur);
    s.L = pl.slen[b];
    s.bk = b * pl.Hkv + kvh;
    s.c_first = -1;   // filled in by parts_of when the segment's result is parked
    s.nparts = 0;
    cur = end;
    return true;
}

__device__ __forceinline__ void parts_of(const Plan &pl, Segment &s) {
    const int pages = pl.pages_of(s.b);
    s.c_first = pl.cta_of(s.b, s.kvh, pages, 0);
    s.nparts = pl.cta_of(s.b, s.kvh, pages, pages - 1) - s.c_first + 1;
}

// Head dimension 64: a tile is 2 KB (one box), the products have half the steps, and the softmax weights enter the
// second product as two bf16 terms (p = hi + lo: 16 significant bits, like the fp32 weights of the CUDA-core kernel this
// form replaced, to within the rounding of the output); the memory system sets the pace, so the second term costs nothing.
template <int G, int STAGES, bool APPEND, int KV, int HD>
__global__ void __launch_bounds__(kNT, 1)
decode_step_kernel(const StepArgs a, const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map) {
    constexpr int kOwnStages = STAGES / 2;             // of one producer warp
    constexpr int kBatch = kOwnStages < 32 ? kOwnStages : 32;   // lanes of a producer warp issuing side by side
    using C = Cfg<G, HD>;
    using Tail = arb::Tail<STAGES>;
    constexpr int WREC = C::WREC, kOStride = C::kOStride;
    constexpr int kD = HD, kTileBytes = HD / 64 * kHalfTile;   // a tile of a bf16 cache
    constexpr bool SPLIT_P = HD == 64;
    constexpr bool E4M3 = KV == kKvE4m3, I4 = KV == kKvI4, CODES = KV != kKvBf16;
    constexpr int kStageBytes = E4M3 ? kCodeTileBytes : I4 ? kI4StageBytes : kTileBytes;   // a ring stage
    constexpr int kTxBytes = I4 ? kI4CodeBytes + kI4ScaleBytes : kStageBytes;               // what the copies of a stage bring
    constexpr int kRowBytes = E4M3 ? kD : I4 ? kD / 2 : kD * 2;         // bytes of a cache row
    constexpr int kRingBytes = STAGES * kStageBytes;
    constexpr int kRowWords = E4M3 ? 8 : 4;                             // 32-bit words of codes a lane takes per key row for S^T
    static_assert(!CODES || HD == 128, "code caches have 128-dimension rows");
    static_assert(G >= 1 && G <= 8, "the group's heads are the 8 columns of the tile");
    static_assert(STAGES % (2 * kCW) == 0, "a ring stage always belongs to the same warp of a segment");

    extern __shared__ char smem_raw[];
    char *base = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    char *ring = base;
    float *osm = reinterpret_cast<float *>(base + kRingBytes);
    Tail *tail = reinterpret_cast<Tail *>(base + kRingBytes + C::OSM_BYTES);
    int *pref = reinterpret_cast<int *>(tail + 1);
    int *row0 = pref + a.batch + 1;
    int *act = row0 + a.batch + 1;
    int *slen = act + a.batch + 1;
    int *raw_n = slen + a.batch, *raw_len = raw_n + a.batch;   // q_lens and seq_lens as they were read

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int B = a.batch, Hkv = a.Hkv;

    if (tid == kCT) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&k_map)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&v_map)) : "memory");
    }
    // The CTA's number: in the order in which CTAs start, which is what the waits of the merge rest on (see kEmpty).  The
    // successor may come up, and draw from the same counter, only once this has been drawn.
    if (tid == kAuxWarp * 32) {
        tail->ticket = (int)atomicInc(a.ticket, gridDim.x - 1);
        if (!a.beside) let_successor_start();
    }
    if (warp == 0) {
        for (int st = lane; st < STAGES; st += 32) {
            mbar_init(&tail->full[st], 1);
            mbar_init(&tail->empty[st], 1);
        }
        if (lane == 0) {
            tail->abort = 0;
            tail->ended = 0;
            pref[0] = 0;
            row0[0] = 0;
            act[0] = 0;
        }
        mbar_fence_init();
    }
    if (!a.guess) {
        wait_for_predecessor();
        // (beside: it does not wait for this kernel, but it may read what the predecessor wrote.  One thread's call counts for the
        // CTA, so it is the one that has drawn the ticket: the kernel behind the next draws from the same counter.)
        if (a.beside && tid == kAuxWarp * 32) let_successor_start();
    }
    for (int b = tid; b < B; b += kNT) {
        raw_n[b] = load_now(a.q_lens + b);
        raw_len[b] = load_now(a.seq_lens + b);
    }
    __syncthreads();   // barriers, ticket and lengths are there
    const int cta = tail->ticket;

    // ---- prologue: lengths -> page counts and q row offsets -------------------------------------------------
    // Every warp works the plan out for itself, and all store the same values into the tables.  (One warp planning for all, with
    // two barriers and a search of its tables, took 1.2 us; a draft-shaped token 12.9 -> 12.6 us, one of a single 256-token
    // sequence 6.8 -> 6.5 us.)  Of a batch of more than 32 the block makes the tables together.
    Plan pl;
    pl.pref = pref; pl.act = act; pl.slen = slen; pl.B = B; pl.Hkv = Hkv;
    // total work and items -> what a boundary counts for, the padded list's length, the even share of it
    int ctas;   // that take part
    auto per_cta = [&](int x) -> int { return fast_div(x + ctas - 1, ctas); };
    auto chunk_work = [&](int n, int L) -> float {   // of one sequence, in page tiles
        if (n < 2 || L < n) return 0.f;
        const int tiles = (n * G + 127) / 128;
        return (float)Hkv * (float)((L + 127) / 128) * (float)((tiles >> 1) * kBesidePairTile + (tiles & 1) * kBesideLoneTile);
    };
    auto shares = [&](int total, int items, float chunks) {
        ctas = (int)gridDim.x;
        if (a.beside) {
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) chunks += __shfl_xor_sync(0xffffffffu, chunks, off);
            const float mine = kBesideWeight * (float)total;
            ctas = min(ctas, max(4, __float2int_ru((float)ctas * __fdividef(mine, mine + chunks + 1.f))));
        }
        const int others = ctas - items;
        pl.mergers = !a.beside && items * kMergerShare <= ctas && items * kMergerParts >= ctas && total >= a.min_chunk * others &&
                     (long long)others * kMergerPages >= (long long)total / ctas * items;
        if (pl.mergers) ctas -= items;
        pl.stream = ctas;
        const int even = max(a.min_chunk, per_cta(total));
        pl.pen = items > 1 ? (min(even, kBoundaryCap) * a.boundary_pct + 99) / 100 : 0;
        pl.total_padded = total + pl.pen * items;
        pl.chunk = max(a.min_chunk, per_cta(pl.total_padded));
    };
    int ends[2], seq0 = 0;   // this CTA's range, and the sequence it begins in
    auto lengths_of = [&](int b, int &pages, int &rows, int &ok, int &L) {
        const int n = raw_n[b], L0 = raw_len[b];
        ok = step_ok<APPEND>(n, L0, a.max_pages) ? 1 : 0;
        L = L0 + (APPEND ? 1 : 0);
        pages = ok ? (L + kPage - 1) / kPage * Hkv : 0;
        rows = n > 0 ? n : 0;
    };
    auto scan3 = [&](int &vp, int &vr, int &va) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int tp = __shfl_up_sync(0xffffffffu, vp, off);
            const int tr = __shfl_up_sync(0xffffffffu, vr, off);
            const int ta = __shfl_up_sync(0xffffffffu, va, off);
            if (lane >= off) { vp += tp; vr += tr; va += ta; }
        }
    };
    auto make_plan = [&]() {
        if (B <= 32) {
            int vp = 0, vr = 0, va = 0, L = 0;
            if (lane < B) lengths_of(lane, vp, vr, va, L);
            const int own = vp, ok = va, rows = vr;
            scan3(vp, vr, va);
            if (lane < B) { pref[lane + 1] = vp; row0[lane + 1] = vr; act[lane + 1] = va; slen[lane] = L; }
            const int total = __shfl_sync(0xffffffffu, vp, 31);
            shares(total, __shfl_sync(0xffffffffu, va, 31) * Hkv, a.beside ? chunk_work(rows, L) : 0.f);
            // the lane whose sequence holds an end of the range works it out (see Plan)
            const int pages = ok ? (L + kPage - 1) / kPage : 0, item = pages + pl.pen;
            const int first = vp - own + pl.pen * Hkv * (va - ok);
    #pragma unroll
            for (int w = 0; w < 2; ++w) {
                const long long rel = (long long)(cta + w) * pl.chunk - first;
                const bool here = ok && rel >= 0 && rel < (long long)item * Hkv;
                const int r = here ? (int)rel : 0, kvh = fast_div(r, max(item, 1));
                const int pos = vp - own + kvh * pages + max(0, r - kvh * item - pl.pen);
                const unsigned mask = __ballot_sync(0xffffffffu, here);
                const int src = __ffs(mask) - 1;
                const int at = __shfl_sync(0xffffffffu, pos, src & 31);
                ends[w] = mask ? at : total;   // nobody's: behind the end of the list
                if (w == 0) seq0 = max(src, 0);
            }
            __syncwarp();
        } else {
            for (int b = tid; b < B; b += kNT) {
                int vp, vr, va, L;
                lengths_of(b, vp, vr, va, L);
                pref[b + 1] = vp; row0[b + 1] = vr; act[b + 1] = va; slen[b] = L;
            }
            __syncthreads();
            if (warp == 0) {
                int carry_p = 0, carry_r = 0, carry_a = 0;
                for (int b0 = 0; b0 < B; b0 += 32) {
                    const int b = b0 + lane;
                    int vp = b < B ? pref[b + 1] : 0, vr = b < B ? row0[b + 1] : 0, va = b < B ? act[b + 1] : 0;
                    scan3(vp, vr, va);
                    if (b < B) { pref[b + 1] = vp + carry_p; row0[b + 1] = vr + carry_r; act[b + 1] = va + carry_a; }
                    carry_p += __shfl_sync(0xffffffffu, vp, 31);
                    carry_r += __shfl_sync(0xffffffffu, vr, 31);
                    carry_a += __shfl_sync(0xffffffffu, va, 31);
                }
            }
            __syncthreads();
            // both ends of the range with one ballot per 32 sequences: the padded starts ascend, so the sequence that holds a
            // position is the last one that starts at or before it
            const int total = pref[B];
            float chunks = 0.f;
            if (a.beside)
                for (int b = lane; b < B; b += 32) chunks += chunk_work(row0[b + 1] - row0[b], slen[b]);
            shares(total, act[B] * Hkv, chunks);
    #pragma unroll
            for (int w = 0; w < 2; ++w) {
                const long long t = (long long)(cta + w) * pl.chunk;
                int best = 0;
                for (int b0 = 0; b0 < B; b0 += 32) {
                    const int b = b0 + lane;
                    const unsigned mask = __ballot_sync(0xffffffffu, b < B && pl.padded_start(b) <= t);
                    if (mask) best = b0 + 31 - __clz(mask);
                }
                ends[w] = t >= pl.total_padded ? total : pl.real_in(best, t);
                if (w == 0) seq0 = best;
            }
        }
    };

    // ---- the producers' and consumers' first steps ----------------------------------------------------------
    // The kv head of flat triple r, and where its page's number stands in the table.
    auto find_page = [&](int r, const int32_t *&entry, int &kvh) {
        const int lo = pl.seq_of(r, seq0);
        int pg;
        kvh = small_div(r - pref[lo], pl.pages_of(lo), pg);
        const bool in = ARB_IN_RANGE(a.status, pg, a.max_pages) && ARB_IN_RANGE(a.status, kvh, Hkv);
        entry = a.block_table + (in ? (size_t)lo * a.max_pages + pg : 0);
    };
    const int pw = warp - kProdWarp;       // of a producer warp: 0 brings K, 1 V
    const bool is_v = pw == 1;
    const CUtensorMap *map = is_v ? &v_map : &k_map;
    auto issue = [&](uint32_t st, int row) {   // the copies of the page tile that begins at `row` of the 2-D view of the pool
        mbar_arrive_expect_tx(&tail->full[st], kTxBytes);
        if constexpr (I4) {   // 16 rows x 64 bytes of codes, then the rows' 16 scales
            tma_box_load(ring + st * kStageBytes, map, 0, row, &tail->full[st]);
            bulk_load(ring + st * kStageBytes + kI4CodeBytes, (is_v ? a.v_scales : a.k_scales) + row, kI4ScaleBytes, &tail->full[st]);
        } else if constexpr (E4M3) {
            tma_box_load(ring + st * kStageBytes, map, 0, row, &tail->full[st]);   // 16 rows x 128 codes
        } else if constexpr (HD == 64) {
            tma_box_load(ring + st * kTileBytes, map, 0, row, &tail->full[st]);    // 16 rows x 64 dims
        } else if (a.whole_rows) {
            tma_box_load3(ring + st * kTileBytes, map, 0, row, 0, &tail->full[st]);
        } else {
            tma_box_load(ring + st * kTileBytes, map, 0, row, &tail->full[st]);
            tma_box_load(ring + st * kTileBytes + kHalfTile, map, 64, row, &tail->full[st]);
        }
    };
    const int gq = lane >> 2, tq = lane & 3;   // fragment coordinates
    const bool head_ok = gq < G;               // as a B-fragment column: this lane's head is a real one
    // B fragments of q^T (kD dims x 8 heads): k-slice ks holds dims 16 ks + 2 tq, + 1 and + 8 of head gq.  The
    // fragments of the next segment are asked for while this one streams.
    uint32_t qb[kD / 16][2], qn[kD / 16][2];
    auto q_of = [&](const Segment &g, int head) -> const char * {   // of the group's heads
        const int row = row0[g.b];   // (guessed lengths may point anywhere)
        return a.q + ((size_t)((unsigned)row < (unsigned)a.rows ? row : 0) * a.Hq + g.kvh * G + head) * kD * 2;
    };
    auto q_fragments = [&](const char *qh, uint32_t (&dst)[kD / 16][2]) {   // this lane's head in memory of either kind
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) {
            if constexpr (CODES) {   // dimensions 32 tq + 4 ks .. + 3, in the order the codes come in
                const uint2 w = head_ok ? *reinterpret_cast<const uint2 *>(qh + tq * 64 + ks * 8) : make_uint2(0u, 0u);
                dst[ks][0] = E4M3 ? bf16x2_to_f16x2(w.x) : w.x;   // (the operands of one MMA share a type)
                dst[ks][1] = E4M3 ? bf16x2_to_f16x2(w.y) : w.y;
                continue;
            }
            dst[ks][0] = head_ok ? *reinterpret_cast<const uint32_t *>(qh + ks * 32 + tq * 4) : 0u;
            dst[ks][1] = head_ok ? *reinterpret_cast<const uint32_t *>(qh + ks * 32 + 16 + tq * 4) : 0u;
        }
    };
    auto load_q = [&](const Segment &g, uint32_t (&dst)[kD / 16][2]) {
        const int row = row0[g.b];   // (guessed lengths may point anywhere)
        const char *qh = a.q + ((size_t)((unsigned)row < (unsigned)a.rows ? row : 0) * a.Hq + g.kvh * G + (head_ok ? gq : 0)) * kD * 2;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) {
            if constexpr (CODES) {   // dimensions 32 tq + 4 ks .. + 3, in the order the codes come in
                const uint2 w = head_ok ? __ldg(reinterpret_cast<const uint2 *>(qh + tq * 64 + ks * 8)) : make_uint2(0u, 0u);
                dst[ks][0] = E4M3 ? bf16x2_to_f16x2(w.x) : w.x;   // (the operands of one MMA share a type)
                dst[ks][1] = E4M3 ? bf16x2_to_f16x2(w.y) : w.y;
                continue;
            }
            dst[ks][0] = head_ok ? __ldg(reinterpret_cast<const uint32_t *>(qh + ks * 32 + tq * 4)) : 0u;
            dst[ks][1] = head_ok ? __ldg(reinterpret_cast<const uint32_t *>(qh + ks * 32 + 16 + tq * 4)) : 0u;
        }
    };
    Segment s = {};
    int cur = 0, seq_at = 0, page_next = 0, row_next = 0;   // (of a producer's lane: page number and row of its next triple)
    bool have = false;

    // `guess`: in the first round the plan comes from what lengths and table held before the predecessor was known to have
    // ended.  Behind the wait the first ring of tiles and the first q are asked for, while one warp reads lengths and the
    // look-ups' table entries again and tells everyone whether all of it still holds.  Until then nothing has been written
    // and only tiles and q rows were read, in bounds whatever the guess: every warp plans from the same guessed lengths, which
    // are replaced once the block has met.  Where something differs (lengths that the kernel right
    // in front moves, as a rollback does) the copies are waited for, the barriers made new, and the second round plans from
    // what is final.  Three dependent round trips (lengths, table, tile) and the plan become one behind the predecessor's end:
    // tokens of one sequence of 256 / 2048 / 32768 tokens 7.3 / 8.1 / 15.7 -> 6.1 / 6.9 / 13.4 us, draft-shaped 12.4 -> 10.7 us
    // with the mergers.
    // Without a cache write the copies wait for the comparison: what precedes such a call is often the append that
    // moved the lengths.  Or it is a kernel that never lets its successor start early; then nothing was gained by guessing, and
    // the comparison must not cost a round trip.  So where the predecessor has ended by the time of the look-ups, the lengths are
    // compared beside them, and q is on its way into shared memory meanwhile: decode rows of 8 sequences of 2300 tokens, 2 kv heads,
    // behind such a kernel 12.6 -> 11.9 us, behind one another 9.0 -> 8.5, behind an append 15.3 -> 15.6 us.  (With a cache write
    // the first copies do not wait, and the same order made chains slower: 8.3 -> 8.5 us.)
#pragma unroll 1
    for (bool guess = a.guess != 0;; guess = false) {
        make_plan();
        const int nflat = ends[1] - ends[0];
        const int32_t *entry = a.block_table;
        // Without a cache write: has the predecessor ended by now?  (The consumers get to their wait a look-up earlier than the others.)
        // Then what is read from here on is final, and nothing is left to ask into L2 ahead.
        bool over = false;
        int n_now = 0, len_now = 0;   // a batch of at most 32: what is final, of sequence `lane`
        if constexpr (!APPEND) {
            if (guess && warp < kVerifyWarp) {
                wait_for_predecessor();
                if (tid == 0) raise_flag(&tail->ended);
            }
        }
        if (warp >= kVerifyWarp) {
            const bool there = lane < nflat;
            int kvh = 0;
            if (there) find_page(ends[0] + lane, entry, kvh);
            if constexpr (!APPEND)
                if (guess && warp == kVerifyWarp) over = __all_sync(0xffffffffu, flag_raised(&tail->ended));
            if (there && (!guess || warp == kVerifyWarp)) page_next = load_now(entry);
            // A guess is read once, by the warp that compares it, and handed on: what is compared is what is used.
            if (guess && warp == kVerifyWarp) {
                if constexpr (!APPEND)
                    if (over && lane < B && B <= 32) { n_now = load_now(a.q_lens + lane); len_now = load_now(a.seq_lens + lane); }
                tail->pages[lane] = page_next;
                barrier_arrive(kBarPages, 128);
            } else if (guess) {
                named_barrier(kBarPages, 128);
                page_next = tail->pages[lane];
                if constexpr (!APPEND) over = flag_raised(&tail->ended);
            }
            if (there) row_next = (((unsigned)page_next < (unsigned)a.num_pages ? page_next : 0) * Hkv + kvh) * kPage;
        }
        if (guess) {
            if (warp == kAuxWarp && !over && lane < min(nflat, kAheadPages)) {
                const size_t off = (size_t)row_next * kRowBytes;
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.k_pool + off), "r"(kPage * kRowBytes) : "memory");
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.v_pool + off), "r"(kPage * kRowBytes) : "memory");
            }
            wait_for_predecessor();
        }
        bool differs = false;
        if (guess && warp == kVerifyWarp) {
            int entry_now = page_next;
            if (!over && lane < nflat) entry_now = load_now(entry);
            if (!APPEND && over && B <= 32) {
                differs = lane < B && (n_now != raw_n[lane] || len_now != raw_len[lane]);
            } else {
#pragma unroll 4
                for (int b = lane; b < B; b += 32) {
                    n_now = load_now(a.q_lens + b);
                    len_now = load_now(a.seq_lens + b);
                    if (n_now != raw_n[b] || len_now != raw_len[b]) {
                        differs = true;
                        // What has moved goes where the next plan reads it.  Of a batch of more than 32 the plan above has read it in
                        // front of barriers of the block; of a smaller one the other warps may not have read it yet.
                        if (B > 32) { raw_n[b] = n_now; raw_len[b] = len_now; }
                    }
                }
            }
            differs = differs || entry_now != page_next;
            differs = __any_sync(0xffffffffu, differs);
            if (lane == 0) tail->differs = differs;
            barrier_arrive(kBarProducersTold, 96);
            barrier_arrive(kBarAuxTold, 64);
        }
        // Whether the guess was wrong: all but the comparing warp wait for it.  (Barriers of the block's own warps, like
        // __syncthreads: everyone is told the same.)
        auto wrong = [&]() -> bool {
            if (warp < kCW) named_barrier(kBarConsumersTold, kCT);
            else if (warp == kAuxWarp) named_barrier(kBarAuxTold, 64);
            else named_barrier(kBarProducersTold, 96);
            return *(volatile int *)&tail->differs != 0;
        };
        const bool first_copy = (warp == kProdWarp || warp == kProdWarp + 1) && lane < min(nflat, kBatch);
        if constexpr (!APPEND) {   // q comes into shared memory meanwhile: behind the first ring of tiles it takes a microsecond longer
            if (guess && warp < kCW) {
                cur = ends[0];
                seq_at = seq0;
                have = next_segment(cur, ends[1], seq_at, pl, s);
                const char *from = q_of(s, 0);
                for (int c = tid; have && c < G * kD / 8; c += kCT)
                    cp_async16(tail->q + c / (kD / 8) * kQPitch + c % (kD / 8) * 16, from + c * 16);
            }
        }
        const bool sure = !guess || (!APPEND && !wrong());
        if (APPEND || sure) {
            if (first_copy && ARB_IN_RANGE(a.status, row_next, (long long)a.num_pages * Hkv * kPage)) issue(2u * lane + (uint32_t)pw, row_next);
            if (!APPEND && guess) {
                if (warp < kCW) {
                    cp_async_wait_all();
                    named_barrier(kBarConsumers, kCT);
                    q_fragments(tail->q + (head_ok ? gq : 0) * kQPitch, qb);
                }
            } else if (warp < kCW) {
                cur = ends[0];
                seq_at = seq0;
                have = next_segment(cur, ends[1], seq_at, pl, s);
                if constexpr (!APPEND) cp_async_wait_all();   // (a guess that was wrong has asked for q too)
                if (have) load_q(s, qb);
            }
        }
        if (sure || (APPEND && !wrong())) break;
        if (APPEND && first_copy) mbar_wait(&tail->full[2 * lane + pw], 0, &tail->abort, a.status);
        __syncthreads();   // every warp is done with the plan, and with the lengths it came from
        if (B <= 32 && warp == kVerifyWarp && lane < B) { raw_n[lane] = n_now; raw_len[lane] = len_now; }
        if constexpr (APPEND) {
            if (tid == 0) {
                for (int st = 0; st < STAGES; ++st) {
                    mbar_inval(&tail->full[st]);
                    mbar_inval(&tail->empty[st]);
                    mbar_init(&tail->full[st], 1);
                    mbar_init(&tail->empty[st], 1);
                }
                mbar_fence_init();
            }
        }
        __syncthreads();
    }

    if (warp == kAuxWarp) {
        // ================================ bookkeeping warp ==========================================
        // Lengths: nobody in this CTA reads them again, so it counts itself in.  The CTA whose count completes the grid
        // knows that nobody will read seq_lens again and moves them forward: for the sequences that take part
        // and whose new row has a page inside the pool to go to (the same test the writer of the row makes).
        if constexpr (APPEND) {
            // (what the last one needs is on its way meanwhile)
            const int L0 = lane < B ? slen[lane] - 1 : 0, n = lane < B ? row0[lane + 1] - row0[lane] : 0;
            const bool moves = lane < B && step_ok<true>(n, L0, a.max_pages);
            const int pid = moves ? load_now(a.block_table + (size_t)lane * a.max_pages + L0 / kPage) : -1;
            int last = 0;
            if (lane == 0) last = atomicAdd(a.lens_counter, 1) == (int)gridDim.x - 1;
            last = __shfl_sync(0xffffffffu, last, 0);
            if (last) {
                if (moves && (unsigned)pid < (unsigned)a.num_pages) a.seq_lens[lane] = L0 + 1;
                for (int b = lane + 32; b < B; b += 32) {
                    const int L = slen[b] - 1;
                    if (step_ok<true>(row0[b + 1] - row0[b], L, a.max_pages)) {
                        const int page = load_now(a.block_table + (size_t)b * a.max_pages + L / kPage);
                        if ((unsigned)page < (unsigned)a.num_pages) a.seq_lens[b] = L + 1;
                    }
                }
                __threadfence();
                __syncwarp();
                if (lane == 0) *a.lens_counter = 0;
            }
            // Where this CTA leaves, one of the next kernel comes up, and its guess is right once the lengths have moved.  A CTA with
            // little or no work stays until then, or for as long as that should take: its place would only be waited in.
            const long long t0 = clock64();
            while (load_now(a.lens_counter) != 0 && clock64() - t0 < kLensCycles) {
            }
        }
        // Sequences that were asked to decode but cannot: status bit, rows of zeros.
        if (cta == 0) {
            for (int b = 0; b < B; ++b) {
                const int n = row0[b + 1] - row0[b];
                if (n != 1 || pref[b + 1] != pref[b]) continue;
                if (lane == 0) atomicOr(a.status, (uint32_t)ARB_DEV_BAD_SEQ_LEN);
                uint4 *o = reinterpret_cast<uint4 *>(a.out + (size_t)row0[b] * a.Hq * kD * 2);
                for (int i = lane; i < a.Hq * kD * 2 / 16; i += 32) o[i] = make_uint4(0, 0, 0, 0);
            }
        }
        return;
    }

    const int r0 = ends[0], r1 = ends[1];
    const bool merges_only = r0 >= r1;
    if (merges_only && (!pl.mergers || cta < pl.stream || warp >= kCW)) return;
    volatile int *abort = &tail->abort;

    if (warp >= kProdWarp) {
        // ================================ producer warps ===========================================
        // The CTA's flat range of (sequence, kv head, page) triples goes through in groups of 32: lane i finds
        // triple i of the group (a short walk up the prefix table from the range's first sequence) and fetches its block-table entry; the entries
        // of the next group are asked for before the tiles of this one are issued, so that the look-up is off the
        // path after the first group, across sequence boundaries too.  Tiles enter the ring page by page, K then
        // V: one warp issues the K tiles, one the V tiles.  Lanes
        // 0 .. kBatch-1 of a warp each own one stage at a time.
        const int nflat = r1 - r0;
        auto tile_row = [&](int r) -> int {
            const int32_t *entry;
            int kvh;
            find_page(r, entry, kvh);
            int pid = *entry;
            if ((unsigned)pid >= (unsigned)a.num_pages) {
                atomicOr(a.status, (uint32_t)ARB_DEV_BAD_PAGE);
                pid = 0;
            }
            return (pid * Hkv + kvh) * kPage;
        };
        if (lane < nflat && (unsigned)page_next >= (unsigned)a.num_pages) atomicOr(a.status, (uint32_t)ARB_DEV_BAD_PAGE);
        for (int g0 = 0; g0 < nflat; g0 += 32) {
            const int row_cur = row_next;
            const int npages = min(32, nflat - g0);
#pragma unroll 1
            for (int i0 = g0 == 0 ? kBatch : 0; i0 < npages; i0 += kBatch) {   // (the first ring is on its way)
                // the next group's look-up goes out behind this group's first copies, not in front of them
                if (i0 == kBatch && g0 + 32 + lane < nflat) row_next = tile_row(r0 + g0 + 32 + lane);
                const int i = i0 + lane;
                const int row = __shfl_sync(0xffffffffu, row_cur, i & 31);
                const uint32_t cc = 2u * (uint32_t)(g0 + i) + (uint32_t)pw, st = cc % STAGES, par = (cc / STAGES) & 1u;
                // The lanes wait for different stages.  A blocking wait would put the whole warp to sleep until its
                // time limit whenever one stage is not free yet, and copies for stages that are would go out late, in
                // clumps (seen: 0.7 us apart).  So the warp polls, converged: every round each lane tests its own
                // stage without blocking and issues its copy the moment the stage is free.
                bool pending = lane < kBatch && i < npages && ARB_IN_RANGE(a.status, row, (long long)a.num_pages * Hkv * kPage);
                const long long t0 = clock64();
                while (__any_sync(0xffffffffu, pending)) {
                    if (pending && mbar_test_wait(&tail->empty[st], par ^ 1u)) {
                        issue(st, row);
                        pending = false;
                    }
                    if (pending && (*abort || clock64() - t0 > kWaitCycles)) {   // give up, like every other wait
                        if (!*abort) {
                            *abort = 1;
                            atomicOr(a.status, (uint32_t)ARB_DEV_WAIT_TIMEOUT);
                        }
                        pending = false;
                    }
                }
            }
            if (npages <= kBatch && g0 + 32 + lane < nflat) row_next = tile_row(r0 + g0 + 32 + lane);
        }
        // After a timeout the consumers may have left copies unconsumed: wait (bounded) for the last ring's
        // worth, so that no copy is in flight into this CTA's shared memory when it exits.
        if (lane == 0 && *abort) {
            const int n = min(nflat, kOwnStages);
            for (int i = 0; i < n; ++i) {
                const uint32_t cc = (uint32_t)(2 * (nflat - 1 - i) + pw);
                const long long t0 = clock64();
                while (!mbar_try_wait(&tail->full[cc % STAGES], (cc / STAGES) & 1u) && clock64() - t0 < (1ll << 24)) {
                }
            }
        }
        return;
    }

    // ==================================== consumer warps ==========================================
    const int h0 = 2 * tq, h1 = 2 * tq + 1;    // as accumulator columns: the two heads this lane holds
    uint32_t seg_base = 0;                     // ring counter of the segment's first tile
    // A part of a split item is either in this CTA's last segment or its only one, and then it goes to a slot, or it is the last
    // part of its item, in the CTA's first segment: that goes to a slot too, or, without mergers, this CTA merges.
    constexpr int kLph = kD / 4;               // lanes of a head: one per 4-dimension piece
    constexpr int VECS = G * kLph;             // 4-dimension pieces of the group's outputs, one per consumer thread
    constexpr int kMergeBatch = 16;            // parts merged per round of loads, straight into registers (24: they spill, + 0.5 us)
    // Of an item of more parts than two rounds bring, the last of every kMergeFan parts hands on the sum: a round for a run, one for
    // the sums and the rest.  Runs of 32 took two and one: 4 items of 37 parts 11.8 -> 10.8 us, 2 of 74 11.8 -> 10.9 us.
    constexpr int kLongBatch = 20, kMergeFan = kMergeBatch + 1, kDirectParts = 2 * kMergeBatch + 1;
    static_assert(VECS <= kCT, "one piece per consumer thread");
    static_assert(kMergeBatch <= kLph, "a lane of a head per part");
    int gather_first = -1, gather_part = 0;    // the item to merge: the CTA of its first part, the number of this CTA's part
    bool gather_last = false;                  // ... and whether that completes the item (else the sum of a run goes on)
    bool in_runs = false;                      // ... of kMergeFan parts
    size_t gather_out = 0;
    float4 own = make_float4(0.f, 0.f, 0.f, 0.f);   // this CTA's part of it
    float own_m = -INFINITY, own_l = 0.f;
    auto publish = [&](float4 x, float M, float l, int part) {
        if (!ARB_IN_RANGE(a.status, cta, gridDim.x)) return;
        const int slot = 2 * cta + (part == 0);
        store_slot4(reinterpret_cast<float4 *>(a.part_o) + (size_t)slot * VECS + tid,
                    make_float4(not_empty(x.x), not_empty(x.y), not_empty(x.z), not_empty(x.w)));
        if (tid % kLph == 0)
            store_slot2(reinterpret_cast<float2 *>(a.part_ml) + (size_t)slot * kMaxGroup + tid / kLph, make_float2(not_empty(M), not_empty(l)));
    };
    const int eh = tid / (kD / 4);     // head of this thread's piece
    auto write_row = [&](size_t out_base, float4 x, float inv) {
        if (!ARB_IN_RANGE(a.status, out_base + G * kD - 1, (size_t)a.rows * a.Hq * kD)) return;
        *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(a.out) + out_base + (size_t)tid * 4) =
            make_uint2(pack_bf16(x.x * inv, x.y * inv), pack_bf16(x.z * inv, x.w * inv));
    };

    Segment s_next;
    while (have) {
        const bool have_next = next_segment(cur, r1, seq_at, pl, s_next);
        if (have_next) load_q(s_next, qn);
        parts_of(pl, s);   // (before the pages, the first of which is still on its way; behind them everyone waits 0.6 us for it)
        const int qrow = row0[s.b];
        // The token's new row: it belongs in slot (L - 1) mod 16 of the sequence's last page.  The warp that owns
        // that page fetches the row (lanes 0..15: K, lanes 16..31: V, 16 bytes each), stores it to the pool and
        // patches it into the tiles when they arrive.
        const int seg_pages = s.pg1 - s.pg0;
        const int last_pg = (s.L - 1) / kPage, new_slot = (s.L - 1) % kPage;
        bool patch = false;
        uint4 new_row = make_uint4(0, 0, 0, 0);   // bf16 cache: 16 bytes of the row; code caches: the codes (x, and y for E4M3)
        float new_scale = 0.f;   // 4-bit cache: the scale of the new K row (lanes 0..15) / V row (lanes 16..31)
        if constexpr (APPEND) {
            patch = last_pg >= s.pg0 && last_pg < s.pg1 && ((last_pg - s.pg0) % kCW) == warp;
            if (patch) {
                const char *src = (lane < 16 ? a.k_new : a.v_new) + ((size_t)qrow * Hkv + s.kvh) * kD * 2 + (lane & 15) * 16;
                const bool in_row = (lane & 15) < kD / 8;
                if (in_row) new_row = __ldg(reinterpret_cast<const uint4 *>(src));
                const int pid = a.block_table[(size_t)s.b * a.max_pages + last_pg];
                const bool store = (unsigned)pid < (unsigned)a.num_pages && ARB_IN_RANGE(a.status, qrow, a.rows);
                // (a page outside the pool: the producer has raised ARB_DEV_BAD_PAGE; nothing is written)
                if constexpr (I4) {
                    // The row's scale is max|x| / 7 over its 128 values (16 lanes), the codes rint(x * (7 / max|x|))
                    // clamped to -7 .. 7, both divisions IEEE; this lane's eight values are one word of nibbles
                    // (code + 8; nibbles 0..7 = dimensions 0, 2, 4, 6, 1, 3, 5, 7 of the eight).
                    const uint32_t w[4] = {new_row.x, new_row.y, new_row.z, new_row.w};
                    float x[8];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        x[2 * j] = __uint_as_float(w[j] << 16);
                        x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
                    }
                    float m = 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(x[j]));
#pragma unroll
                    for (int off = 8; off >= 1; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
                    new_scale = m > 0.f ? __fdiv_rn(m, 7.f) : 0.f;
                    const float inv = m > 0.f ? __fdiv_rn(7.f, m) : 0.f;
                    uint32_t word = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int c = max(-7, min(7, __float2int_rn(__fmul_rn(x[j], inv))));
                        word |= (uint32_t)(c + 8) << (4 * ((j >> 1) + 4 * (j & 1)));
                    }
                    if (store) {
                        const size_t slot_row = ((size_t)pid * Hkv + s.kvh) * kPage + new_slot;
                        *reinterpret_cast<uint32_t *>((lane < 16 ? a.k_pool : a.v_pool) + slot_row * (kD / 2) + (lane & 15) * 4) = word;
                        if ((lane & 15) == 0) (lane < 16 ? a.k_scales : a.v_scales)[slot_row] = new_scale;
                    }
                    new_row.x = word;
                } else if constexpr (E4M3) {
                    // quantise this lane's eight values as arb_kv_append_e4m3 does (x * inv_scale in fp32, nearest code,
                    // ties to even, saturating), store the codes, and keep them for the tile
                    const float inv = lane < 16 ? a.k_inv_scale : a.v_inv_scale;
                    const uint32_t w[4] = {new_row.x, new_row.y, new_row.z, new_row.w};
                    uint32_t code[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        code[j] = e4m3x2_from_f32(__uint_as_float(w[j] << 16) * inv, __uint_as_float(w[j] & 0xffff0000u) * inv);
                    if (store) {
                        char *dst = (lane < 16 ? a.k_pool : a.v_pool) +
                                    (((size_t)pid * Hkv + s.kvh) * kPage + new_slot) * kD + (lane & 15) * 8;
                        *reinterpret_cast<uint2 *>(dst) = make_uint2(code[0] | (code[1] << 16), code[2] | (code[3] << 16));
                    }
                    new_row.x = code[0] | (code[1] << 16);
                    new_row.y = code[2] | (code[3] << 16);
                } else if (store && in_row) {
                    char *dst = (lane < 16 ? a.k_pool : a.v_pool) +
                                (((size_t)pid * Hkv + s.kvh) * kPage + new_slot) * (kD * 2) + (lane & 15) * 16;
                    *reinterpret_cast<uint4 *>(dst) = new_row;
                }
            }
        }

        // this lane's columns (heads h0, h1): running max (the same in the 8 lanes of a column pair), its share of
        // the sum, and the m-tiles of O^T: o[mt][0..1] = dim 16 mt + gq of heads h0, h1; o[mt][2..3] = dim + 8
        float m_run0 = -INFINITY, m_run1 = -INFINITY, l_run0 = 0.f, l_run1 = 0.f;
        float o[kD / 16][4];
#pragma unroll
        for (int mt = 0; mt < kD / 16; ++mt) { o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f; }

        for (int gi = warp; gi < seg_pages; gi += kCW) {
            const int pg = s.pg0 + gi;
            const int ntok = min(s.L - pg * kPage, kPage);
            const bool patch_here = APPEND && patch && pg == last_pg;
            const uint32_t ck = seg_base + 2u * (uint32_t)gi;

            // ---- S^T = K q^T: 16 keys x 8 heads, two accumulators so that the chain is four deep ----------
            float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};
            float ksc0 = 1.f, ksc1 = 1.f, vsc0 = 1.f, vsc1 = 1.f;   // 4-bit cache: the scales of keys gq and gq + 8
            {
                const uint32_t st = ck % STAGES, par = (ck / STAGES) & 1u;
                mbar_wait(&tail->full[st], par, abort, a.status);
                char *tile_p = ring + st * kStageBytes;
                if constexpr (CODES) {   // the codes come into registers; the ring stage is free at once
                    uint32_t row0_w[kRowWords], row1_w[kRowWords];
#pragma unroll
                    for (int c = 0; c < kRowWords / 4; ++c) {
                        const int at = E4M3 ? (((2 * tq + c) ^ (gq & 7)) << 4) : tq * 16;   // (rows gq and gq + 8: same swizzle)
                        const char *src = tile_p + gq * (E4M3 ? 128 : 64) + at;
                        const uint4 x = *reinterpret_cast<const uint4 *>(src);
                        const uint4 y = *reinterpret_cast<const uint4 *>(src + 8 * (E4M3 ? 128 : 64));
                        row0_w[4 * c] = x.x; row0_w[4 * c + 1] = x.y; row0_w[4 * c + 2] = x.z; row0_w[4 * c + 3] = x.w;
                        row1_w[4 * c] = y.x; row1_w[4 * c + 1] = y.y; row1_w[4 * c + 2] = y.z; row1_w[4 * c + 3] = y.w;
                    }
                    if constexpr (I4) {
                        const float *sc = reinterpret_cast<const float *>(tile_p + kI4CodeBytes);
                        ksc0 = sc[gq];
                        ksc1 = sc[gq + 8];
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tail->empty[st]);
                    if (patch_here) {   // lanes 0..15 hold the new K row, dimensions 8 lane ..
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t x = __shfl_sync(0xffffffffu, new_row.x, 4 * tq + j);
                            const uint32_t y = E4M3 ? __shfl_sync(0xffffffffu, new_row.y, 4 * tq + j) : 0u;
                            const int w = E4M3 ? 2 * j : j;
                            if (gq == new_slot) { row0_w[w] = x; if (E4M3) row0_w[w + 1] = y; }
                            if (gq + 8 == new_slot) { row1_w[w] = x; if (E4M3) row1_w[w + 1] = y; }
                        }
                        if constexpr (I4) {
                            const float ns = __shfl_sync(0xffffffffu, new_scale, 0);
                            if (gq == new_slot) ksc0 = ns;
                            if (gq + 8 == new_slot) ksc1 = ns;
                        }
                    }
#pragma unroll
                    for (int ks = 0; ks < kD / 16; ++ks) {
                        uint32_t af[4];
                        k_fragment<E4M3>(row0_w, ks, af[0], af[2]);
                        k_fragment<E4M3>(row1_w, ks, af[1], af[3]);
                        if (ks & 1) mma_16816<E4M3>(sb, af, qb[ks][0], qb[ks][1]);
                        else mma_16816<E4M3>(sa, af, qb[ks][0], qb[ks][1]);
                    }
                } else {
                    if (patch_here) {
                        if (lane < kD / 8) *reinterpret_cast<uint4 *>(tile_p + tile_off(new_slot, lane)) = new_row;
                        __syncwarp();
                    }
                    const uint32_t tile = smem_u32(tile_p);
#pragma unroll
                    for (int ks = 0; ks < kD / 16; ++ks) {
                        uint32_t af[4];   // rows: keys; matrices: (keys 0-7 | 8-15) x (dims 16 ks + 0-7 | 8-15)
                        ldmatrix_x4(tile + tile_off((lane & 7) + ((lane >> 3) & 1) * 8, 2 * ks + (lane >> 4)), af);
                        if (ks & 1) mma_16816<E4M3>(sb, af, qb[ks][0], qb[ks][1]);
                        else mma_16816<E4M3>(sa, af, qb[ks][0], qb[ks][1]);
                    }
                    __syncwarp();
                    if (patch_here) fence_proxy_async_smem();   // the stage's next writer is the TMA unit
                    if (lane == 0) mbar_arrive(&tail->empty[st]);
                }
            }
            if constexpr (I4) {   // a key is scale * code: the scores of keys gq and gq + 8 take their rows' scales
                sa[0] *= ksc0; sa[1] *= ksc0; sb[0] *= ksc0; sb[1] *= ksc0;
                sa[2] *= ksc1; sa[3] *= ksc1; sb[2] *= ksc1; sb[3] *= ksc1;
            }

            // ---- online softmax: this lane has keys gq and gq + 8 of heads h0 and h1 -------------------
            const bool k0 = gq < ntok, k1 = gq + 8 < ntok;
            const float s00 = k0 ? (sa[0] + sb[0]) * a.scale_log2 : -INFINITY;
            const float s01 = k0 ? (sa[1] + sb[1]) * a.scale_log2 : -INFINITY;
            const float s10 = k1 ? (sa[2] + sb[2]) * a.scale_log2 : -INFINITY;
            const float s11 = k1 ? (sa[3] + sb[3]) * a.scale_log2 : -INFINITY;
            float mx0 = fmaxf(s00, s10), mx1 = fmaxf(s01, s11);
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) {
                mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
                mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
            }
            const float mn0 = fmaxf(m_run0, mx0), mn1 = fmaxf(m_run1, mx1);   // finite: key 0 of the page is visible
            const float f0 = fast_exp2(m_run0 - mn0), f1 = fast_exp2(m_run1 - mn1);   // 0 on the first page
            m_run0 = mn0;
            m_run1 = mn1;
            // P^T, rounded to bf16 (f16 over an E4M3 cache); the sums use the rounded weights, like the tensor core
            const float p00 = fast_exp2(s00 - mn0), p01 = fast_exp2(s01 - mn1);
            const float p10 = fast_exp2(s10 - mn0), p11 = fast_exp2(s11 - mn1);
            uint32_t w0 = E4M3 ? pack_f16(p00, p01) : pack_bf16(p00, p01);   // key gq:     heads h0, h1
            uint32_t w1 = E4M3 ? pack_f16(p10, p11) : pack_bf16(p10, p11);   // key gq + 8
            if constexpr (I4 || SPLIT_P) {   // (4-bit: the weights that reach the tensor core carry the value scales, packed below)
                l_run0 = fmaf(l_run0, f0, p00 + p10);
                l_run1 = fmaf(l_run1, f1, p01 + p11);
            } else if constexpr (E4M3) {
                const float2 r0 = unpack_f16(w0), r1 = unpack_f16(w1);
                l_run0 = fmaf(l_run0, f0, r0.x + r1.x);
                l_run1 = fmaf(l_run1, f1, r0.y + r1.y);
            } else {
                l_run0 = fmaf(l_run0, f0, __uint_as_float(w0 << 16) + __uint_as_float(w1 << 16));
                l_run1 = fmaf(l_run1, f1, __uint_as_float(w0 & 0xffff0000u) + __uint_as_float(w1 & 0xffff0000u));
            }
            // B fragment of P^T (16 keys x 8 heads): keys 2 tq, + 1 (and + 8) of head gq
            uint32_t pb0 = 0, pb1 = 0, lb0 = 0, lb1 = 0;
            if constexpr (!I4) {
                pb0 = movmatrix_trans(w0);
                pb1 = movmatrix_trans(w1);
            }
            if constexpr (SPLIT_P) {   // what the rounding to bf16 left over
                lb0 = movmatrix_trans(pack_bf16(p00 - __uint_as_float(w0 << 16), p01 - __uint_as_float(w0 & 0xffff0000u)));
                lb1 = movmatrix_trans(pack_bf16(p10 - __uint_as_float(w1 << 16), p11 - __uint_as_float(w1 & 0xffff0000u)));
            }
            if (__any_sync(0xffffffffu, f0 != 1.0f || f1 != 1.0f)) {
#pragma unroll
                for (int mt = 0; mt < kD / 16; ++mt) { o[mt][0] *= f0; o[mt][1] *= f1; o[mt][2] *= f0; o[mt][3] *= f1; }
            }

            // ---- O^T += V^T P^T: m-tiles of 16 dims ---------------------------------------------------
            {
                const uint32_t cv = ck + 1u, st = cv % STAGES, par = (cv / STAGES) & 1u;
                mbar_wait(&tail->full[st], par, abort, a.status);
                char *tile_p = ring + st * kStageBytes;
                if constexpr (CODES) {
                    constexpr int kVWords = kRowWords / 2;   // of this lane's 16 dimensions
                    const int key[4] = {2 * tq, 2 * tq + 1, 2 * tq + 8, 2 * tq + 9};
                    uint32_t vw[4][kVWords];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if constexpr (E4M3) {
                            const uint4 x = *reinterpret_cast<const uint4 *>(tile_p + key[j] * 128 + ((gq ^ (key[j] & 7)) << 4));
                            vw[j][0] = x.x; vw[j][1] = x.y; vw[j][2] = x.z; vw[j][3] = x.w;
                        } else {
                            const uint2 x = *reinterpret_cast<const uint2 *>(tile_p + key[j] * 64 + gq * 8);
                            vw[j][0] = x.x; vw[j][1] = x.y;
                        }
                    }
                    if constexpr (I4) {
                        const float *sc = reinterpret_cast<const float *>(tile_p + kI4CodeBytes);
                        vsc0 = k0 ? sc[gq] : 0.f;        // (the scale of a slot past the sequence end may be anything)
                        vsc1 = k1 ? sc[gq + 8] : 0.f;
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tail->empty[st]);
                    if (patch_here) {   // lanes 16..31 hold the new V row, dimensions 8 (lane - 16) ..
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const uint32_t x = __shfl_sync(0xffffffffu, new_row.x, 16 + 2 * gq + j);
                            const uint32_t y = E4M3 ? __shfl_sync(0xffffffffu, new_row.y, 16 + 2 * gq + j) : 0u;
                            const int w = E4M3 ? 2 * j : j;
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (key[i] == new_slot) { vw[i][w] = x; if (E4M3) vw[i][w + 1] = y; }
                        }
                        if constexpr (I4) {
                            const float ns = __shfl_sync(0xffffffffu, new_scale, 16);
                            if (gq == new_slot) vsc0 = ns;
                            if (gq + 8 == new_slot) vsc1 = ns;
                        }
                    }
                    if constexpr (I4) {   // a value is scale * code: the weight of a key takes its row's scale
                        w0 = pack_bf16(p00 * vsc0, p01 * vsc0);
                        w1 = pack_bf16(p10 * vsc1, p11 * vsc1);
                        pb0 = movmatrix_trans(w0);
                        pb1 = movmatrix_trans(w1);
                    } else if (ntok < kPage) {   // codes past the sequence end may be NaN: not even times zero
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (key[j] >= ntok) {
#pragma unroll
                                for (int w = 0; w < kVWords; ++w) vw[j][w] = 0u;
                            }
                    }
#pragma unroll
                    for (int mt = 0; mt < kD / 16; ++mt) {
                        uint32_t af[4];
                        v_fragment<E4M3>(vw[0], vw[1], mt, af[0], af[1]);
                        v_fragment<E4M3>(vw[2], vw[3], mt, af[2], af[3]);
                        mma_16816<E4M3>(o[mt], af, pb0, pb1);
                    }
                } else {
                    if (patch_here) {
                        if (lane >= 16 && lane - 16 < kD / 8)
                            *reinterpret_cast<uint4 *>(tile_p + tile_off(new_slot, lane - 16)) = new_row;
                        __syncwarp();
                    }
                    if (ntok < kPage) {
                        // slots past the sequence end may hold anything; they must not reach the tensor core, not even
                        // times zero: blank them in shared memory
                        for (int i = lane; i < (kPage - ntok) * (kD / 8); i += 32)
                            *reinterpret_cast<uint4 *>(tile_p + tile_off(ntok + i / (kD / 8), i % (kD / 8))) = make_uint4(0, 0, 0, 0);
                        __syncwarp();
                    }
                    const uint32_t tile = smem_u32(tile_p);
#pragma unroll
                    for (int mt = 0; mt < kD / 16; ++mt) {
                        uint32_t af[4];   // transposed on the way: rows dims (16 mt + 0-7 | 8-15), columns keys (0-7 | 8-15)
                        ldmatrix_x4_trans(tile + tile_off((lane & 7) + (lane >> 4) * 8, 2 * mt + ((lane >> 3) & 1)), af);
                        mma_16816<E4M3>(o[mt], af, pb0, pb1);
                        if constexpr (SPLIT_P) mma_16816<false>(o[mt], af, lb0, lb1);
                    }
                    __syncwarp();
                    if (patch_here || ntok < kPage) fence_proxy_async_smem();
                    if (lane == 0) mbar_arrive(&tail->empty[st]);
                }
            }
        }
        seg_base += 2u * (uint32_t)seg_pages;

        // ---- segment end: every warp leaves (max, sum, accumulators); all consumer threads merge them ----
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            l_run0 += __shfl_xor_sync(0xffffffffu, l_run0, off);
            l_run1 += __shfl_xor_sync(0xffffffffu, l_run1, off);
        }
        float *rec = osm + warp * WREC;
        if (gq == 0) {
            rec[h0] = m_run0; rec[h1] = m_run1;
            rec[8 + h0] = l_run0; rec[8 + h1] = l_run1;
        }
#pragma unroll
        for (int mt = 0; mt < kD / 16; ++mt) {
            if constexpr (CODES) {   // dimensions 16 gq + 2 mt and + 1
                const int d = 16 * gq + 2 * mt;
                if (h0 < G) *reinterpret_cast<float2 *>(rec + 16 + h0 * kOStride + d) = make_float2(o[mt][0], o[mt][2]);
                if (h1 < G) *reinterpret_cast<float2 *>(rec + 16 + h1 * kOStride + d) = make_float2(o[mt][1], o[mt][3]);
                continue;
            }
            const int d = 16 * mt + gq;
            if (h0 < G) { rec[16 + h0 * kOStride + d] = o[mt][0]; rec[16 + h0 * kOStride + d + 8] = o[mt][2]; }
            if (h1 < G) { rec[16 + h1 * kOStride + d] = o[mt][1]; rec[16 + h1 * kOStride + d + 8] = o[mt][3]; }
        }
        named_barrier(kBarConsumers, kCT);
        // A whole item goes to `out`, a part of a split one to the workspace, from the registers the merge leaves it in.
        const size_t out_base = ((size_t)qrow * a.Hq + s.kvh * G) * kD;
        const int part = cta - s.c_first;   // (of s.nparts)
        const bool last = part == s.nparts - 1 && !pl.mergers;   // of the item, and merged here
        const bool gathers = s.nparts > 1 && (last || (s.nparts > kDirectParts && part % kMergeFan == kMergeFan - 1));
        if (tid < VECS) {
            float M = -INFINITY, mw[kCW];
#pragma unroll
            for (int w = 0; w < kCW; ++w) { mw[w] = osm[w * WREC + eh]; M = fmaxf(M, mw[w]); }
            float l = 0.f;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < kCW; ++w) {
                const float ff = fast_exp2(mw[w] - M);   // 0 for a warp that had no page
                const float4 v = *reinterpret_cast<const float4 *>(osm + w * WREC + 16 + eh * kOStride + (tid % (kD / 4)) * 4);
                l = fmaf(ff, osm[w * WREC + 8 + eh], l);
                x.x = fmaf(ff, v.x, x.x); x.y = fmaf(ff, v.y, x.y); x.z = fmaf(ff, v.z, x.z); x.w = fmaf(ff, v.w, x.w);
            }
            if constexpr (E4M3) { x.x *= a.v_scale; x.y *= a.v_scale; x.z *= a.v_scale; x.w *= a.v_scale; }   // values are v_scale * code
            if (s.nparts == 1) {
                write_row(out_base, x, 1.0f / l);
            } else if (gathers) {
                own = x;
                own_m = M;
                own_l = l;
            } else {
                publish(x, M, l, part);
            }
        }
        if (gathers) {
            gather_first = s.c_first;
            gather_part = part;
            in_runs = s.nparts > kDirectParts;
            gather_last = last;
            gather_out = out_base;
        }
        if (have_next) named_barrier(kBarConsumers, kCT);   // warp records are free for the next segment
        s = s_next;
        have = have_next;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) { qb[ks][0] = qn[ks][0]; qb[ks][1] = qn[ks][1]; }
    }
    if (merges_only) {   // the item this CTA is for: number cta - stream of those that take part
        const int item = cta - pl.stream;
        int b = 0;
        while (b + 1 < B && act[b + 1] * Hkv <= item) ++b;
        s.b = b;
        s.kvh = item - act[b] * Hkv;
        parts_of(pl, s);
        if (s.nparts > 1) {
            gather_first = s.c_first;
            gather_part = s.nparts;
            in_runs = s.nparts > kDirectParts;
            gather_last = true;
            gather_out = ((size_t)row0[b] * a.Hq + s.kvh * G) * kD;
        }
    }
    if (gather_first < 0 || warp * 32 >= VECS) return;

    // ---- the merge of a split (sequence, kv head) ---------------------------------------------------------
    //     m = max_p m_p,  w_p = 2^(m_p - m),  out = sum_p w_p o_p / sum_p w_p l_p,
    // one 4-dimension piece of the group's outputs per thread.  Read are the parts of this CTA's own run, as they
    // are, and of every run before it the slot of its last part, which holds the run's sum; kMergeBatch of them at a time, in a
    // fixed order whenever they come.  Lane p of a head's lanes has the (max, sum) of part p of a batch.
    const int run0 = in_runs ? gather_part / kMergeFan * kMergeFan : 0;        // first part of the own run
    const int runs = in_runs && gather_last ? gather_part / kMergeFan : 0;     // sums to read besides
    const int n = runs + gather_part - run0;
    const bool mine = tid < VECS;
    const int piece = mine ? tid : 0;
    auto merge = [&](int p0, auto batch) {
        constexpr int kBatch = decltype(batch)::value;
        const int np = min(kBatch, n - p0);
        auto slot_of = [&](int i) -> int {   // of the i-th part to read; always an earlier CTA's
            const int at = gather_first + (i < runs ? i * kMergeFan + kMergeFan - 1 : run0 + i - runs);
            return 2 * (ARB_IN_RANGE(a.status, at, cta) ? at : 0) + (at == gather_first);
        };
        float4 v[kBatch];
        float2 ml = make_float2(-INFINITY, 0.f);
        const bool has_ml = mine && lane % kLph < np;
        float2 *ml_at = reinterpret_cast<float2 *>(a.part_ml) + (size_t)slot_of(has_ml ? p0 + lane % kLph : p0) * kMaxGroup + piece / kLph;
        float4 *o_at = reinterpret_cast<float4 *>(a.part_o) + piece;
        unsigned missing = mine ? (1u << np) - 1u : 0u;
        bool ml_missing = has_ml;
        long long t0 = 0;
#pragma unroll
        for (int p = 0; p < kBatch; ++p) v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        while (true) {
            const unsigned before = missing;
            if (ml_missing) ml = load_slot2(ml_at);
#pragma unroll
            for (int p = 0; p < kBatch; ++p)
                if (missing >> p & 1u) v[p] = load_slot4(o_at + (size_t)slot_of(p0 + p) * VECS);
            ml_missing = ml_missing && (is_empty(ml.x) || is_empty(ml.y));
#pragma unroll
            for (int p = 0; p < kBatch; ++p)
                if ((missing >> p & 1u) && !any_empty(v[p])) missing &= ~(1u << p);
            if (!__any_sync(0xffffffffu, ml_missing || missing != 0u)) break;
            if (__all_sync(0xffffffffu, missing == before)) __nanosleep(merges_only ? 200 : 100);
            if (t0 == 0) t0 = clock64();
            if (*abort || clock64() - t0 > kWaitCycles) {   // give up, like every other wait
                if (!*abort) {
                    *abort = 1;
                    atomicOr(a.status, (uint32_t)ARB_DEV_WAIT_TIMEOUT);
                }
                break;
            }
        }
        __syncwarp();
        // read: empty again for the next call
        const float e = __uint_as_float(kEmpty);
        if (has_ml) store_slot2(ml_at, make_float2(e, e));
#pragma unroll
        for (int p = 0; p < kBatch; ++p)
            if (mine && p < np) store_slot4(o_at + (size_t)slot_of(p0 + p) * VECS, make_float4(e, e, e, e));
        float mb = fmaxf(own_m, ml.x);
#pragma unroll
        for (int off = 1; off < kLph; off <<= 1) mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, off));
        const float f = fast_exp2(own_m - mb), w = fast_exp2(ml.x - mb);
        float l = w * ml.y;
#pragma unroll
        for (int off = 1; off < kLph; off <<= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        own_m = mb;
        own_l = fmaf(own_l, f, l);
        own.x *= f; own.y *= f; own.z *= f; own.w *= f;
#pragma unroll
        for (int p = 0; p < kBatch; ++p) {
            const float wp = __shfl_sync(0xffffffffu, w, (lane / kLph) * kLph + p);   // 0 where the batch has no part p
            own.x = fmaf(wp, v[p].x, own.x); own.y = fmaf(wp, v[p].y, own.y); own.z = fmaf(wp, v[p].z, own.z); own.w = fmaf(wp, v[p].w, own.w);
        }
    };
    // 148 CTAs over 8 items are 18 and a half parts each: a round of twenty instead of two of sixteen
    if (kLongBatch <= kLph && n > kMergeBatch && n <= kLongBatch) merge(0, std::integral_constant<int, kLongBatch <= kLph ? kLongBatch : kMergeBatch>());
    else
        for (int p0 = 0; p0 < n; p0 += kMergeBatch) merge(p0, std::integral_constant<int, kMergeBatch>());
    if (!mine) return;
    if (gather_last) write_row(gather_out, own, 1.0f / own_l);
    else publish(own, own_m, own_l, gather_part);
}

// Ring depth: 32 stages, 128 KB of tiles in flight per SM with one CTA per SM.  A 16-stage ring with room for two
// CTAs per SM (so that the next kernel of a chain is resident before this one ends) was measured and is slower on
// every workload: a lone call is bound by bytes in flight, and the successor's CTAs come up SM by SM as this
// kernel's CTAs leave anyway.
// Ring stages.  What is in flight per SM is stages x bytes of a stage, and it has to cover latency x bandwidth: 32 tiles
// of a bf16 cache are 128 KB; the tiles of the code caches are 2 KB and 1.1 KB, so their rings are deeper (with 32
// stages a large call over 4-bit codes could keep 16 KB per SM in flight: 1.4 TB/s).  Tiles of 64-dimension heads are 2 KB: 64 stages keep the same 128 KB in flight.
template <int KV, int HD>
constexpr int stages_of() { return KV == kKvBf16 ? (HD == 64 ? 64 : 32) : KV == kKvE4m3 ? 64 : 128; }

template <int G, bool APPEND, int KV, int HD = 128>
arb_status launch_variant(Ctx *ctx, const StepArgs &a, const CUtensorMap &km, const CUtensorMap &vm, cudaStream_t stream) {
    constexpr int STAGES = stages_of<KV, HD>();
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device & 63]) {
        if (cudaFuncSetAttribute(decode_step_kernel<G, STAGES, APPEND, KV, HD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem_bytes<G, STAGES, KV, HD>(kMaxBatch)) != cudaSuccess)
            return ARB_ERR_CUDA;
        attr_set[ctx->device & 63] = true;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctx->num_sms);
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = smem_bytes<G, STAGES, KV, HD>(a.batch);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, decode_step_kernel<G, STAGES, APPEND, KV, HD>, a, km, vm) != cudaSuccess) return ARB_ERR_CUDA;
    ctx->launches++;
    return ARB_OK;
}

// The 4-bit form exists with the cache write only.
template <int G>
arb_status launch_g(Ctx *ctx, const StepArgs &a, int kv, int head_dim, const CUtensorMap &km, const CUtensorMap &vm,
                    cudaStream_t stream) {
    if (kv == kKvE4m3)
        return a.k_new != nullptr ? launch_variant<G, true, kKvE4m3>(ctx, a, km, vm, stream)
                                  : launch_variant<G, false, kKvE4m3>(ctx, a, km, vm, stream);
    if (kv == kKvI4) return launch_variant<G, true, kKvI4>(ctx, a, km, vm, stream);
    if (head_dim == 64)
        return a.k_new != nullptr ? launch_variant<G, true, kKvBf16, 64>(ctx, a, km, vm, stream)
                                  : launch_variant<G, false, kKvBf16, 64>(ctx, a, km, vm, stream);
    return a.k_new != nullptr ? launch_variant<G, true, kKvBf16>(ctx, a, km, vm, stream)
                              : launch_variant<G, false, kKvBf16>(ctx, a, km, vm, stream);
}

}  // namespace

// every word kEmpty between calls: memset to 0xff
size_t decode_step_slot_bytes(int num_sms) { return sizeof(float) * 2 * (size_t)num_sms * kMaxGroup * (kD + 2); }

bool decode_step_supported(const arb_attn_params &p) {
    const int g = p.num_q_heads / p.num_kv_heads;
    return p.dtype == ARB_BF16 && (p.head_dim == 64 || p.head_dim == 128) && g >= 1 && g <= 8 && tma_available();
}

// k_new == nullptr: attention only (seq_lens is not written).  scales != nullptr: an E4M3 cache with scales =
// {k_scale, v_scale, k_inv_scale, v_inv_scale}; k_row_scales != nullptr: a 4-bit cache with its two scale pools
// (k_new is required); neither: a bf16 cache.
// beside: the decode rows of a call that has chunks too.  The chunk kernel, launched next, reads and writes nothing that this
// one does, so it starts as soon as this kernel's predecessor is known to have completed, and this one takes only its share
// of the SMs (kBesideWeight).
arb_status launch_decode_step(Ctx *ctx, const arb_attn_params &p, const void *q, const void *k_new, const void *v_new,
                              void *k_pages, void *v_pages, const float *scales, const int32_t *block_table,
                              int32_t *seq_lens, const int32_t *q_lens, void *out, cudaStream_t stream, bool beside,
                              float *k_row_scales, float *v_row_scales) {
    alignas(64) CUtensorMap km, vm;
    const bool e4m3 = scales != nullptr, i4 = k_row_scales != nullptr;
    if (i4 && k_new == nullptr) return ARB_ERR_INVALID_ARG;
    if (e4m3 && i4) return ARB_ERR_INVALID_ARG;
    bool whole_rows = false;
    if (i4) {
        if (!pool_map(ctx, &km, k_pages, p.num_pages, p.num_kv_heads, PoolView::kI4) ||
            !pool_map(ctx, &vm, v_pages, p.num_pages, p.num_kv_heads, PoolView::kI4))
            return ARB_ERR_CUDA;
    } else if (e4m3) {
        if (!pool_map(ctx, &km, k_pages, p.num_pages, p.num_kv_heads, PoolView::kE4m3) ||
            !pool_map(ctx, &vm, v_pages, p.num_pages, p.num_kv_heads, PoolView::kE4m3))
            return ARB_ERR_CUDA;
    } else if (p.head_dim == 64) {
        if (!pool_map(ctx, &km, k_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16D64) ||
            !pool_map(ctx, &vm, v_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16D64))
            return ARB_ERR_CUDA;
    } else {
        whole_rows = pool_map(ctx, &km, k_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16WholeRows) &&
                     pool_map(ctx, &vm, v_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16WholeRows);
        if (!whole_rows && (!pool_map(ctx, &km, k_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16HalfRows) ||
                            !pool_map(ctx, &vm, v_pages, p.num_pages, p.num_kv_heads, PoolView::kBf16HalfRows)))
            return ARB_ERR_CUDA;
    }
    const int g = p.num_q_heads / p.num_kv_heads;
    StepArgs a;
    a.q = static_cast<const char *>(q);
    a.k_new = static_cast<const char *>(k_new);
    a.v_new = static_cast<const char *>(v_new);
    a.k_pool = static_cast<char *>(k_pages);
    a.v_pool = static_cast<char *>(v_pages);
    a.block_table = block_table;
    a.seq_lens = seq_lens;
    a.q_lens = q_lens;
    a.out = static_cast<char *>(out);
    a.part_o = ctx->step_slots;
    a.part_ml = a.part_o + 2 * (size_t)ctx->num_sms * kMaxGroup * kD;
    a.ticket = reinterpret_cast<unsigned *>(ctx->rot + (size_t)kRotSets * kRotCounters + kRotSets + 5);
    a.lens_counter = ctx->rot + (size_t)kRotSets * kRotCounters + kRotSets + 4;
    // (Beside chunks an append that moved the lengths is what precedes the call: its guess would always be wrong.  And a guessed
    // length is at most what the table holds: its pages must be countable.)
    a.guess = !beside && (long long)p.batch * p.num_kv_heads * p.max_pages_per_seq < (1ll << 30) ? 1 : 0;
    a.status = ctx->status;
    a.batch = p.batch;
    a.beside = beside ? 1 : 0;
    a.Hq = p.num_q_heads;
    a.Hkv = p.num_kv_heads;
    a.num_pages = p.num_pages;
    a.max_pages = p.max_pages_per_seq;
    a.whole_rows = whole_rows ? 1 : 0;
    a.rows = p.total_q;
    a.boundary_pct = ctx->step_boundary_pct;
    a.min_chunk = ctx->step_min_chunk;
    const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 1.0f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * (e4m3 ? scales[0] : 1.0f) * 1.4426950408889634f;
    a.v_scale = e4m3 ? scales[1] : 1.0f;
    a.k_inv_scale = e4m3 ? scales[2] : 1.0f;
    a.v_inv_scale = e4m3 ? scales[3] : 1.0f;
    a.k_scales = k_row_scales;
    a.v_scales = v_row_scales;
    const int kv = i4 ? kKvI4 : e4m3 ? kKvE4m3 : kKvBf16;
    switch (g) {
        case 1: return launch_g<1>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 2: return launch_g<2>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 3: return launch_g<3>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 4: return launch_g<4>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 5: return launch_g<5>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 6: return launch_g<6>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 7: return launch_g<7>(ctx, a, kv, p.head_dim, km, vm, stream);
        case 8: return launch_g<8>(ctx, a, kv, p.head_dim, km, vm, stream);
        default: return ARB_ERR_UNSUPPORTED;
    }
}

}  // namespace arb
