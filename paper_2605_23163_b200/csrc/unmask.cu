// Confidence-threshold parallel unmasking: vocabulary-wide soft-max statistics and
// (Gumbel-perturbed) arg-max per MASKED row, then the per-rollout commit rule.
//
// Kernel 1 (unmask_stream_kernel): persistent grid, every warp on its own.  The MASKED rows of the
// call, cut into tiles of 2048 ids, are split into pieces of a few tiles: one piece per warp when there are few rows,
// else equal ranges or pieces that the warps draw from a counter (one record per piece, merged by the
// second kernel).  A warp streams its tiles from HBM once, through a ring of bulk asynchronous
// copies (cp.async.bulk, completion on an mbarrier, no multicast) into its own part of shared
// memory, three tiles deep; a lane takes 64 consecutive ids of a tile (16-byte reads, chunk order
// rotated by the lane so that the banks do not collide) and keeps running soft-max statistics.
// There is no CTA-wide barrier after the set-up, and nothing but the few logits that can win the
// arg-max is looked at twice.  Rows that are not MASKED are not read (ragged rows: but for the bytes that share a
// 16-byte granule with a row that is).
//
// Noise (temperature > 0).  The Gumbel draws are g = -ln(E) with E an exponential race over groups
// of 16 consecutive ids: group j has the 32-bit word R = word j % 4 of Philox block j / 4 (so the 64
// ids of a lane share one block), which fixes the "leader" 16 j + R % 16 holding the group's
// smallest E = -ln(U) / 16, U = ((R >> 4) + (f + 0.5) 2^-23) / 2^28; every other id of the group has
// E = E_leader - ln((f + 0.5) 2^-23) with 23 fine bits f of its own (second Philox stream, one block
// per 4 ids).  The word alone bounds all 16 draws from above, g < 32 ln 2 - ln(2^28 - 1 - (R >> 4)),
// and the leader's draw from below, which is what makes the kernel cheap.  While a lane's 64 ids
// are in shared memory the streaming pass takes the largest of their four words and forms
//   an upper bound of every score of the block: its largest logit + T * (bound of that word), and
//   a lower bound of one score: the logit of that word's leader + T * (lower bound of its draw);
// the warp keeps the largest lower bound so far, L (also: the largest logit so far with the smallest
// draw there is), shares it with the warps that work on other pieces of the row (a word per row in global memory, read
// a tile ahead of its use), and notes the blocks whose upper bound reaches it in a short list in shared
// memory.  After the piece L is a lower bound of the row's best score, and only the noted blocks
// that still reach it (half a block per piece where each piece by itself had six) are read again, from L2, and scored
// exactly with the second stream.
// Any id left out cannot reach L, so the arg-max (lowest id on ties) is exact.
//
// What bounds it: a greedy launch over many rows streams at 0.9 of the measured HBM rate once it runs; with noise the
// 53 % busy issue slots and special-function units of four warps a scheduler (three CTAs an SM, with the registers
// cut to 80, were no faster).  Small launches are bound by latency: 1.6 us to the first copies, 0.7 to the first
// tile, 1.5 for a noisy tile, 1 for the look at the list.  Measured against equal ranges with a running maximum and
// re-scoring piece by piece, whole calls: 408 rows of 50257 bf16 logits, greedy, 28.8 -> 22.5-23.3 us; 720 rows of 151936
// fp32 logits with noise 90 -> 82-85; a draft / verify cycle over 176 rows of 151936 bf16 logits with noise 124.5 ->
// 106.7.
//
// Kernel 2 (unmask_finalize_kernel): one CTA per rollout merges the records of its rows, forms the
// confidences and applies the threshold / at-least-one rule.
#include "fdd_internal.h"
#include "tc_ptx.cuh"

#include <math_constants.h>

#include <atomic>

namespace {

constexpr int kWarps = 8;                             // per CTA; every warp works alone
constexpr int kThreads = kWarps * 32;
constexpr int kGroup = 16;                            // ids per group of the noise construction
constexpr int kLaneIds = 64;                          // consecutive ids a lane takes per tile: one Philox block of group words
constexpr int kTile = kUnmaskTile;                    // ids per tile (one bulk copy, one warp)
constexpr int kStages = 3;                            // tiles a warp holds in shared memory (two in flight while one is reduced)
constexpr int kMaxRows = kUnmaskMaxRows;              // rows of one launch (32 per thread in the set-up)
constexpr int kPiecePad = 1;                          // items that stand for what a piece costs beside its tiles
constexpr int kMinPiecesPerRow = 8;                   // a warp gets one piece when each row can have this many warps
constexpr int kDealtShare = 6, kDealtLeast = 3, kDealtMost = 12;   // short pieces that are dealt out: a sixth of a warp's share, of 3 to 12 tiles
constexpr int kMaxList = 224;                         // blocks in reach of the running lower bound kept per piece (a few dozen expected)
constexpr long long kCopyWaitLimit = 4000000000LL;    // SM clocks a warp waits for one of its own copies (about two seconds)
static_assert(kTile == 32 * kLaneIds, "a tile is 64 ids for each of 32 lanes");
static_assert(kMaxRows <= kThreads * 32, "the set-up gives every thread at most 32 rows");

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRefSlack = 4.0f;                     // a lane's sum stays relative to the same logit until one is larger by more than this
constexpr float kRefLeast = -2e38f;                   // ids masked with the type's lowest value: times log2(e) it has to stay finite
constexpr float kGumbelMin = -2.95f;                  // no draw is smaller: E <= 36 / 16 + 23 ln 2 + ln 2 < e^2.95

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;
constexpr uint32_t kFineStream = 0x80000000u;         // added to the position word for the fine bits

// Philox4x32 with 10 rounds (Salmon et al., SC'11), written from the published round function:
// (c0, c1, c2, c3) -> (hi(M1 c2) ^ c1 ^ k0, lo(M1 c2), hi(M0 c0) ^ c3 ^ k1, lo(M0 c0)), the key
// bumped by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k.x += kPhiloxW0; k.y += kPhiloxW1; }
        const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * c.x;
        const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * c.z;
        c = make_uint4(static_cast<uint32_t>(p1 >> 32) ^ c.y ^ k.x, static_cast<uint32_t>(p1),
                       static_cast<uint32_t>(p0 >> 32) ^ c.w ^ k.y, static_cast<uint32_t>(p0));
    }
    return c;
}
__device__ __forceinline__ uint32_t pick_word(const uint4& r, int k) {
    return k == 0 ? r.x : (k == 1 ? r.y : (k == 2 ? r.z : r.w));
}

// One bulk asynchronous copy global -> shared of this CTA; `bytes` and both addresses are multiples
// of 16.  Completion is counted in bytes on the mbarrier.
// The logits are read once: the copy marks their lines as the first to leave L2, so that a step's
// hundreds of MB do not push out what the attention kernel of the next step reads again (the
// shared prefix and the caches).
__device__ __forceinline__ uint64_t read_once_policy() {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy)
                 : "memory");
}

// Wait for one of the warp's own copies; false once the time limit has run out.
__device__ __forceinline__ bool wait_copy(uint32_t bar, uint32_t parity) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!tc::mbar_try_wait(bar, parity))
        if (clock64() - t0 > kCopyWaitLimit) return false;
    return true;
}
// Reductions over the warp in one instruction each.
__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xFFFFFFFF;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ int warp_min(int x) { return __reduce_min_sync(0xFFFFFFFFu, x); }
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, off);
    return x;
}
// Position of the (k + 1)-th set bit of mask (k < popc(mask)).
__device__ __forceinline__ int nth_set_bit(uint32_t mask, int k) {
    int at = 0;
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
        const int c = __popc(mask & ((1u << half) - 1u));
        if (k >= c) { k -= c; mask >>= half; at += half; }
    }
    return at;
}

// Words that the warps of a launch share, zero between launches: which piece is dealt out next, and for every row the
// largest lower bound of its best score that any of its pieces has found so far (floats in the order of unsigned
// numbers; 0 is below all of them and reads as NaN, which no maximum takes).
constexpr int kSharedNext = 0, kSharedBars = 32;
__device__ __forceinline__ uint32_t bar_key(float x) {
    const uint32_t b = __float_as_uint(x);
    return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float bar_value(uint32_t k) { return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xFFFFFFFFu)); }
__device__ __forceinline__ uint32_t load_shared_word(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

template <typename T> struct Logit;
template <> struct Logit<__nv_bfloat16> {
    static constexpr int kPerChunk = 8;                  // logits per 16-byte chunk
    __device__ static float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    __device__ static void widen(const uint4& w, float* out) {
        const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            out[2 * i] = __uint_as_float(x[i] << 16);
            out[2 * i + 1] = __uint_as_float(x[i] & 0xFFFF0000u);
        }
    }
    // the largest logit of N chunks (two logits per instruction, on the packed words)
    template <int N> __device__ static float largest(const uint4* w) {
        __nv_bfloat162 m[4];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t x[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&x[u]);
                m[u] = i == 0 ? v : __hmax2(m[u], v);
            }
        }
        const __nv_bfloat162 r = __hmax2(__hmax2(m[0], m[1]), __hmax2(m[2], m[3]));
        return fmaxf(__low2float(r), __high2float(r));
    }
    // the chunk `w` with its first ms elements taken from `n`
    __device__ static uint4 splice(const uint4& w, const uint4& n, int ms) {
        const uint32_t x[4] = {w.x, w.y, w.z, w.w}, y[4] = {n.x, n.y, n.z, n.w};
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t lo = 2 * i < ms ? y[i] : x[i], hi = 2 * i + 1 < ms ? y[i] : x[i];
            o[i] = (lo & 0xFFFFu) | (hi & 0xFFFF0000u);
        }
        return make_uint4(o[0], o[1], o[2], o[3]);
    }
};
template <> struct Logit<float> {
    static constexpr int kPerChunk = 4;
    __device__ static float load1(const float* p) { return *p; }
    __device__ static void widen(const uint4& w, float* out) {
        out[0] = __uint_as_float(w.x); out[1] = __uint_as_float(w.y);
        out[2] = __uint_as_float(w.z); out[3] = __uint_as_float(w.w);
    }
    template <int N> __device__ static float largest(const uint4* w) {
        float m[8];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int u = i % 8;
            const float a = __uint_as_float(w[i].x), b = __uint_as_float(w[i].y), c = __uint_as_float(w[i].z), d = __uint_as_float(w[i].w);
            m[u] = i < 8 ? tc::max3(a, b, fmaxf(c, d)) : tc::max3(tc::max3(m[u], a, b), c, d);
        }
        return tc::max3(tc::max3(m[0], m[1], m[2]), tc::max3(m[3], m[4], m[5]), fmaxf(m[6], m[7]));
    }
    __device__ static uint4 splice(const uint4& w, const uint4& n, int ms) {
        return make_uint4(0 < ms ? n.x : w.x, 1 < ms ? n.y : w.y, 2 < ms ? n.z : w.z, 3 < ms ? n.w : w.w);
    }
};

// 16 logits starting at vocabulary id v0 (a multiple of 16), from global memory; ids >= vocab read as -inf.
template <typename T>
__device__ __forceinline__ void load_group(const T* row_ptr, int v0, int vocab, int vec_ok, float* val) {
    if (vec_ok && v0 + kGroup <= vocab) {
        const uint4* p = reinterpret_cast<const uint4*>(row_ptr + v0);
#pragma unroll
        for (int c = 0; c < kGroup / Logit<T>::kPerChunk; ++c) Logit<T>::widen(p[c], val + c * Logit<T>::kPerChunk);
    } else {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) val[j] = (v0 + j < vocab) ? Logit<T>::load1(row_ptr + v0 + j) : -CUDART_INF_F;
    }
}

struct Best {
    float score, logit;
    int index;
};
__device__ __forceinline__ Best better(const Best& a, const Best& b) {
    // larger score wins; equal scores -> lower vocabulary id
    if (b.score > a.score || (b.score == a.score && b.index < a.index)) return b;
    return a;
}
__device__ __forceinline__ Best warp_best(const Best& b) {
    const float score = warp_max(b.score);
    const bool first = b.score == score;
    const int index = warp_min(first ? b.index : 0x7FFFFFFF);
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, first && b.index == index);
    return Best{score, __shfl_sync(0xFFFFFFFFu, b.logit, __ffs(who) - 1), index};
}

// ---- phase 2 of the noisy step: exact scores of the 16 ids of one group.
struct RowNoise {                                       // what fixes the draws of one row
    uint2 keys;                                         // the rollout's seed
    uint32_t pos, step, block_idx;
};
// Upper bound of every draw of a group from its word alone: U < (h + 1) / 2^28 = 1 - d / 2^28 with
// d = 2^28 - 1 - h, so -ln U > d / 2^28, E > d / 2^32 and g < 32 ln 2 - ln d (no bound for d = 0).
__device__ __forceinline__ float word_gumbel_bound(uint32_t R) {
    const uint32_t d = 0x0FFFFFFFu - (R >> 4);
    return d == 0u ? CUDART_INF_F : 22.18070977791825f - __logf(static_cast<float>(d)) + 1e-3f;
}
// Lower bound of the draw of a group's leader from its word alone: -ln U <= -ln(1 - y) <= y (1 + y) with y = (d + 1) / 2^28
// while y <= 1 / 2, so g >= 32 ln 2 - ln(d + 1) - ln(1 + y).
__device__ __forceinline__ float word_gumbel_least(uint32_t R) {
    const float d1 = static_cast<float>(0x10000000u - (R >> 4));
    const float y = d1 * 3.7252902984619140625e-09f;
    return y <= 0.5f ? 22.18070977791825f - __logf(d1) - y - 1e-3f : kGumbelMin;
}
// E of a group's leader, -ln(U) / 16 with U = (h + (f + 0.5) 2^-23) / 2^28, h = R >> 4, on the fast
// logarithm (absolute error 4e-7 on [0.5, 2], 3 ulp elsewhere).  In the upper half of the range the
// logarithm goes through y = 1 - U, which fp32 holds almost exactly there: a series below 2^-6, where
// the fast logarithm of a number next to 1 would lose the leading digits of -ln U.
__device__ __forceinline__ float leader_exponential(uint32_t R, uint32_t f23) {
    const uint32_t h = R >> 4;
    const float frac = (static_cast<float>(f23) + 0.5f) * 1.1920928955078125e-07f;
    float nl;                                               // -ln(U)
    if (h >= (1u << 27)) {
        const float y = (static_cast<float>((1u << 28) - h) - frac) * 3.7252902984619140625e-09f;   // 1 - U
        nl = y < 0.015625f ? y * fmaf(y, fmaf(y, fmaf(y, 0.25f, 0.33333334f), 0.5f), 1.0f) : -__logf(1.0f - y);
    } else {
        nl = 19.408121055678468f - __logf(static_cast<float>(h) + frac);                            // 28 ln 2 - ln(2^28 U)
    }
    return nl * 0.0625f;
}
// Four consecutive ids of group v0 (a multiple of 16): quad lane `part` takes ids v0 + 4 part ... + 3, with one Philox block
// for the group's word and one for its own fine bits; the leader's fine bits come from the quad lane that has them.
// E = E_leader for the leader, E_leader - ln((f + 0.5) 2^-23) for the others, g = -ln E.  Warp-wide (every lane calls).
template <typename T>
__device__ __forceinline__ Best score_quarter(const T* row_ptr, int v0, int part, bool act, float temperature, int vocab, const RowNoise& n) {
    const int v = v0 + 4 * part;
    float val[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) val[i] = act && v + i < vocab ? Logit<T>::load1(row_ptr + v + i) : -CUDART_INF_F;
    const int j = v0 >> 4;
    const uint32_t R = pick_word(philox4x32_10(make_uint4(static_cast<uint32_t>(j >> 2), n.pos, n.step, n.block_idx), n.keys), j & 3);
    const uint4 r = philox4x32_10(make_uint4(static_cast<uint32_t>(v >> 2), n.pos | kFineStream, n.step, n.block_idx), n.keys);
    const uint32_t f[4] = {r.x >> 9, r.y >> 9, r.z >> 9, r.w >> 9};
    const int li = static_cast<int>(R & 15u);
    const int k = li & 3;
    const uint32_t f_mine = k == 0 ? f[0] : (k == 1 ? f[1] : (k == 2 ? f[2] : f[3]));
    const uint32_t f_lead = __shfl_sync(0xFFFFFFFFu, f_mine, li >> 2, 4);
    const float e_lead = leader_exponential(R, f_lead);
    Best best{-CUDART_INF_F, -CUDART_INF_F, 0x7FFFFFFF};
#pragma unroll
    for (int i = 3; i >= 0; --i) {                      // downwards: equal scores keep the lower id
        const float e = 4 * part + i == li ? e_lead : e_lead + (15.942385152878742f - __logf(static_cast<float>(f[i]) + 0.5f));   // 23 ln 2 - ln(f + 0.5)
        const float sc = fmaf(temperature, -__logf(e), val[i]);
        if (val[i] > -CUDART_INF_F && sc >= best.score) best = Best{sc, val[i], v + i};
    }
    return best;
}
// Bounds of group v0 from its word R: no score of the group exceeds ub, and one is at least lo (-inf: no such score).
template <typename T>
__device__ __forceinline__ void group_bounds(const T* row_ptr, int v0, uint32_t R, float temperature, int vocab, int vec_ok, float* ub, float* lo) {
    float val[kGroup];
    load_group(row_ptr, v0, vocab, vec_ok, val);
    float gmax = val[0];
#pragma unroll
    for (int i = 1; i < kGroup; ++i) gmax = fmaxf(gmax, val[i]);
    *ub = gmax > -CUDART_INF_F ? fmaf(temperature, word_gumbel_bound(R), gmax) : -CUDART_INF_F;
    const int v = v0 + static_cast<int>(R & 15u);
    *lo = v < vocab ? fmaf(temperature, word_gumbel_least(R), Logit<T>::load1(row_ptr + v)) : -CUDART_INF_F;
}

// A block (the 64 ids of one lane in one tile) whose upper bound reached the running lower bound.
struct Reach {
    float ub;            // upper bound of the block's scores
    uint16_t tile;       // tile inside the piece
    uint16_t lane;
};
static_assert(sizeof(Reach) == 8, "eight bytes per kept block");

// Equal ranges over the rows' items, laid end to end: a row is row_axis places long, its items behind `pad` empty ones.
struct Ranges {
    int row_axis, pad;
    int ppr;                                            // > 0: no ranges, every row is cut into ppr pieces
    int axis;                                           // all rows
};

// Shared memory of the streaming kernel beyond its static arrays: the rings, the lists of kept blocks, the barriers.
// A ragged row's tile comes with the 16-byte granules it shares with its neighbours.
template <typename T, bool RAGGED>
__host__ __device__ constexpr int stream_stage_bytes() {
    return kTile * static_cast<int>(sizeof(T)) + (RAGGED ? 16 : 0);
}
template <typename T, bool RAGGED>
constexpr int stream_smem_bytes() {
    return kWarps * kStages * stream_stage_bytes<T, RAGGED>() + kWarps * kMaxList * 8 + kWarps * kStages * 8;
}

// RAGGED: rows start at any multiple of sizeof(T) (a vocabulary that is not a multiple of 16 bytes, or
// an unaligned base).  A tile is still one bulk copy, of the 16-byte granules that cover it, so that it
// lies `ms` elements into its stage (ms is the row's); a lane's 64 ids are then its chunks as
// before, except that the first one holds the last ms ids of the lane before it, in whose place the
// lane takes the first ms ids of the chunk after its last.  Which 64 ids a lane has is all the sums and
// maxima need, not their order.  The splice is a select per 32-bit word of the one chunk (half an
// instruction per logit).  Measured, 408 rows of 50257 bf16 logits, greedy, whole call: 28.8 us, against
// 57.8 us when the warp filled its stage with plain 2-byte loads, with nothing in flight behind them.
template <typename T, bool NOISY, bool RAGGED>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 2 ? 2 : 1)
unmask_stream_kernel(const T* __restrict__ logits, const uint8_t* state,
                     const __grid_constant__ UnmaskSets sets, UnmaskPartial* __restrict__ partial,
                     int vocab, int tiles_per_item, float temperature,
                     uint32_t block_idx, uint32_t step, int select_state,
                     const uint32_t* step_counter, int* __restrict__ status, uint32_t* shared_words) {
    // The launch may have been made resident before the kernel ahead of it on the stream was done (its
    // set-up then overlaps that kernel's tail); nothing is read before the wait.  The kernel behind
    // this one (the per-rollout step) may come in as soon as every CTA here has started.
    const int rows = sets.row_off[sets.n_sets];
    __shared__ uint32_t s_mask[kMaxRows / 32];          // which rows are selected (MASKED, or DRAFT for the verifier), 32 to a word
    __shared__ int2 s_open[kWarps][8];                  // (row, piece of the row) of the pieces a warp has begun to copy
    __shared__ int s_n_list[kWarps];
    constexpr bool kEqual = sizeof(T) == 2 && !NOISY && !RAGGED;                      // all pieces are equal ranges
    __shared__ Ranges s_ranges[kEqual ? kWarps : 1];    // (a copy for every warp: the tile loop has no registers to spare)
    __shared__ int4 s_cut[kEqual ? kWarps : 1][8];      // ... and for the pieces in s_open: first tile, tile behind the last, pieces of the row
    extern __shared__ __align__(128) unsigned char s_dyn[];
    constexpr int kStageBytes = stream_stage_bytes<T, RAGGED>();
    constexpr int kPerChunk = Logit<T>::kPerChunk;
    constexpr int kLaneChunks = kLaneIds / kPerChunk;   // 16-byte chunks of a lane's 64 ids: 8 (bf16) or 16 (fp32)
    constexpr int kLaneGroups = kLaneIds / kGroup;      // groups of a lane's 64 ids

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* ring = s_dyn + warp * (kStages * kStageBytes);
    Reach* list = reinterpret_cast<Reach*>(s_dyn + kWarps * kStages * kStageBytes) + warp * kMaxList;
    uint64_t* bars = reinterpret_cast<uint64_t*>(s_dyn + kWarps * kStages * kStageBytes + kWarps * kMaxList * 8) + warp * kStages;

    if (lane == 0) {
        s_n_list[warp] = 0;
        for (int s = 0; s < kStages; ++s) tc::mbar_init(tc::smem_u32(&bars[s]), 1);
        tc::fence_barrier_init();
    }
    tc::grid_dependency_wait();
    tc::grid_launch_dependents();
    // the denoising step as counted on the device (by the kernel ahead of this one: a plain load could be moved ahead of the wait)
    if (step_counter != nullptr) step += load_shared_word(step_counter);

    // ---- set-up (the only CTA-wide part): which rows are selected.  Every warp then keeps the count of selected rows
    // before the words of each lane, which is all it takes to find the ri-th of them.
    const int n_words = (rows + 31) / 32, per_lane = (n_words + 31) / 32;     // <= 256 and <= 8 (rows <= 8192)
    constexpr int kWordsAtOnce = 4;                     // (loads in flight together)
    for (int w0 = warp; w0 < per_lane * 32; w0 += kWarps * kWordsAtOnce) {
        int st[kWordsAtOnce];
#pragma unroll
        for (int u = 0; u < kWordsAtOnce; ++u) {
            const int r = (w0 + u * kWarps) * 32 + lane;
            st[u] = r < rows ? state[r] : -1;
        }
#pragma unroll
        for (int u = 0; u < kWordsAtOnce; ++u) {
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, st[u] == select_state);
            if (lane == 0 && w0 + u * kWarps < per_lane * 32) s_mask[w0 + u * kWarps] = m;
        }
    }
    __syncthreads();
    int rows_before, n_rows;
    {
        int mine = 0;
        for (int j = 0; j < per_lane; ++j) mine += __popc(s_mask[lane * per_lane + j]);
        int incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= off) incl += up;
        }
        rows_before = incl - mine;
        n_rows = __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (n_rows == 0) return;
    auto selected_row = [&](int ri) {                   // (warp-wide)
        const int at = __popc(__ballot_sync(0xFFFFFFFFu, rows_before <= ri)) - 1;
        int k = ri - __shfl_sync(0xFFFFFFFFu, rows_before, at), w = at * per_lane, c = __popc(s_mask[w]);
        while (k >= c) {
            k -= c;
            c = __popc(s_mask[++w]);
        }
        return w * 32 + nth_set_bit(s_mask[w], k);
    };

    // ---- the pieces.  An item is tiles_per_item consecutive tiles of a row (the last item of a row may be shorter);
    // a row has ipr of them and as many record slots.  Every row is cut into ppr pieces of about the same number of
    // items, and a piece leaves one record.  (A call has far fewer than 2^31 tiles: they lie in the GPU's memory.)
    //  - Few rows: as many pieces as there are warps, one for each, where each row can have kMinPiecesPerRow of them or
    //    where that makes no piece longer than an equal share.
    //  - Otherwise, greedy over bf16 rows that start on 16 bytes (kEqual): the rows' items end to end in equal ranges, a warp
    //    each.  Every piece costs about as much as a tile beside its own (opening, look-up, record), so kPiecePad items in
    //    front of every row stand for that where ranges are long.  These launches are bound by instructions more than the
    //    others, most of all at the lower clocks of a loaded GPU, and pieces dealt out as below cost them more than an even finish
    //    gives.  Whole calls, dealt out -> equal ranges, us, clocks free and (after heavy products) lowered, 151936 ids: 1216 rows 71.0 -> 70.9
    //    (97.6 -> 95.5), 608 rows 60.5 -> 55.4 (62.9 -> 57.6), 800 rows 56.6 -> 52.7 (74.6 -> 69.7), 1520 rows 86.2 -> 84.6 (117.7 ->
    //    113.7); 1216 rows of 128256 63.5 -> 60.7 (87.3 -> 83.3).  Without the padding 1520 rows took 86.5 (116.7).
    //  - Otherwise most of every row goes into long pieces, as many for each row as there are whole warps for it, and the rest
    //    into pieces of a few tiles, which the warps draw from a counter while they still work on the piece before (warps without
    //    a long piece from the start).  SMs stream at rates that differ by a quarter (with equal ranges the warps of a
    //    launch over 1216 rows of 152k ids with noise ended after 71 us at the median and 89 us at the latest).
    //    Whole calls, equal ranges -> long and short pieces, us: 1216 rows of 151936 bf16 logits with noise 95.2 -> 91.2, 608 rows
    //    60.4 -> 53.6, 1064 rows 86.1 -> 76.0, 1216 rows of 50257 49.3 -> 45.2 greedy and 73.1 -> 62.7 with noise, 720 rows of fp32
    //    logits 78.6 -> 74.4 and 83.1 -> 80.1.  A long piece for every warp, whole rows' long parts cut into equal ranges or some
    //    rows with one long piece more than others, was faster at 1216 rows (89.5 and 90.8 us with noise) and slower at 1064 (82.1 and 82.7).
    const int tiles_per_row = (vocab + kTile - 1) / kTile;
    const int ipr = (tiles_per_row + tiles_per_item - 1) / tiles_per_item;
    const int warps_all = static_cast<int>(gridDim.x) * kWarps;
    const int gw = warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);   // warps of a CTA lie a grid apart: few pieces spread over all SMs
    constexpr int kLongShare = sizeof(T) == 2 ? 8 : 6;            // tenths of a warp's share that are its long piece
    int ppr = min(ipr, warps_all / n_rows), n_long = 0, long_items = 0;
    int r_at = 0, r_end = 0;                            // (kEqual) the warp's range, on the axis of all rows' items end to end
    Ranges& R = s_ranges[kEqual ? warp : 0];
    if (kEqual) {
        const int share = (n_rows * ipr + warps_all - 1) / warps_all;
        const bool by_row = !(ppr < min(ipr, kMinPiecesPerRow) && (ppr == 0 || (ipr + ppr - 1) / ppr > share));
        const int pad = !by_row && share >= 16 * kPiecePad ? kPiecePad : 0, row_axis = ipr + pad;
        if (lane == 0) R = Ranges{row_axis, pad, by_row ? ppr : 0, n_rows * row_axis};
        if (by_row) {
            const int ri = gw / ppr, pc = gw - ri * ppr;
            if (ri >= n_rows) return;
            r_at = ri * ipr + static_cast<int>(static_cast<long long>(ipr) * pc / ppr);
            r_end = ri * ipr + static_cast<int>(static_cast<long long>(ipr) * (pc + 1) / ppr);
        } else {
            r_at = static_cast<int>(static_cast<long long>(n_rows * row_axis) * gw / warps_all);
            r_end = static_cast<int>(static_cast<long long>(n_rows * row_axis) * (gw + 1) / warps_all);
        }
        __syncwarp();
    } else {
        const int share = (n_rows * ipr + warps_all - 1) / warps_all;
        if (ppr < min(ipr, kMinPiecesPerRow) && (ppr == 0 || (ipr + ppr - 1) / ppr > share)) {
            const int len = max(1, min(max(share * tiles_per_item / kDealtShare, kDealtLeast), kDealtMost) / tiles_per_item);
            const int at_most = max(1, warps_all / n_rows), rounds = (n_rows * at_most + warps_all - 1) / warps_all;
            long_items = min(share * kLongShare / 10 / rounds, ipr * kLongShare / 10 / at_most);
            if (long_items > 2 * len) n_long = at_most;
            ppr = n_long + (ipr - n_long * long_items + len - 1) / len;
        }
    }
    const int n_short = max(1, ppr - n_long), n_pieces = n_rows * ppr;
    const int short_items = (ipr - n_long * long_items) / n_short, short_more = ipr - n_long * long_items - short_items * n_short;
    // first item of a piece (the first short_more short pieces of a row have one item more)
    auto first_item = [&](int pc) {
        if (pc <= n_long) return pc * long_items;
        return n_long * long_items + (pc - n_long) * short_items + min(pc - n_long, short_more);
    };
    if (!kEqual && gw >= n_pieces) return;

    const uint32_t full = 0xFFFFFFFFu;
    const int sw = lane & 7;                            // rotation of the chunk order (bank conflicts)
    bool alive = true;                                  // false once a wait for a copy ran out

    // ---- producer side (lane 0 issues, every lane keeps the same cursor): tile k of the warp's
    // sequence goes to stage k % kStages, which is the stage the consumer has just left
    const uint32_t ring_u32 = tc::smem_u32(ring), bars_u32 = tc::smem_u32(bars);
    int p_next = gw;                                    // next piece to open (lane 0's, once it comes from the counter)
    int p_open = 0;                                     // pieces opened so far
    int p_tile = 0, p_tile_end = 0;
    const T* p_row_ptr = nullptr;
    uint32_t p_k = 0;
    const uint64_t l2_policy = read_once_policy();
    // (ragged) whole 16-byte granules inside the call's logits: no copy reaches beyond them
    const uintptr_t whole_begin = (reinterpret_cast<uintptr_t>(logits) + 15) & ~uintptr_t(15);
    const uintptr_t whole_end = reinterpret_cast<uintptr_t>(logits + static_cast<size_t>(rows) * vocab) & ~uintptr_t(15);
    auto produce_one = [&](int stage) {
        if (kEqual) {
            while (p_tile == p_tile_end) {
                if (r_at >= r_end) return;
                const int ri = r_at / R.row_axis, o = r_at - ri * R.row_axis, o_end = min(R.row_axis, o + r_end - r_at);
                r_at += o_end - o;
                p_tile = max(0, o - R.pad) * tiles_per_item;
                p_tile_end = min(tiles_per_row, max(0, o_end - R.pad) * tiles_per_item);
                if (p_tile == p_tile_end) continue;     // (padding alone)
                const int row = selected_row(ri);
                p_row_ptr = logits + static_cast<size_t>(row) * vocab;
                int first = ri * R.ppr, of = R.ppr;     // the warp that holds the row's first item, and how many hold one
                if (R.ppr == 0) {
                    const long long at = static_cast<long long>(ri) * R.row_axis;
                    first = static_cast<int>(((at + R.pad + 1) * warps_all - 1) / R.axis);
                    of = static_cast<int>(((at + R.row_axis) * warps_all - 1) / R.axis) - first + 1;
                }
                if (lane == 0) {
                    s_open[warp][p_open & 7] = make_int2(row, gw - first);
                    s_cut[kEqual ? warp : 0][p_open & 7] = make_int4(p_tile, p_tile_end, of, 0);
                }
                ++p_open;
                __syncwarp();
            }
        } else if (p_tile == p_tile_end) {
            const int id = __shfl_sync(full, p_next, 0);
            if (id >= n_pieces) return;
            // (the long pieces of all rows come first)
            const bool is_long = id < n_rows * n_long;
            const int among = is_long ? id : id - n_rows * n_long, per_row = is_long ? n_long : n_short, ri = among / per_row;
            const int pc = among - ri * per_row + (is_long ? 0 : n_long), row = selected_row(ri);
            p_tile = first_item(pc) * tiles_per_item;
            p_tile_end = min(tiles_per_row, first_item(pc + 1) * tiles_per_item);
            p_row_ptr = logits + static_cast<size_t>(row) * vocab;
            // (at most kStages pieces are ahead of the one being reduced; the answer of the counter is not needed before
            // the last tile of this piece is on its way)
            if (lane == 0) {
                s_open[warp][p_open & 7] = make_int2(row, pc);
                p_next = n_pieces > warps_all ? warps_all + static_cast<int>(atomicAdd(shared_words + kSharedNext, 1u)) : n_pieces;
            }
            ++p_open;
            __syncwarp();
        }
        if (lane == 0) {
            const int v0 = p_tile * kTile;
            const uint32_t bytes = static_cast<uint32_t>(min(kTile, vocab - v0)) * sizeof(T);
            const uint32_t bar = bars_u32 + stage * 8;
            if (!RAGGED) {
                tc::mbar_arrive_expect_tx(bar, bytes);
                bulk_load(ring_u32 + stage * kStageBytes, p_row_ptr + v0, bytes, bar, l2_policy);
            } else {
                const uintptr_t first = reinterpret_cast<uintptr_t>(p_row_ptr + v0), at0 = first & ~uintptr_t(15);
                const uintptr_t from = at0 > whole_begin ? at0 : whole_begin;
                const uintptr_t last = (first + bytes + 15) & ~uintptr_t(15), to = last < whole_end ? last : whole_end;
                const uint32_t n = to > from ? static_cast<uint32_t>(to - from) : 0u;
                tc::mbar_arrive_expect_tx(bar, n);
                if (n != 0u)
                    bulk_load(ring_u32 + stage * kStageBytes + static_cast<uint32_t>(from - at0), reinterpret_cast<const void*>(from), n, bar, l2_policy);
            }
        }
        ++p_tile;
        ++p_k;
    };
    for (int s = 0; s < kStages; ++s) produce_one(s);

    uint32_t c_k = 0;                                   // tiles consumed so far: the next one sits in stage c_k % kStages
    int stage = 0;
    uint32_t phase = 0;                                 // parity of the stage's current use
    for (int c_open = 0; c_open != p_open && alive; ++c_open) {
        // ---- open the piece: tiles [tile0, tile1) of one row
        const int row = s_open[warp][c_open & 7].x, pc = s_open[warp][c_open & 7].y;
        int tile0, tile1, of;                           // its tiles, and how many pieces the row has
        if (kEqual) {
            const int4 cut = s_cut[kEqual ? warp : 0][c_open & 7];
            tile0 = cut.x;
            tile1 = cut.y;
            of = cut.z;
        } else {
            tile0 = first_item(pc) * tiles_per_item;
            tile1 = min(tiles_per_row, first_item(pc + 1) * tiles_per_item);
            of = ppr;
        }
        const int seg_end = min(vocab, tile1 * kTile);
        uint32_t* const row_bar = shared_words + kSharedBars + row;
        const T* row_ptr = logits + static_cast<size_t>(row) * vocab;
        const int ms = RAGGED ? static_cast<int>((reinterpret_cast<uintptr_t>(row_ptr) & 15u) / sizeof(T)) : 0;
        const int vec_ok = ms == 0;                     // the row can be read in 16-byte chunks
        int set = 0;
        while (set + 1 < sets.n_sets && row >= sets.row_off[set + 1]) ++set;
        const int local = row - sets.row_off[set];
        const int fork = local / sets.d[set], pos = local - fork * sets.d[set];   // rollout inside its set
        uint2 keys = make_uint2(0u, 0u);
        if (NOISY) {
            const uint64_t seed = sets.seeds[set][fork];
            // (through a shuffle, which tells the compiler that the key is the same in every lane: the
            // round keys of the Philox blocks then live in uniform registers)
            keys = make_uint2(__shfl_sync(0xFFFFFFFFu, static_cast<uint32_t>(seed), 0),
                              __shfl_sync(0xFFFFFFFFu, static_cast<uint32_t>(seed >> 32), 0));
        }

        // ---- pass 1: stream the piece; per lane s = sum of 2^((l - ref) log2 e), where ref is the largest logit of the
        // lane's first 64 ids and moves only when a logit exceeds it by more than kRefSlack: the exponentials wait for
        // no running maximum, and their sum keeps the precision it has with one (arguments stay below 6).  The greedy
        // step also keeps the lane's maximum u1 and the first tile t1 that showed it; the noisy step keeps the warp's
        // running lower bound lb of the piece's best score and lists the blocks that reach it.
        float ref = -CUDART_INF_F, s = 0.0f, nref = 0.0f;   // nref = -ref log2(e) once ref is finite
        auto move_ref = [&](float bm) {
            if (bm > ref + kRefSlack) {                 // (also the first time: ref is -inf then)
                const float to = fmaxf(bm, kRefLeast);
                s *= tc::ex2((ref - to) * kLog2e);
                ref = to;
                nref = -to * kLog2e;
            }
        };
        float u1 = -CUDART_INF_F, lb = -CUDART_INF_F;
        int t1 = tile0;
        Best best{-CUDART_INF_F, -CUDART_INF_F, 0x7FFFFFFF};
        for (int tile = tile0; tile < tile1; ++tile) {
            unsigned char* buf = ring + stage * kStageBytes;
            const int tile_base = tile * kTile;
            if (!wait_copy(bars_u32 + stage * 8, phase)) alive = false;
            alive = __all_sync(full, alive);
            if (!alive) break;
            if (RAGGED) {
                // the ends of the logits themselves: elements outside the whole granules were not copied
                const uintptr_t first = reinterpret_cast<uintptr_t>(row_ptr + tile_base);
                const uintptr_t end = first + static_cast<uintptr_t>(min(kTile, vocab - tile_base)) * sizeof(T);
                if ((first & ~uintptr_t(15)) < whole_begin || end > whole_end) {
                    T* dst = reinterpret_cast<T*>(buf) + ms;
                    for (int i = lane; i < min(kTile, vocab - tile_base); i += 32) {
                        const uintptr_t p = first + static_cast<uintptr_t>(i) * sizeof(T);
                        if (p < whole_begin || p >= whole_end) dst[i] = row_ptr[tile_base + i];
                    }
                    tc::fence_proxy_async();            // (a later copy may go to the same stage)
                    __syncwarp();
                }
            }
            const int vb = tile_base + lane * kLaneIds;  // first id of the lane's 64
            const uint4* sp = reinterpret_cast<const uint4*>(buf) + lane * kLaneChunks;
            const T* lp = reinterpret_cast<const T*>(buf) + lane * kLaneIds + ms;
            float bm64 = -CUDART_INF_F;
            uint32_t others = 0u;                       // what the row's other pieces have found (looked at behind the sums)
            if (NOISY && ppr > 1) others = load_shared_word(row_bar);
            // (per lane: in a row's last tile the lanes whose 64 ids all exist take the fast path too, the
            // lanes beyond the row's end have nothing to do, and at most one lane straddles the end)
            const bool whole = vb + kLaneIds <= seg_end;
            uint4 rq = make_uint4(0u, 0u, 0u, 0u);      // the words of the block's four groups
            const uint4 counter = make_uint4(static_cast<uint32_t>(vb >> 6), static_cast<uint32_t>(pos), step, block_idx);
            if (whole) {
                // the lane's 64 logits as they lie in the stage, chunk c read from place c ^ sw (the eight
                // lanes of a quarter warp then touch eight different 16-byte columns of the banks)
                uint4 w[kLaneChunks];
#pragma unroll
                for (int k = 0; k < kLaneChunks; ++k) w[k] = sp[k ^ sw];
                if (RAGGED) {
                    const uint4 after = sp[kLaneChunks];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k == sw) w[k] = Logit<T>::splice(w[k], after, ms);          // (place 0)
                }
                if (tile == tile0) move_ref(Logit<T>::template largest<kLaneChunks>(w));
                // (the reference stands in all but a few tiles: the sum does not wait for the maximum, and is
                // formed again where a logit exceeds the reference by too much)
                for (;;) {
                    if (NOISY) rq = philox4x32_10(counter, keys);          // (here, so that its rounds overlap the exponentials)
                    // packed fp32x2 arithmetic: one FMA and one add per two logits
                    const uint64_t l2e2 = tc::pack2(kLog2e, kLog2e), nm2 = tc::pack2(nref, nref);
                    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int k = 0; k < kLaneChunks; ++k) {
                        float v[kPerChunk];
                        Logit<T>::widen(w[k], v);
#pragma unroll
                        for (int i = 0; i < kPerChunk; i += 2) {
                            float x0, x1;
                            tc::unpack2(tc::fma2(tc::pack2(v[i], v[i + 1]), l2e2, nm2), x0, x1);
                            acc[(i >> 1) & 3] = tc::add2(acc[(i >> 1) & 3], tc::pack2(tc::ex2(x0), tc::ex2(x1)));
                        }
                    }
                    bm64 = Logit<T>::template largest<kLaneChunks>(w);
                    if (bm64 > ref + kRefSlack) {
                        move_ref(bm64);
                        continue;
                    }
                    float a0, a1;
                    tc::unpack2(tc::add2(tc::add2(acc[0], acc[1]), tc::add2(acc[2], acc[3])), a0, a1);
                    s += a0 + a1;
                    break;
                }
            } else if (vb < seg_end) {
                // the lane that straddles the row's end: ids from seg_end on do not exist
                if (NOISY) rq = philox4x32_10(counter, keys);
                for (int e = 0; e < kLaneIds; ++e)
                    if (vb + e < seg_end) bm64 = fmaxf(bm64, Logit<T>::load1(lp + e));
                move_ref(bm64);
                float add = 0.0f;
                for (int e = 0; e < kLaneIds; ++e)
                    if (vb + e < seg_end) add += tc::ex2(fmaf(Logit<T>::load1(lp + e), kLog2e, nref));
                s += add;
            }
            if (!NOISY) {
                t1 = bm64 > u1 ? tile : t1;             // strictly: t1 is the first tile that holds the lane's maximum
                u1 = fmaxf(u1, bm64);
            } else {
                // The block's four words: the largest one bounds every draw of the block, and its group's
                // leader gives a score that exists.  d = 2^28 - 1 - (R >> 4), cut to 23 bits (d5 = d / 32,
                // rounded down) so that it turns into a float exactly; both bounds stay on the safe side.
                uint32_t rmax;
                int gp;                                 // the group (of the block's four) that holds rmax
                if (whole) {
                    const uint32_t r01 = max(rq.x, rq.y), r23 = max(rq.z, rq.w);
                    rmax = max(r01, r23);
                    gp = rmax == rq.x ? 0 : (rmax == rq.y ? 1 : (rmax == rq.z ? 2 : 3));
                } else {
                    rmax = rq.x;                        // (group 0 exists: the block does)
                    gp = 0;
#pragma unroll
                    for (int g = 1; g < kLaneGroups; ++g)
                        if (vb + g * kGroup < seg_end && pick_word(rq, g) > rmax) { rmax = pick_word(rq, g); gp = g; }
                }
                const uint32_t d5 = (0x0FFFFFFFu - (rmax >> 4)) >> 5;
                const float fd5 = __uint_as_float(0x4B000000u | d5) - 8388608.0f;          // d5 as a float, exactly
                // g < 32 ln 2 - ln d <= 27 ln 2 - ln d5
                const float g_hi = d5 == 0u ? CUDART_INF_F : fmaf(-kLn2, __log2f(fd5), 18.71497388f + 2e-3f);
                const float ub = fmaf(temperature, g_hi, bm64);
                lb = fmaxf(lb, bar_value(others));
                const bool reaches = bm64 > -CUDART_INF_F && ub >= lb - 1e-3f;
                // (no block in reach: no score of this tile step can raise the bound either, since the
                // lower bounds below lie under the blocks' upper bounds)
                if (__any_sync(full, reaches)) {
                    // g_leader >= 32 ln 2 - ln((d + 1) (1 + y)), y = (d + 1) / 2^28 <= 1 / 2; d + 1 <= 32 (d5 + 1)
                    const float y = (fd5 + 1.0f) * 1.1920928955078125e-07f;                 // >= (d + 1) / 2^28
                    const float g_lo = y <= 0.5f ? fmaf(-kLn2, __log2f(fd5 + 1.0f), 18.71497388f - 2e-3f) - y : kGumbelMin;
                    const int li = gp * kGroup + static_cast<int>(rmax & 15u);
                    // a score that exists in this block: that leader's, or the largest logit's with the smallest draw there is
                    float lo = bm64 > -CUDART_INF_F ? fmaf(temperature, kGumbelMin, bm64) : -CUDART_INF_F;
                    if (vb + li < seg_end) lo = fmaxf(lo, fmaf(temperature, g_lo, Logit<T>::load1(lp + li)));
                    lo = warp_max(lo);
                    if (lo > lb) {                      // (the same in every lane)
                        lb = lo;
                        if (ppr > 1 && lane == 0) atomicMax(row_bar, bar_key(lb));
                    }
                    if (reaches && ub >= lb - 1e-3f) {
                        const int slot = atomicAdd(&s_n_list[warp], 1);
                        if (slot < kMaxList) list[slot] = Reach{ub, static_cast<uint16_t>(tile - tile0), static_cast<uint16_t>(lane)};
                    }
                }
            }
            __syncwarp();                               // every lane is done with the stage
            produce_one(stage);                         // tile c_k + kStages goes into it
            ++c_k;
            if (++stage == kStages) {
                stage = 0;
                phase ^= 1u;
            }
        }
        if (!alive) break;

        if (NOISY) {
            // ---- pass 2: lb is now a lower bound of the row's best score as far as its pieces have come.  The listed blocks
            // that still reach it (none in most pieces, eight or so in a row) are read again (the piece has just gone through L2) and scored exactly, group by
            // group: a turn deals out eight blocks, one group per lane, so that the loads are in flight
            // together.  (A list that ran over, or a piece of more than 65536 tiles: every block.)
            __syncwarp();
            const RowNoise noise{keys, static_cast<uint32_t>(pos), step, block_idx};
            const int n_seen = *reinterpret_cast<volatile int*>(&s_n_list[warp]);
            if (n_seen > 0 && ppr > 1) lb = fmaxf(lb, bar_value(load_shared_word(row_bar)));
            const float cut = lb - 1e-3f;
            const bool every = n_seen > kMaxList || tile1 - tile0 > 65536;
            int n_blocks = 0;
            if (every) {
                n_blocks = (tile1 - tile0) * 32;
            } else {
                // keep the blocks that reach the final bound, in place
                for (int c0 = 0; c0 < n_seen; c0 += 32) {
                    const int c = c0 + lane;
                    Reach r{-CUDART_INF_F, 0, 0};
                    if (c < n_seen) r = list[c];
                    const bool keep = r.ub >= cut;
                    const uint32_t km = __ballot_sync(full, keep);
                    if (keep) list[n_blocks + __popc(km & ((1u << lane) - 1u))] = r;
                    n_blocks += __popc(km);
                    __syncwarp();
                }
            }
            // Two stages, eight blocks at a time.  Stage one, a group per lane: the bounds of single groups (the group's word
            // with the group's largest logit, and its leader's score), which are tighter than the block's and raise lb.
            // Stage two: the few groups that still reach lb are scored exactly, four ids per lane.  The best exact
            // score so far raises lb for the next eight.
            for (int c0 = 0; c0 < n_blocks; c0 += 32 / kLaneGroups) {
                const int c = c0 + lane / kLaneGroups, g = lane % kLaneGroups;
                int v_own = seg_end;
                if (c < n_blocks) {
                    const int tl = every ? c / 32 : list[c].tile, fl = every ? c % 32 : list[c].lane;
                    v_own = (tile0 + tl) * kTile + fl * kLaneIds + g * kGroup;
                }
                float ub = -CUDART_INF_F, lo = -CUDART_INF_F;
                if (v_own < seg_end) {
                    // (a listed block lies inside the piece as a whole; only the row's end can cut it short,
                    // and ids beyond the vocabulary read as -inf)
                    const uint4 rq = philox4x32_10(make_uint4(static_cast<uint32_t>(v_own >> 6), static_cast<uint32_t>(pos), step, block_idx), keys);
                    group_bounds(row_ptr, v_own, pick_word(rq, g), temperature, vocab, vec_ok, &ub, &lo);
                }
                lb = fmaxf(lb, warp_max(lo));
                const uint32_t reach = __ballot_sync(full, ub > -CUDART_INF_F && ub >= lb - 1e-3f);
                const int total = __popc(reach);
                for (int j0 = 0; j0 < total; j0 += 8) {
                    const int r = j0 + (lane >> 2);
                    const bool act = r < total;
                    const int v0 = __shfl_sync(full, v_own, act ? nth_set_bit(reach, r) : 0);
                    best = better(best, score_quarter<T>(row_ptr, v0, lane & 3, act, temperature, vocab, noise));
                }
                if (c0 + 32 / kLaneGroups < n_blocks) lb = fmaxf(lb, warp_max(best.score));
            }
            if (lane == 0) s_n_list[warp] = 0;          // the list is empty again for the next piece
        } else {
            // ---- greedy: the piece's maximum and its first place: of the lanes that hold the maximum the one whose
            // first tile with it has the lowest ids; the warp reads those 64 ids together (equal values in later
            // tiles have higher ids).
            const float pm = warp_max(u1);
            if (pm > -CUDART_INF_F) {
                const int v = warp_min(u1 == pm ? t1 * kTile + lane * kLaneIds : 0x7FFFFFFF) + lane;
                const bool h0 = v < vocab && Logit<T>::load1(row_ptr + v) == pm, h1 = v + 32 < vocab && Logit<T>::load1(row_ptr + v + 32) == pm;
                const uint32_t m0 = __ballot_sync(full, h0), m1 = __ballot_sync(full, h1);
                best = Best{pm, pm, v - lane + (m0 != 0u ? __ffs(m0) - 1 : 31 + __ffs(m1))};
            }
        }

        // ---- the piece's record
        const float row_ref = warp_max(ref);
        s = warp_sum(ref > -CUDART_INF_F ? s * tc::ex2((ref - row_ref) * kLog2e) : 0.0f);
        if (NOISY) best = warp_best(best);              // (greedy: the same in every lane)
        if (lane == 0) {
            UnmaskPartial out;
            out.row_max = row_ref; out.sum_exp = s; out.best_score = best.score; out.best_logit = best.logit;
            out.best_index = best.index;
            out.pad[0] = of;                            // how many records this row has (read from record 0)
            out.pad[1] = out.pad[2] = 0;
            partial[static_cast<size_t>(row) * ipr + pc] = out;
        }
        __syncwarp();
    }

    if (!alive) {
        // A copy did not arrive in time: say so, then give the copies still in flight one more bounded
        // wait each before the shared memory they write to is handed back.
        if (lane == 0 && status != nullptr) atomicCAS(status, 0, FDD_ERR_DEVICE_TIMEOUT);
        for (uint32_t k = c_k; k < p_k; ++k) {
            const long long t0 = clock64();
            while (!tc::mbar_try_wait(tc::smem_u32(&bars[k % kStages]), (k / kStages) & 1u))
                if (clock64() - t0 > kCopyWaitLimit) break;
        }
    }
}

constexpr int kFinalizeThreads = 512;               // the first 128 are the positions of the rollout; all of them merge records

// What the per-rollout kernels share: where the rollout's rows lie, and the merged records of its selected rows.
struct RolloutRows {
    int fork, d, row0;                              // rollout over all sets of the call, its block length and first row
};
__device__ __forceinline__ RolloutRows rollout_rows(const UnmaskSets& sets) {
    RolloutRows r;
    r.fork = blockIdx.x;
    int set = 0;
    while (set + 1 < sets.n_sets && r.fork >= sets.fork_off[set + 1]) ++set;
    r.d = sets.d[set];
    r.row0 = sets.row_off[set] + (r.fork - sets.fork_off[set]) * r.d;
    return r;
}
struct MergeShared {
    int tok[128], nrec[128], rows[128];             // token, records and position of the selected rows
    float conf[128];
    int n_rows, max_rec;
};

// The selected positions and how many records each has; thread i is position i.
__device__ __forceinline__ void list_rows(MergeShared& sh, int i, bool selected, int n_rec) {
    if (i < 128) {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, selected);
        const int most = __reduce_max_sync(0xFFFFFFFFu, selected ? n_rec : 1);
        int base = 0;
        if ((i & 31) == 0 && m != 0u) {
            base = atomicAdd(&sh.n_rows, __popc(m));
            atomicMax(&sh.max_rec, most);
        }
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (selected) {
            sh.nrec[i] = n_rec;
            sh.rows[base + __popc(m & ((1u << (i & 31)) - 1u))] = i;
        }
    }
}

// Merge the records of the listed rows: a group of w lanes per position (w = the largest record count, rounded up
// to a power of two, 32 at most), so that all records of 32 / w positions are fetched in one round
// trip per warp (three records a lane at once: a row of 152k ids has 75).  Early steps have many positions with two or
// three records, late steps a few positions with up to a record per tile.  CONF: also the confidence of the best id.
template <bool CONF>
__device__ __forceinline__ void merge_rows(MergeShared& sh, const UnmaskPartial* partial, int row0, int items_per_row, int i) {
    constexpr int kAtOnce = 3;
    const int warp = i >> 5, lane = i & 31;
    const int n_rows = sh.n_rows, max_rec = sh.max_rec;
    int w = 1;
    while (w < max_rec && w < 32) w <<= 1;
    const int per = 32 / w, sub = lane / w, sl = lane - sub * w;
    for (int base = warp * per; base < n_rows; base += (kFinalizeThreads / 32) * per) {   // (warp-uniform bounds)
        const int k = base + sub;
        const bool valid = k < n_rows;
        const int j = valid ? sh.rows[k] : 0;
        const int nr = valid ? sh.nrec[j] : 0;
        const UnmaskPartial* p = partial + static_cast<size_t>(row0 + j) * items_per_row;
        float M = -CUDART_INF_F, S = 0.0f;
        Best B{-CUDART_INF_F, -CUDART_INF_F, 0x7FFFFFFF};
        for (int c0 = sl; c0 < nr; c0 += kAtOnce * w) {
            float4 st4[kAtOnce];                                            // row_max, sum_exp, best_score, best_logit
            int idx[kAtOnce];
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) {
                const int c = c0 + u * w;
                st4[u] = make_float4(-CUDART_INF_F, 0.0f, -CUDART_INF_F, -CUDART_INF_F);
                idx[u] = 0x7FFFFFFF;
                if (c < nr) {
                    st4[u] = *reinterpret_cast<const float4*>(&p[c]);
                    idx[u] = p[c].best_index;
                }
            }
            if (CONF) {
                const float mn = fmaxf(M, tc::max3(st4[0].x, st4[1].x, st4[2].x));
                if (mn > -CUDART_INF_F) {
                    S *= __expf(M - mn);
#pragma unroll
                    for (int u = 0; u < kAtOnce; ++u) S = fmaf(st4[u].y, __expf(st4[u].x - mn), S);
                }
                M = mn;
            }
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) B = better(B, Best{st4[u].z, st4[u].w, idx[u]});
        }
        const float own = M;
        for (int off = w >> 1; off > 0; off >>= 1) {
            if (CONF) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, off));
            Best o;
            o.score = __shfl_xor_sync(0xFFFFFFFFu, B.score, off);
            o.logit = __shfl_xor_sync(0xFFFFFFFFu, B.logit, off);
            o.index = __shfl_xor_sync(0xFFFFFFFFu, B.index, off);
            B = better(B, o);
        }
        if (CONF) {
            S = own > -CUDART_INF_F ? S * __expf(own - M) : 0.0f;
            for (int off = w >> 1; off > 0; off >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, off);
        }
        if (valid && sl == 0) {
            if (CONF) sh.conf[j] = expf(B.logit - M) / S;
            sh.tok[j] = B.index;
        }
    }
}

// Bound by latencies (one CTA of 512 threads a rollout, a few KB): the chain is state and record counts, records,
// their reduction, the rule.  What does not depend on the streaming kernel stands ahead of the wait for it.  (What that
// kernel writes is not declared read-only here: such loads could be moved ahead of the wait.)
__global__ void __launch_bounds__(kFinalizeThreads)
unmask_finalize_kernel(const UnmaskPartial* partial, int32_t* __restrict__ tokens,
                       uint8_t* state, int32_t* __restrict__ n_committed,
                       int32_t* __restrict__ n_left, float* __restrict__ conf_out,
                       const __grid_constant__ UnmaskSets sets, int items_per_row, float threshold, int commit_state,
                       uint32_t* __restrict__ step_bump, int2* __restrict__ left_mirror, int mirror_stamp,
                       uint32_t* __restrict__ shared_words, int32_t* __restrict__ gate_out) {
    tc::grid_launch_dependents();                       // the next kernel may be made resident; it waits for this one
    __shared__ MergeShared sh;
    const int i = threadIdx.x;
    const RolloutRows r = rollout_rows(sets);
    const int d = r.d, row = r.row0 + i;
    if (i == 0) { sh.n_rows = 0; sh.max_rec = 1; }
    if (i < 128) sh.conf[i] = -1.0f;
    __syncthreads();
    tc::grid_dependency_wait();                         // the streaming kernel's records are complete and visible
    // (the streaming kernel of this call has read the counter; the next call sees it advanced)
    if (step_bump != nullptr && blockIdx.x == 0 && i == 0) *step_bump += 1u;

    // ---- the MASKED positions of the rollout (d <= 128: threads beyond it only help with the merge)
    bool masked = false;
    int n_rec = 1;
    if (i < d) {
        // records the first kernel wrote for this row (never more than the row has slots; not looked at if it is not
        // MASKED): the two loads are independent, one round trip
        n_rec = partial[static_cast<size_t>(row) * items_per_row].pad[0];
        masked = state[row] == FDD_MASKED;
        shared_words[kSharedBars + row] = 0u;
        n_rec = max(1, min(items_per_row, n_rec));
    }
    if (blockIdx.x == 0 && i == 0) shared_words[kSharedNext] = 0u;     // (the streaming kernel is through with them)
    list_rows(sh, i, masked, n_rec);
    __syncthreads();
    const int n_masked = sh.n_rows;
    merge_rows<true>(sh, partial, r.row0, items_per_row, i);
    __syncthreads();

    // ---- the commit rule of the rollout
    const float conf = i < 128 ? sh.conf[i] : -1.0f;
    if (i < d && conf_out) conf_out[row] = masked ? conf : CUDART_NAN_F;
    const bool pass = masked && conf > threshold;
    const int n_pass = __syncthreads_count(pass);
    bool commit = pass;
    if (n_masked > 0 && n_pass == 0) {
        // at-least-one rule: the most confident MASKED position, lowest index on ties (each warp finds it for itself)
        int best_i = -1;
        float best_c = -1.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float c = sh.conf[k * 32 + (i & 31)];
            if (c > best_c) { best_c = c; best_i = k * 32 + (i & 31); }
        }
        const float top = warp_max(best_c);
        commit = i == warp_min(best_i >= 0 && best_c == top ? best_i : 0x7FFFFFFF);
    }
    if (commit && i < d) {
        tokens[row] = sh.tok[i];
        state[row] = static_cast<uint8_t>(commit_state);
    }
    if (i == 0) {
        const int nc = (n_masked == 0) ? 0 : (n_pass > 0 ? n_pass : 1);
        n_committed[r.fork] = nc;
        n_left[r.fork] = n_masked - nc;
        if (gate_out != nullptr) gate_out[r.fork] = n_masked - nc;
        // host memory the GPU can write: count and stamp go out as one 8-byte store, so a host that
        // sees the stamp of this call sees its count
        if (left_mirror != nullptr)
            *reinterpret_cast<unsigned long long*>(left_mirror + r.fork) =
                (static_cast<unsigned long long>(static_cast<uint32_t>(mirror_stamp)) << 32) | static_cast<uint32_t>(n_masked - nc);
    }
}


// Accept scan of Scaffold Speculative Decoding: one CTA per rollout.  The first kernel has left, for
// every DRAFT row, the verifier's token (arg-max of its perturbed logits).  Going left to right, a
// draft is accepted while it equals the verifier's token; at the first mismatch the verifier's token
// replaces it and every later draft goes back to MASKED.
__global__ void __launch_bounds__(kFinalizeThreads)
ss_accept_kernel(const UnmaskPartial* partial, int32_t* __restrict__ tokens,
                 uint8_t* state, int32_t* __restrict__ n_accepted, int32_t* __restrict__ n_left,
                 const __grid_constant__ UnmaskSets sets, int items_per_row, uint32_t* __restrict__ shared_words) {
    tc::grid_launch_dependents();
    __shared__ MergeShared sh;
    __shared__ int s_first_mismatch;
    const int i = threadIdx.x;
    const RolloutRows r = rollout_rows(sets);
    const int d = r.d, row = r.row0 + i;
    if (i == 0) { sh.n_rows = 0; sh.max_rec = 1; s_first_mismatch = 0x7FFFFFFF; }
    __syncthreads();
    tc::grid_dependency_wait();                         // the streaming kernel's records are complete and visible
    int st = FDD_SCAFFOLD, n_rec = 1, drafted = 0;
    if (i < d) {
        n_rec = partial[static_cast<size_t>(row) * items_per_row].pad[0];
        st = state[row];
        drafted = tokens[row];
        shared_words[kSharedBars + row] = 0u;
        n_rec = max(1, min(items_per_row, n_rec));
    }
    const bool draft = st == FDD_DRAFT;
    if (blockIdx.x == 0 && i == 0) shared_words[kSharedNext] = 0u;
    list_rows(sh, i, draft, n_rec);
    __syncthreads();
    merge_rows<false>(sh, partial, r.row0, items_per_row, i);
    __syncthreads();
    const int tok = draft ? sh.tok[i] : 0;
    if (draft && tok != drafted) atomicMin(&s_first_mismatch, i);
    __syncthreads();
    const int stop = s_first_mismatch;                  // position of the replacement token, if any
    const bool accepted = draft && i <= stop;
    if (accepted) {
        if (i == stop) tokens[row] = tok;               // the verifier's token, always accepted
        state[row] = FDD_COMMITTED;
    } else if (draft) {
        state[row] = FDD_MASKED;                        // discarded draft
    }
    const int n_accept = __syncthreads_count(accepted);
    const int n_masked = __syncthreads_count((draft && !accepted) || (i < d && st == FDD_MASKED));
    if (i == 0) {
        n_accepted[r.fork] = n_accept;
        n_left[r.fork] = n_masked;
    }
}

}  // namespace

namespace {

// Per-device set-up of the streaming kernels (they need more dynamic shared memory than a kernel
// gets without asking) and the device's SM count, done by the first launch on each device.
constexpr int kMaxDevices = 64;
std::atomic<int> g_device_ready[kMaxDevices];
int g_device_sms[kMaxDevices];
int g_device_ctas[kMaxDevices][8];          // resident CTAs per SM of each instantiation: bf16 noisy, bf16 greedy, fp32 noisy, fp32 greedy; the ragged ones behind them

template <typename T, bool NOISY, bool RAGGED>
cudaError_t setup_one(int* ctas_per_sm) {
    auto kernel = unmask_stream_kernel<T, NOISY, RAGGED>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, stream_smem_bytes<T, RAGGED>());
    // all of the SM's configurable memory as shared memory: two CTAs of the bf16 kernel need 215 KB
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, kernel, kThreads, stream_smem_bytes<T, RAGGED>());
    if (e == cudaSuccess && *ctas_per_sm < 1) e = cudaErrorLaunchOutOfResources;
    return e;
}

// Bytes of the shared words of a launch over at most `rows` rows (a multiple of 128: the records lie behind them).
size_t unmask_shared_bytes(int rows) { return ((kSharedBars + static_cast<size_t>(rows)) * sizeof(uint32_t) + 127) / 128 * 128; }

cudaError_t device_setup(int dev, int* sm_count, const int** ctas_per_sm) {
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!g_device_ready[dev].load(std::memory_order_acquire)) {
        int* c = g_device_ctas[dev];
        cudaError_t e = setup_one<__nv_bfloat16, true, false>(c + 0);
        if (e == cudaSuccess) e = setup_one<__nv_bfloat16, false, false>(c + 1);
        if (e == cudaSuccess) e = setup_one<float, true, false>(c + 2);
        if (e == cudaSuccess) e = setup_one<float, false, false>(c + 3);
        if (e == cudaSuccess) e = setup_one<__nv_bfloat16, true, true>(c + 4);
        if (e == cudaSuccess) e = setup_one<__nv_bfloat16, false, true>(c + 5);
        if (e == cudaSuccess) e = setup_one<float, true, true>(c + 6);
        if (e == cudaSuccess) e = setup_one<float, false, true>(c + 7);
        int sms = 0;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        g_device_sms[dev] = sms > 0 ? sms : 148;
        g_device_ready[dev].store(1, std::memory_order_release);
    }
    *sm_count = g_device_sms[dev];
    *ctas_per_sm = g_device_ctas[dev];
    return cudaSuccess;
}

template <typename T, bool NOISY, bool RAGGED>
void launch_stream(const UnmaskProblem& p, UnmaskPartial* partial, uint32_t* shared_words, int tiles_per_item, int select_state,
                   int* status, int resident_ctas, cudaStream_t st) {
    const int rows = p.sets.row_off[p.sets.n_sets];
    const int tiles_per_row = (p.vocab + kTile - 1) / kTile;
    const long long items = static_cast<long long>(rows) * ((tiles_per_row + tiles_per_item - 1) / tiles_per_item);
    // persistent: as many CTAs as fit on the SMs, fewer when there is not an item for every warp
    const long long fit = resident_ctas;
    const long long need = (items + kWarps - 1) / kWarps;
    const unsigned grid = static_cast<unsigned>(need < fit ? (need < 1 ? 1 : need) : fit);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = stream_smem_bytes<T, RAGGED>();
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    const int n_attr = overlap_launch_attribute(st, attr);
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    cudaLaunchKernelEx(&cfg, unmask_stream_kernel<T, NOISY, RAGGED>, static_cast<const T*>(p.logits), static_cast<const uint8_t*>(p.state),
                       p.sets, partial, p.vocab, tiles_per_item, p.temperature, p.block_idx, p.step, select_state,
                       static_cast<const uint32_t*>(p.step_counter), status, shared_words);
}

// Both entry points launch the same two kernels; only the home of the records differs.
// mode 0: unmasking step; 1: draft of Scaffold Speculative Decoding (every MASKED row becomes DRAFT);
// 2: its accept scan (rows in state DRAFT are read, then the scan runs).
// tiles_per_item: how many 2048-id tiles share one record slot (a row has ceil(tiles / tiles_per_item) slots).
cudaError_t launch_unmask_kernels(const UnmaskProblem& p, UnmaskPartial* partial, uint32_t* shared_words, int tiles_per_item, int dev,
                                  int* status, cudaStream_t st, int mode = 0) {
    const int select_state = mode == 2 ? FDD_DRAFT : FDD_MASKED;
    const int rows = p.sets.row_off[p.sets.n_sets];
    const int forks = p.sets.fork_off[p.sets.n_sets];
    if (rows > kMaxRows) return cudaErrorInvalidValue;
    int sm_count = 0;
    const int* per_sm = nullptr;
    cudaError_t e = device_setup(dev, &sm_count, &per_sm);
    if (e != cudaSuccess) return e;
    const int items_per_row = unmask_items_per_row(p.vocab, tiles_per_item);
    const bool noisy = p.temperature != 0.0f;
    // rows that all start on a 16-byte boundary (base and row pitch), or ragged ones
    const bool bf16 = p.logits_dtype == FDD_LOGITS_BF16;
    const bool ragged = p.vocab % (bf16 ? 8 : 4) != 0 || reinterpret_cast<uintptr_t>(p.logits) % 16 != 0;
    const int which = (ragged ? 4 : 0) + (bf16 ? 0 : 2) + (noisy ? 0 : 1);
    using Launch = void (*)(const UnmaskProblem&, UnmaskPartial*, uint32_t*, int, int, int*, int, cudaStream_t);
    static const Launch launches[8] = {
        launch_stream<__nv_bfloat16, true, false>, launch_stream<__nv_bfloat16, false, false>,
        launch_stream<float, true, false>, launch_stream<float, false, false>,
        launch_stream<__nv_bfloat16, true, true>, launch_stream<__nv_bfloat16, false, true>,
        launch_stream<float, true, true>, launch_stream<float, false, true>};
    launches[which](p, partial, shared_words, tiles_per_item, select_state, status, sm_count * per_sm[which], st);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(forks);
    cfg.blockDim = dim3(kFinalizeThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    cfg.numAttrs = overlap_launch_attribute(st, attr);
    cfg.attrs = attr;
    if (mode == 2) {
        cudaLaunchKernelEx(&cfg, ss_accept_kernel, static_cast<const UnmaskPartial*>(partial), p.tokens, p.state, p.n_committed,
                           p.n_left, p.sets, items_per_row, shared_words);
    } else {
        cudaLaunchKernelEx(&cfg, unmask_finalize_kernel, static_cast<const UnmaskPartial*>(partial), p.tokens, p.state,
                           p.n_committed, p.n_left, p.conf, p.sets, items_per_row, p.threshold,
                           mode == 1 ? static_cast<int>(FDD_DRAFT) : static_cast<int>(FDD_COMMITTED),
                           p.bump_counter ? p.step_counter : static_cast<uint32_t*>(nullptr), p.left_mirror, p.mirror_stamp, shared_words, p.gate_out);
    }
    e = cudaGetLastError();
    // (the words have to be zero for the next launch whatever became of the kernel that clears them)
    if (e != cudaSuccess) (void)cudaMemsetAsync(shared_words, 0, unmask_shared_bytes(rows), st);
    return e;
}

}  // namespace

// Scratch of a context: the shared words, then the records.
static int launch_rows(long long max_rows) { return static_cast<int>(max_rows < kMaxRows ? max_rows : kMaxRows); }   // a launch takes at most kMaxRows rows
size_t unmask_workspace_bytes(int vocab, int max_rows) {
    return unmask_shared_bytes(launch_rows(max_rows)) + static_cast<size_t>(launch_rows(max_rows)) * unmask_items_per_row(vocab, 1) * sizeof(UnmaskPartial);
}

cudaError_t launch_unmask(fdd_ctx* ctx, const UnmaskProblem& p, cudaStream_t st, int* n_launches, int mode) {
    *n_launches += 2;
    char* records = static_cast<char*>(ctx->ws_unmask) + unmask_shared_bytes(launch_rows(static_cast<long long>(ctx->cfg.max_forks) * ctx->cfg.max_block));
    return launch_unmask_kernels(p, reinterpret_cast<UnmaskPartial*>(records), static_cast<uint32_t*>(ctx->ws_unmask), 1, ctx->device, ctx->d_status, st, mode);
}

// -------------------------------------------------------------------------------------------------
// fdd_unmask_static: the same unmasking step for callers that must not allocate.
//
// Its scratch (the per (row, chunk) records) lives in a fixed device array that is part of the
// loaded library image, so the call needs no context, no fork set and no allocation of any kind.
// -------------------------------------------------------------------------------------------------
namespace {

constexpr int kStaticMaxRecords = FDD_UNMASK_STATIC_MAX_RECORDS;
constexpr int kStaticTilesPerItem = kUnmaskChunk / kUnmaskTile;    // one record slot per 8192 ids

// Held by every GPU that loads the library until the process exits (2 MiB).
static __device__ __align__(256) UnmaskPartial g_static_partials[kStaticMaxRecords];
static __device__ __align__(256) uint32_t g_static_shared[kSharedBars + kMaxRows];

// Device address of g_static_partials per device ordinal, resolved on first use.  In host code the
// array's name is only a handle for the runtime; the address a kernel can use must be asked for.
UnmaskPartial* g_static_ptr[kMaxDevices];
uint32_t* g_static_shared_ptr[kMaxDevices];
bool g_static_ready[kMaxDevices];

void put_error(char* err, size_t err_len, const char* text) {
    if (err && err_len) snprintf(err, err_len, "%s", text);
}

}  // namespace

extern "C" fdd_status fdd_unmask_static(const void* logits, int logits_dtype, int n_forks, int block_len,
                                        int vocab, int32_t* tokens, uint8_t* state, const uint64_t* seeds,
                                        float threshold, float temperature, uint32_t block_idx,
                                        uint32_t step, int32_t* n_committed, int32_t* n_left, float* conf,
                                        void* stream, char* err, size_t err_len) {
    CallRange range("fdd_unmask_static");
    if (!logits || !tokens || !state || !seeds || !n_committed || !n_left) {
        put_error(err, err_len, "fdd_unmask_static: a required pointer is NULL");
        return FDD_ERR_INVALID_ARG;
    }
    if (logits_dtype != FDD_LOGITS_F32 && logits_dtype != FDD_LOGITS_BF16) {
        put_error(err, err_len, "fdd_unmask_static: logits_dtype must be FDD_LOGITS_F32 or FDD_LOGITS_BF16");
        return FDD_ERR_INVALID_ARG;
    }
    if (n_forks < 1 || block_len < 1 || vocab < 1 || !(temperature >= 0.0f) || threshold != threshold) {
        put_error(err, err_len, "fdd_unmask_static: sizes must be >= 1, temperature >= 0, threshold not NaN");
        return FDD_ERR_INVALID_ARG;
    }
    if (block_len > 128) {
        put_error(err, err_len, "fdd_unmask_static: block_len above 128 is not supported");
        return FDD_ERR_UNSUPPORTED;
    }
    const long long n_rows = static_cast<long long>(n_forks) * block_len;
    if (n_rows > kUnmaskMaxRows) {
        if (err && err_len)
            snprintf(err, err_len, "fdd_unmask_static: n_forks * block_len = %lld exceeds the %d rows one call takes",
                     n_rows, kUnmaskMaxRows);
        return FDD_ERR_CAPACITY;
    }
    const long long records = n_rows * unmask_items_per_row(vocab, kStaticTilesPerItem);
    if (records > kStaticMaxRecords) {
        if (err && err_len)
            snprintf(err, err_len,
                     "fdd_unmask_static: n_forks * block_len * ceil(vocab / %d) = %lld exceeds the fixed scratch of %d records",
                     kUnmaskChunk, records, kStaticMaxRecords);
        return FDD_ERR_CAPACITY;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        put_error(err, err_len, "fdd_unmask_static: no usable current CUDA device");
        return FDD_ERR_CUDA;
    }
    if (!g_static_ready[dev]) {
        // once per device, with that device current: resolve the array's device address
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_partials);
        if (e != cudaSuccess || !p) {
            if (err && err_len) snprintf(err, err_len, "fdd_unmask_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
            return FDD_ERR_CUDA;
        }
        void* words = nullptr;
        e = cudaGetSymbolAddress(&words, g_static_shared);
        if (e != cudaSuccess || !words) {
            if (err && err_len) snprintf(err, err_len, "fdd_unmask_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
            return FDD_ERR_CUDA;
        }
        g_static_ptr[dev] = static_cast<UnmaskPartial*>(p);
        g_static_shared_ptr[dev] = static_cast<uint32_t*>(words);
        g_static_ready[dev] = true;
    }
    UnmaskProblem p;
    p.logits = logits; p.tokens = tokens; p.state = state;
    p.n_committed = n_committed; p.n_left = n_left; p.conf = conf;
    p.sets.n_sets = 1;
    p.sets.row_off[0] = 0; p.sets.row_off[1] = n_forks * block_len;
    p.sets.fork_off[0] = 0; p.sets.fork_off[1] = n_forks;
    p.sets.d[0] = block_len; p.sets.seeds[0] = seeds;
    p.vocab = vocab; p.logits_dtype = logits_dtype;
    p.threshold = threshold; p.temperature = temperature; p.block_idx = block_idx; p.step = step;
    e = launch_unmask_kernels(p, g_static_ptr[dev], g_static_shared_ptr[dev], kStaticTilesPerItem, dev, nullptr, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        if (err && err_len) snprintf(err, err_len, "fdd_unmask_static: launch failed: %s", cudaGetErrorString(e));
        return FDD_ERR_CUDA;
    }
    return FDD_OK;
}
