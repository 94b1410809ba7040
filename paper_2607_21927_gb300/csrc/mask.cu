// RIS mask sampler (paper, Methods, "Memory-Bounded Geometry Generation" and "Sampling
// Modes: Stochastic and Structural").
//
// Instead of one N x N boolean tensor per seed, every (mask, row) is expanded once into a
// causal bitmap row with all seeds OR-merged in registers (the paper's streaming merge,
// without ever holding a seed's mask), then compacted into ascending per-row key lists.
//
//   k_mask_bits : per (mask, row) CTA, per group of 4 keys: one Philox4x32-10 call per seed until every key
//                 of the warp's step is kept, the smallest word over the seeds against the
//                 threshold, then per 32-key word the forced window/anchors, Structural block
//                 clique and causal cut; writes the word and the row's key count.
//   k_mask_draws: index-draw sampler only: per (mask, row) CTA, the row's index draws of
//                 every seed (one Philox call = 4 draws), j = floor(u N / 2^32), kept when
//                 j < i by an atomic OR into the zeroed bitmap row; k_mask_bits then ORs the
//                 forced and clique keys into those words and counts the row.
//   k_scan_*    : exclusive scan of the counts into row_ptr (int64).
//   k_mask_fill : per (mask, row) warp, expands the bitmap row into ascending key indices.
//
// Integer-only; every decision is an exact comparison of a 32-bit word with a host-resolved
// 64-bit threshold, so the result is bit-exact across devices and hosts.
#include <cmath>
#include <cstdint>

#include "ris_internal.h"

namespace ris {
namespace {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32 -> 64-bit
// products (multipliers 0xD2511F53 on word 0, 0xCD9E8D57 on word 2) whose high halves are
// xored with the other counter words and the round key; the key advances by the Weyl
// constants (0x9E3779B9, 0xBB67AE85) after each round.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k0, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k1, (uint32_t)p0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// bits of a word at and above / at and below bit x (any x)
__device__ __forceinline__ uint32_t bits_from(int x) { return x <= 0 ? 0xFFFFFFFFu : x > 31 ? 0u : 0xFFFFFFFFu << x; }
__device__ __forceinline__ uint32_t bits_to(int x) { return x >= 31 ? 0xFFFFFFFFu : x < 0 ? 0u : 0xFFFFFFFFu >> (31 - x); }

__device__ __forceinline__ int64_t row_word_offset(int64_t i)
{
    const int64_t a = i >> 5, b = i & 31;
    return i + 16 * a * (a - 1) + a * b;
}

constexpr int kBitsThreads = 128;

// What the draws of one (mask, row) share: the row's counter words and the head key's schedule.
struct RowDraws {
    uint32_t i, layer, k1;  // counter word 1, counter word 3, key word 1
    uint32_t s_hi, s_lo;    // the product of round 1 on counter word 2 (the stream)
};

// Smallest word over the seeds s0 .. s1-1 of each of the 4 keys of the groups g .. g + U - 1 (keys
// 4 g .. 4 g + 4 U - 1): a key is kept by some seed iff this minimum is at most tm1. `forced`: the draws of these
// keys do not matter, and whatever is returned for them is kept. A warp whose keys are all kept leaves the loop
// over seeds: it asks after `first_vote` seeds and then every kVoteSeeds.
//
// Philox4x32-10 as in philox4x32_10 above, with what the 10 rounds of a row's calls have in common
// taken out of the loop over seeds (unrolled by SEEDS; 0: one seed in all, s0, without a loop or
// minima). Round 1 multiplies the group (word 0) and the stream (word 2), neither of which depends on the seed; its results z, w depend on the group only (key word 1 is
// the head key) and x, y on the row and seed only. So the second product of round 2 depends on the
// group only and the first on the seed only: per call 8 rounds of two products remain, 16 of 20.
constexpr int kVoteSeeds = 4;
template <int U, int SEEDS>
__device__ __forceinline__ void min_words(const MaskBitsArgs &a, const RowDraws &d, uint32_t g, int s0, int s1,
                                          uint32_t tm1, bool forced, int first_vote, uint32_t (&best)[U][4])
{
    uint32_t hx[U], y2[U], wz[U];  // x2 but for key word 0, y2, z2 but for the seed's product
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * (g + u);
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(p0 >> 32) ^ d.layer ^ d.k1);
        hx[u] = (uint32_t)(p1 >> 32) ^ d.s_lo;
        y2[u] = (uint32_t)p1;
        wz[u] = (uint32_t)p0 ^ (d.k1 + 0xBB67AE85u);
#pragma unroll
        for (int e = 0; e < 4; ++e) best[u][e] = SEEDS > 0 && forced ? 0u : 0xFFFFFFFFu;
    }
    auto seed_pass = [&](int s) {
        uint32_t k0 = a.seeds.v[s], k1 = d.k1 + 0xBB67AE85u;
        const uint64_t ps = (uint64_t)0xD2511F53u * (d.s_hi ^ d.i ^ k0);
        k0 += 0x9E3779B9u;
        uint4 c[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            c[u] = make_uint4(hx[u] ^ k0, y2[u], (uint32_t)(ps >> 32) ^ wz[u], (uint32_t)ps);
#pragma unroll
        for (int r = 2; r < 10; ++r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t p0 = (uint64_t)0xD2511F53u * c[u].x;
                const uint64_t p1 = (uint64_t)0xCD9E8D57u * c[u].z;
                c[u] = make_uint4((uint32_t)(p1 >> 32) ^ c[u].y ^ k0, (uint32_t)p1,
                                  (uint32_t)(p0 >> 32) ^ c[u].w ^ k1, (uint32_t)p0);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            best[u][0] = min(best[u][0], c[u].x);
            best[u][1] = min(best[u][1], c[u].y);
            best[u][2] = min(best[u][2], c[u].z);
            best[u][3] = min(best[u][3], c[u].w);
        }
    };
    if constexpr (SEEDS == 0) {
        seed_pass(s0);
    } else {
        int s = s0, stop = min(s1, s0 + first_vote);
        for (;;) {
#pragma unroll SEEDS
            for (; s < stop; ++s) seed_pass(s);
            if (s >= s1) break;
            uint32_t worst = 0u;
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < 4; ++e) worst = max(worst, best[u][e]);
            if (__all_sync(0xFFFFFFFFu, worst <= tm1)) break;
            stop = min(s1, s + kVoteSeeds);
        }
    }
}

// A (mask, row) of the launch: its bitmap row, its words and drawn groups, its forced keys.
struct RowTask {
    uint32_t *row;
    int i, nw, ng, tail0, last;
    int s0, s1;    // its seeds
    uint32_t tm1;  // u < thr for thr in [1, 2^32] is u <= thr - 1 in 32 bits
    RowDraws d;
};

__device__ __forceinline__ RowTask row_task(const MaskBitsArgs &a, uint32_t m, int i)
{
    const bool one = a.single_row >= 0;
    RowTask t;
    t.i = i;
    t.s0 = a.per_seed ? (int)m / a.heads_keyed : 0;
    t.s1 = a.per_seed ? t.s0 + 1 : a.n_seeds;
    t.row = a.bitmap + (int64_t)m * a.words_per_mask + (one ? 0 : row_word_offset(i));
    // forced keys: local window (i-W, i], anchors [0, A), Structural clique [block start, i]; the draws
    // matter for j < i before the first and the last
    t.tail0 = i - a.W + 1;
    if (a.mode == RIS_MODE_STRUCTURAL) t.tail0 = min(t.tail0, (int)((uint32_t)i / (uint32_t)a.B * (uint32_t)a.B));
    t.last = one ? i - 1 : i;  // a single row keeps keys j < i only
    t.nw = (i >> 5) + 1;
    t.ng = a.thr > 0 ? (max(0, min(i, t.tail0)) + 3) >> 2 : 0;
    t.tm1 = a.thr > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)(a.thr - 1);
    t.d.i = (uint32_t)i;
    t.d.layer = a.layer_key;
    t.d.k1 = (a.heads_keyed > 1) ? m % (uint32_t)a.heads_keyed : 0u;
    const uint64_t ps = (uint64_t)0xCD9E8D57u * a.stream;
    t.d.s_hi = (uint32_t)(ps >> 32);
    t.d.s_lo = (uint32_t)ps;
    return t;
}

// One warp, 16 words (512 keys) from word w0 on: lane l takes the 16 keys of half a word, groups
// 4 l .. 4 l + 3 of the step's 128, and its neighbour the other half. Returns the lane's kept keys.
template <int SEEDS>
__device__ __forceinline__ int row_step(const MaskBitsArgs &a, const RowTask &t, int w0, int lane, int first_vote)
{
    uint32_t word = 0u;
    if (8 * w0 < t.ng && 32u * (uint32_t)(w0 + 16) > (uint32_t)a.A) {  // some key of the step is not forced
        uint32_t best[4][4];
        const int g = 8 * w0 + 4 * lane;
        const bool forced = g >= t.ng || 4u * (uint32_t)(g + 4) <= (uint32_t)a.A;
        min_words<4, SEEDS>(a, t.d, (uint32_t)g, t.s0, t.s1, t.tm1, forced, first_vote, best);
#pragma unroll
        for (int e = 0; e < 16; ++e) word |= best[e >> 2][e & 3] <= t.tm1 ? 1u << e : 0u;
    }
    word |= __shfl_down_sync(0xFFFFFFFFu, word, 1) << 16;
    const int w = w0 + (lane >> 1);
    if ((lane & 1) != 0 || w >= t.nw) return 0;
    const int j0 = w << 5;
    uint32_t bits = word & bits_to(t.i - 1 - j0);  // drawn pairs are j < i
    if (a.or_existing) bits |= t.row[w];
    bits = (bits | bits_from(t.tail0 - j0) | bits_to(a.A - 1 - j0)) & bits_to(t.last - j0);
    t.row[w] = bits;
    return __popc(bits);
}

// One CTA per (mask, row), rows from the last (longest) to the first, its warps 16 words apart.
//
// Bound by the 32 x 32 -> 64-bit products (32 lanes per clock and SM, a quarter of the fp32 rate)
// and, nearly as much, by the ALU pipe (an exclusive or per product, the minima, the key schedule).
// SEEDS = 2, two or more seeds: two a pass and as many registers as the compiler wants, which keeps the key schedules
// in registers (N = 16384 of 1%, against one a pass and eight CTAs per SM: 2 seeds 209 / 217 us, 3 283 / 297, 8 641 /
// 693, 20 1487 / 1644). 70 seeds at N = 32768 take 19.6 ms, 1.5 calls per clock and SM (21.1 one a pass, 29.0
// with rounds 1 and 2 in the loop over seeds and a thread per word). SEEDS = 0, one seed: eight CTAs
// per SM, as a row's other work counts.
template <int SEEDS>
__global__ void __launch_bounds__(kBitsThreads, SEEDS > 0 ? 1 : 8) k_mask_bits(const MaskBitsArgs a, int first_vote)
{
    const uint32_t m = blockIdx.x % (uint32_t)a.n_masks;
    const bool one = a.single_row >= 0;
    const int i = (int)(one ? a.single_row : a.N - 1 - blockIdx.x / (uint32_t)a.n_masks);  // below 2^31
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const RowTask t = row_task(a, m, i);
    int count = 0;
    for (int w0 = 16 * warp; w0 < t.nw; w0 += 16 * (kBitsThreads / 32)) count += row_step<SEEDS>(a, t, w0, lane, first_vote);
    // block reduction of the row count
    __shared__ int red[kBitsThreads / 32];
    count = __reduce_add_sync(0xFFFFFFFFu, count);
    if (lane == 0) red[warp] = count;
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = 0;  // a row holds at most 2^31 - 1 keys
#pragma unroll
        for (int k = 0; k < kBitsThreads / 32; ++k) n += red[k];
        a.counts[one ? (int64_t)m : (int64_t)m * a.N + i] = n;
    }
}

// One seed per mask and rows enough for four of them per CTA (the caller sees to both): the steps of
// the four rows one after the other, dealt to the warps in turn. With one call per four keys a CTA's
// start, its last step and its end are a good part of a short row: ten one-seed masks of N = 8192 take
// 345 us (360 with a row per CTA, 367 with the loop over seeds besides), one of N = 16384 121-127 (130, 138).
constexpr int kOneSeedRows = 4;
__global__ void __launch_bounds__(kBitsThreads, 6) k_mask_bits_one(const MaskBitsArgs a)
{
    const uint32_t tasks = (uint32_t)(a.N * a.n_masks), t0 = blockIdx.x * (uint32_t)kOneSeedRows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int total[kOneSeedRows];
    if (threadIdx.x < kOneSeedRows) total[threadIdx.x] = 0;
    __syncthreads();
    int at = warp;  // the warp's next step, from the start of row q
#pragma unroll 1
    for (int q = 0; q < kOneSeedRows && t0 + q < tasks; ++q) {
        const uint32_t r = (t0 + q) / (uint32_t)a.n_masks, m = t0 + q - r * (uint32_t)a.n_masks;
        const int i = (int)(a.N - 1 - r), steps = ((i >> 5) + 16) >> 4;
        if (at < steps) {
            const RowTask t = row_task(a, m, i);
            int count = 0;
            for (; at < steps; at += kBitsThreads / 32) count += row_step<0>(a, t, 16 * at, lane, 0);
            count = __reduce_add_sync(0xFFFFFFFFu, count);
            if (lane == 0) atomicAdd(&total[q], count);
        }
        at -= steps;
    }
    __syncthreads();
    if (threadIdx.x < kOneSeedRows && t0 + threadIdx.x < tasks) {
        const uint32_t t = t0 + threadIdx.x, r = t / (uint32_t)a.n_masks;
        a.counts[(int64_t)(t - r * (uint32_t)a.n_masks) * a.N + (a.N - 1 - r)] = total[threadIdx.x];
    }
}

constexpr int kDrawThreads = 128;

__global__ void __launch_bounds__(kDrawThreads) k_mask_draws(const MaskBitsArgs a)
{
    const int64_t r = (int64_t)blockIdx.x;
    const int32_t m = (int32_t)(r % a.n_masks);
    const bool one = a.single_row >= 0;
    const int64_t i = one ? a.single_row : a.N - 1 - r / a.n_masks;
    if (i == 0) return;  // no j < 0
    const uint32_t head_key = (a.heads_keyed > 1) ? (uint32_t)(m % a.heads_keyed) : 0u;
    const int32_t s0 = a.per_seed ? m / a.heads_keyed : 0;
    const int32_t s1 = a.per_seed ? s0 + 1 : a.n_seeds;
    uint32_t *row = a.bitmap + (int64_t)m * a.words_per_mask + (one ? 0 : row_word_offset(i));
    const int64_t groups = (a.draws + 3) >> 2;
    const uint64_t n = (uint64_t)a.N;
    for (int32_t s = s0; s < s1; ++s) {
        const uint32_t seed = a.seeds.v[s];
        for (int64_t g = threadIdx.x; g < groups; g += kDrawThreads) {
            const uint4 u = philox4x32_10(make_uint4((uint32_t)g, (uint32_t)i, a.stream + 2u, a.layer_key), seed,
                                          head_key);
            const uint32_t w4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (4 * g + c >= a.draws) break;
                const int64_t j = (int64_t)(((uint64_t)w4[c] * n) >> 32);
                if (j < i) atomicOr(row + (j >> 5), 1u << (j & 31));
            }
        }
    }
}

// ---------------------------------------------------------------- exclusive scan (int64)
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;
constexpr int64_t kScanTile = (int64_t)kScanThreads * kScanPer;

// Block-level inclusive scan of a tile of kScanTile elements held kScanPer per thread.
__device__ __forceinline__ int64_t block_inclusive(int64_t v, int64_t *smem)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) smem[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int64_t w = smem[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= o) w += t;
        }
        smem[lane] = w;
    }
    __syncthreads();
    if (warp > 0) v += smem[warp - 1];
    return v;
}

// In-place inclusive scan of x[0, n) by one CTA, tile after tile: one launch where the three below
// would have a tile or two (n = 3001: 4.8 us instead of 10; four tiles, 14.8 us, are as slow).
constexpr int64_t kScanOneTiles = 2;
__global__ void __launch_bounds__(kScanThreads) k_scan_one(int64_t *x, int64_t n)
{
    __shared__ int64_t smem[32];
    __shared__ int64_t total;
    int64_t carry = 0;
    for (int64_t t0 = 0; t0 < n; t0 += kScanTile) {
        const int64_t base = t0 + (int64_t)threadIdx.x * kScanPer;
        int64_t vals[kScanPer];
        int64_t sum = 0;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            vals[e] = (base + e < n) ? x[base + e] : 0;
            sum += vals[e];
        }
        const int64_t incl = block_inclusive(sum, smem);
        int64_t run = carry + incl - sum;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            run += vals[e];
            if (base + e < n) x[base + e] = run;
        }
        if (threadIdx.x == kScanThreads - 1) total = incl;
        __syncthreads();
        carry += total;
        __syncthreads();
    }
}

// In-place inclusive scan of each tile of x[0, n); tile totals to partials[tile].
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(int64_t *x, int64_t n, int64_t *partials)
{
    __shared__ int64_t smem[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
    int64_t vals[kScanPer];
    int64_t sum = 0;
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
        vals[e] = (base + e < n) ? x[base + e] : 0;
        sum += vals[e];
    }
    const int64_t incl = block_inclusive(sum, smem);
    int64_t run = incl - sum;
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
        run += vals[e];
        if (base + e < n) x[base + e] = run;
    }
    if (threadIdx.x == kScanThreads - 1) partials[blockIdx.x] = incl;
}

// Single-CTA exclusive scan of the tile totals (any count, in chunks with a carry).
__global__ void __launch_bounds__(kScanThreads) k_scan_partials(int64_t *p, int64_t n)
{
    __shared__ int64_t smem[32];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t b = 0; b < n; b += kScanThreads) {
        const int64_t idx = b + threadIdx.x;
        const int64_t v = idx < n ? p[idx] : 0;
        const int64_t incl = block_inclusive(v, smem);
        const int64_t c = carry;
        if (idx < n) p[idx] = c + incl - v;
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1) carry = c + incl;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(int64_t *x, int64_t n, const int64_t *partials)
{
    const int64_t add = partials[blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    for (int e = threadIdx.x; e < kScanTile; e += kScanThreads)
        if (base + e < n) x[base + e] += add;
}

// ---------------------------------------------------------------- CSR fill
constexpr int kFillThreads = 128;

// One warp per (mask, row), a word per lane and step, the next step's words in flight meanwhile. (A CTA
// per row, with two barriers per 128 words, took 79 us for ten one-seed masks of N = 8192.)
template <typename TIdx>
__global__ void __launch_bounds__(kFillThreads) k_mask_fill(const MaskFillArgs a, int64_t n_tasks)
{
    const int64_t r = (int64_t)blockIdx.x * (kFillThreads / 32) + (threadIdx.x >> 5);
    if (r >= n_tasks) return;
    const uint32_t m = (uint32_t)r % (uint32_t)a.n_masks;  // below 2^31
    const bool one = a.single_row >= 0;
    const int64_t i = one ? a.single_row : a.N - 1 - (uint32_t)r / (uint32_t)a.n_masks;
    const int nw = (int)(i >> 5) + 1;
    const uint32_t *row = a.bitmap + (int64_t)m * a.words_per_mask + (one ? 0 : row_word_offset(i));
    TIdx *col = reinterpret_cast<TIdx *>(a.col) + a.row_ptr[one ? (int64_t)m : (int64_t)m * a.N + i];
    const int lane = threadIdx.x & 31;
    uint32_t next = lane < nw ? row[lane] : 0u;
    for (int w0 = 0; w0 < nw; w0 += 32) {
        const int w = w0 + lane;
        uint32_t bits = next;
        next = w + 32 < nw ? row[w + 32] : 0u;
        const int c = __popc(bits);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        TIdx *dst = col + (incl - c);
        while (bits) {
            *dst++ = (TIdx)((w << 5) + __ffs(bits) - 1);
            bits &= bits - 1;
        }
        col += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
}

}  // namespace

cudaError_t launch_mask_bits(const MaskBitsArgs &a, cudaStream_t s)
{
    const int64_t blocks = (int64_t)a.n_masks * (a.single_row >= 0 ? 1 : a.N);
    const int seeds = a.per_seed ? 1 : a.n_seeds;
    // four rows per CTA only if that leaves sixteen CTAs per SM: below, rows in flight count for more
    // (N = 2048, one seed: 7.3 us against 6.4)
    // Seeds after which one warp step of 512 keys in e^3 is full: 512 (1 - hit)^s = 3, hit the chance that a
    // seed keeps a key. Asking costs about a tenth of a seed's pass, so sparse masks (1%: 512 seeds) never ask,
    // and dense ones first where it may help. Mask of N = 8192, every seed drawn / asking: 50% x 256 seeds
    // 4.86 / 0.54 ms, 10% x 256 4.86 / 1.52, 30% x 70 1.53 / 0.67, 10% x 70 1.54 / 1.42; 1% x 70 with every key an
    // anchor 1.53 / 0.29. (A skip per group of four keys and thread: 1.24, 2.31, 0.85, 1.73; 0.46.)
    const double hit = (double)a.thr / 4294967296.0;
    const double full = hit >= 1.0 ? 1.0 : std::ceil(std::log(512.0 / 3.0) / -std::log1p(-hit));
    const int first_vote = a.thr == 0 || full > kMaxSeeds ? kMaxSeeds : (int)full;
    if (seeds == 1 && a.single_row < 0 && blocks >= (int64_t)kOneSeedRows * 16 * 152)
        k_mask_bits_one<<<(unsigned)((blocks + kOneSeedRows - 1) / kOneSeedRows), kBitsThreads, 0, s>>>(a);
    else if (seeds == 1)
        k_mask_bits<0><<<(unsigned)blocks, kBitsThreads, 0, s>>>(a, first_vote);
    else
        k_mask_bits<2><<<(unsigned)blocks, kBitsThreads, 0, s>>>(a, first_vote);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mask_draws(const MaskBitsArgs &a, cudaStream_t s)
{
    const int64_t blocks = (int64_t)a.n_masks * (a.single_row >= 0 ? 1 : a.N);
    k_mask_draws<<<(unsigned)blocks, kDrawThreads, 0, s>>>(a);
    note_launch();
    return cudaGetLastError();
}

int64_t scan_partials_count(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

cudaError_t launch_scan_inplace(int64_t *x, int64_t n, int64_t *partials, cudaStream_t s)
{
    const int64_t tiles = scan_partials_count(n);
    if (tiles <= kScanOneTiles) {
        k_scan_one<<<1, kScanThreads, 0, s>>>(x, n);
        note_launch();
        return cudaGetLastError();
    }
    k_scan_tiles<<<(unsigned)tiles, kScanThreads, 0, s>>>(x, n, partials);
    k_scan_partials<<<1, kScanThreads, 0, s>>>(partials, tiles);
    k_scan_add<<<(unsigned)tiles, kScanThreads, 0, s>>>(x, n, partials);
    note_launch(3);
    return cudaGetLastError();
}

cudaError_t launch_mask_fill(const MaskFillArgs &a, cudaStream_t s)
{
    const int64_t tasks = (int64_t)a.n_masks * (a.single_row >= 0 ? 1 : a.N);
    const unsigned blocks = (unsigned)((tasks + kFillThreads / 32 - 1) / (kFillThreads / 32));
    if (a.col_bytes == 2)
        k_mask_fill<uint16_t><<<blocks, kFillThreads, 0, s>>>(a, tasks);
    else
        k_mask_fill<uint32_t><<<blocks, kFillThreads, 0, s>>>(a, tasks);
    note_launch();
    return cudaGetLastError();
}

}  // namespace ris
