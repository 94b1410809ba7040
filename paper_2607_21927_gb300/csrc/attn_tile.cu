// RIS sparse attention, masked dense-tile design on the 5th-generation tensor cores
// (paper, Methods, "Hybrid Anchor and Pre-Fusion Unified Softmax (PFUS)"; the dense causal
// upper bound of Table tab:results_32k is the same kernel with every causal pair kept).
//
// Where the master mask keeps a large share of the causal pairs (union densities of tens of
// percent, and the dense mode) a dense 128 x 128 score tile with the mask applied as -inf
// beats gathering rows pair by pair. One CTA owns one (128-query tile, query head, set). At head
// dim 128 two CTAs form a cluster that shares its key and value tiles (two heads of a KV group, or
// two query tiles where a group has an odd number of heads) and runs every product as one
// 256-row product over both SMs (see Lay):
//
//   warp 8 (TMA)    loads the query tile, then streams 128-key tiles of the keys (hi parts and
//                   corrections) and of the values (fp16) in 128-byte swizzled boxes into two
//                   shared-memory rings, each CTA its half: a key stage is refilled as soon as its
//                   score products are done, a value stage once its value product is. The copies
//                   of both CTAs complete on barriers of the first;
//   warp 11 (relay) (of the cluster's first CTA) passes what has landed on to the barriers of the
//                   issuing warps;
//   warps 9, 10     (of the cluster's first CTA) issue tcgen05.mma: warp 9 the score tile S (query
//                   and keys from shared memory) into a double-buffered TMEM score tile, warp 10
//                   O += P V (A = P as fp16 in TMEM, double-buffered) into the TMEM output tile,
//                   committing each step to an mbarrier of both CTAs. TMEM holds S (2 x 128
//                   columns), O (128) and P (2 x 64), all 512 columns. P has columns of its own,
//                   so the scores of tile j + 2 start as soon as those of tile j have been read;
//   warps 0-7       two groups of four warps, one thread per query row in each, taking alternate
//                   tiles: per tile tcgen05.ld the row's 128 scores, apply the bitmap (words
//                   fetched four tiles ahead) or the causal cut, take the row max, fp32 online
//                   softmax from the reference maximum that the other group hands over, with lazy
//                   rescaling of O in TMEM (only when the row max grows by more than 2^8), write P
//                   into TMEM, and at the end normalise O (and undo the values' power-of-two
//                   scale) and store it, coalesced, through shared memory.
//
// Precision. With activation outlier channels the scores reach tens of units while the
// output moves by p (v_j - o) per unit of score error, so the scores need about 17
// significant bits. At head dim 128 with rotated inputs (the operands written by
// launch_fp8_prep) S = q_h k_h + 2^-12 (e4m3(q_h) e4m3(k_l) + e4m3(q_l) e4m3(k_h)) with fp16
// hi parts and power-of-two scales taken from bounds of |q~| and |k~| (fp8_score_scales): the
// two e4m3 products (kind::f8f6f4, twice the rate) go first and the fp16 product folds them in
// with scale-input-d; max-abs about 7e-3 in CPU emulation. Where the bounds rule that out, at
// head dim 64, and for inputs not rotated here, S = Q_hi K_hi^T + Q_lo K_hi^T + Q_hi K_lo^T
// with bf16 hi + lo pairs. One fp16 key product alone moves outputs by up to 0.1. P enters the
// value product as one fp16 (11 significant bits; max-abs 6.5e-3 in the same emulation
// against 1.7e-3 for a bf16 hi + lo pair), and the row sum adds P as rounded, so that each
// weight's rounding moves the output by at most 2^-11 of that weight times |v_j - o|. The
// values are exact in fp16 after a power-of-two scale (none unless some |v| reaches 2^14),
// undone in the epilogue.
//
// What bounds it: a tile takes 24 products of 128 x 128 x 16 slots (8 fp16 score products, 2 x 4
// e4m3 corrections at twice the rate, 8 fp16 value products), 1,536 cycles of the tensor pipe. A
// dense 32k layer takes about 1,650 cycles per tile: the pipe is 95% busy and the power limit holds
// the clock at 1.58 GHz. With a bitmap (64k, 10%) 1,870, where the softmax with about 450 cycles of masking is
// as slow as the pipe. Layer calls: N = 8192 226 us, 32k dense 2.9 ms, 64k 11.4 ms.
// Why it is laid out so (in brackets cycles per tile of the dense / the masked layer from clock64()
// stamps, or a layer's time, the other way against this one):
//   - products are issued with warp-uniform operands by an elected lane: inside a branch on the lane
//     each costs the issuing lane about 60 cycles of operand moves, as long as the product itself
//     (2,485 / 2,650, against 2,055 / 2,400);
//   - two softmax groups on alternate tiles, half a period apart: with two threads per row on every
//     tile their meeting set the pace (2,055 / 2,400, against 1,860 / 2,040);
//   - key and value tiles shared by two SMs: 96 KB per tile and SM, 17 TB/s at this pace, come in too
//     late (2,030 / 2,170, against 1,720 / 1,985);
//   - P double-buffered, in columns of its own (1,720 / 1,985, against 1,620 / 1,950);
//   - the reference maximum is handed over after the exponentials, and O rescaled after that: the groups' warps
//     of a scheduler otherwise run their exponentials against each other, and a warp in a hundred
//     that rescales O holds up seven others (N = 8192: 230, against 226 us);
//   - the reference maximum moves at 2^8: at 2^14 the heaviest weight of a row is less often exactly 1, and
//     the log-sum-exp of a dense 32k layer is 5% further off;
//   - row sums that add fp16 as it is, -infinity by predicated moves, the next tile's scores polled for
//     ahead of their use (masked 1,950, against 1,870; a dense layer is not held by the softmax). The
//     bitmap applied to P as packed masks has fewer instructions, but they lie in the chain of
//     exponentials from group to group (N = 8192: 244, against 226 us);
//   - waits of the softmax warps on products are relaxed at cluster scope: acquiring there takes a masked
//     layer 1.2-1.5% longer;
//   - the query tile by TMA and the output through shared memory: with rows loaded and stored 16 bytes per
//     lane a CTA's start and end take 16,000 cycles instead of 7,000.
//
// The suffix pass of the dense-suffix split (SUFFIX) runs the same pipeline over the key
// tiles of each row's dense suffix only (its Structural block and / or local window: every key
// kept, no bitmap), and writes the normalised partial output and its log-sum-exp for the
// register gather to continue from.
//
// Every mbarrier wait is bounded; a wait that gives up sets bit 1 of the device error word,
// every role falls through to the end, TMEM is released and the CTA returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "attn_common.cuh"

namespace ris {

// Device error word of this kernel (bit 1: a bounded wait gave up); read by read_tile_error.
__device__ unsigned int g_ris_tile_error;

namespace {

constexpr int BM = 128;          // query rows per tile (TMEM lanes)
constexpr int BN = 128;          // keys per stage
// Softmax: two groups of four warps, one thread per query row in each (4 warps cover the 128
// TMEM lanes); group x takes the tiles of parity x. The two groups run half a period apart, so
// that one fills the issue slots while the other waits (for scores, TMEM loads and stores,
// barriers), and no thread has to meet a partner inside a tile. Then the TMA and MMA warps, in a
// warpgroup of their own that hands most of its registers to the softmax threads, whose 128
// scores of a tile stay in registers.
constexpr int kGroupWarps = 4;
constexpr int kSoftmaxWarps = 2 * kGroupWarps;
constexpr int kTmaWarp = kSoftmaxWarps, kScoreWarp = kSoftmaxWarps + 1, kValueWarp = kSoftmaxWarps + 2,
              kRelayWarp = kSoftmaxWarps + 3;
constexpr int kThreads = 32 * (kSoftmaxWarps + 4);
// registers per thread: at launch, then after setmaxnreg of a softmax and of a loader / MMA thread
constexpr int kRegs = 168, kSoftmaxRegs = 200, kOtherRegs = 104;
static_assert(2 * kSoftmaxRegs + kOtherRegs == 3 * kRegs, "the shares of the three warpgroups add up to the launch's");
// The reference maximum of a row moves only when its maximum grows by more than this (log2), so P
// stays below 2^8. On a 10% mask of 64k tokens one warp in a hundred rescales O in a tile.
constexpr float kLazyLog2 = 8.f;
constexpr uint32_t kTmemCols = 512;  // S (2 x 128) + O (128) + P (2 x 64)

// How the kernel of head dim DT (128 or 64) is laid out. At 128 two CTAs of a cluster share their
// key and value tiles (CG = 2: tcgen05 cta_group::2, one 256 x 128 product over both SMs, each
// holding half of the B operand: 64 of a tile's keys, 64 of the head dim's value columns). That
// halves the L2 traffic of the tiles (96 KB per tile and SM would be near the L2's whole
// bandwidth at the tensor pipe's rate) and leaves shared memory for a key ring of four stages, past
// the latency of a load, beside the query tile. At 64 the halves of the value columns would be
// 64-byte rows; each CTA works for itself there.
//
// Shared memory (bytes, from a 1024-aligned base): the K ring, the V ring, the query tile (hi part,
// low part), then the barriers, the TMEM base, the notes for the end and what the two softmax groups
// hand to each other for a row: its reference maximum after each tile, and at the end each group's
// row sum over its tiles and the maximum that sum refers to.
template <int DT>
struct Lay {
    static constexpr int CG = DT == 128 ? 2 : 1;
    static constexpr int NSK = 4, NSV = 2;       // stages of the key and of the value ring
    static constexpr int NB = DT / 64;           // 64-column blocks of a row
    static constexpr int KROWS = BN / CG;        // keys of a tile held by one CTA
    static constexpr int K_BLK = KROWS * 128;    // one 64-column block of K hi or K lo
    static constexpr int K_ARR = NB * K_BLK;     // K hi or K lo
    static constexpr int K_STAGE = 2 * K_ARR;
    static constexpr int V_BLK = BN * 128;
    static constexpr int V_STAGE = NB / CG * V_BLK;
    static constexpr int Q_BLK = BM * 128;
    static constexpr int OFF_K = 0;
    static constexpr int Q_ARR = NB * Q_BLK;     // Q hi or Q lo
    static constexpr int OFF_V = NSK * K_STAGE;
    static constexpr int OFF_Q = OFF_V + NSV * V_STAGE;
    static constexpr int OFF_BARS = OFF_Q + 2 * Q_ARR;
    static constexpr int OFF_TMEM = OFF_BARS + 192;  // after the barriers
    static constexpr int OFF_END = OFF_TMEM + 4;     // ClosingNotes
    static constexpr int OFF_M = OFF_BARS + 256;     // float [BM]
    static constexpr int OFF_ML = OFF_M + BM * 4;    // float2 [2][BM]
    static constexpr int BYTES = OFF_ML + 2 * BM * 8;
    static_assert(BYTES <= 232448, "shared memory of a CTA");
    // Barriers, one of each kind per ring stage (a tile's stage is its number mod NSK or NSV), so
    // that no waiter can fall two phases behind a barrier it polls by parity:
    //   Q_FULL          the query tiles have landed (relayed with the first keys)
    //   K_FULL, V_FULL  a tile's keys / values have landed (relayed to S_GO / P_GO)
    //   S_GO            the score products of a tile may start: its keys have landed and the scores
    //                   of the tile two before (if any) have been read out of their buffer
    //   S_FULL          they are done (and the key stage is free)
    //   P_GO            the value product may start: P is written and the values have landed
    //   PV_DONE         it is done (P's buffer and the value stage are free, O has settled)
    // S_FULL and PV_DONE of each CTA get the products' completion. The others are used in the
    // cluster's first CTA, whose warps issue the products: the loaders of both CTAs announce
    // their copies there and the copies complete there (each half of a tile to K_FULL or
    // V_FULL), and the softmax warps of both arrive there.
    //
    // What one CTA tells the other is ordered at cluster scope: a copy's completion releases what it
    // wrote, the relay acquires it and hands it on to the issuing warps of its own CTA; tensor
    // memory that was read or written is ordered by the tcgen05 waits and fences around the arrival and
    // the wait, which themselves need no more than the scope (see mbar_arrive_cluster).
    static constexpr int B_Q_FULL = 0, B_K_FULL = 1, B_S_GO = B_K_FULL + NSK, B_S_FULL = B_S_GO + NSK,
                         B_V_FULL = B_S_FULL + NSK, B_P_GO = B_V_FULL + NSV, B_PV_DONE = B_P_GO + NSV,
                         NBAR = B_PV_DONE + NSV;
    static_assert(NBAR * 8 <= 192, "barriers below the TMEM base word");
};

// What the warps of a cluster leave in each of its CTAs for the end of the kernel.
struct ClosingNotes {
    uint32_t bad;        // a wait gave up in either CTA
    uint32_t scored;     // tiles whose score products were issued and committed
    uint32_t valued;     // tiles whose value products were
    uint32_t keys[2], values[2];  // tiles whose keys / values each CTA requested (in the first CTA)
};
static_assert(4 + sizeof(ClosingNotes) <= 256 - 192, "in the barriers' block");
// the head-dim-128 layout (232,192 of the 232,448 bytes a CTA can have) is requested at either
// head dim: it keeps one CTA per SM, as the CTA holds all 512 TMEM columns
constexpr int SMEM_BYTES = Lay<128>::BYTES;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrival on a barrier of any CTA of the cluster (shared::cluster address, see cluster_addr). What
// it announces is tensor memory that was read or written, which tcgen05.wait and the tcgen05 fences on
// both sides order, and nothing that this thread read or wrote itself: relaxed. (Releasing its
// accesses at cluster scope took 1,000 cycles and more per arrival: 3,130 cycles a tile of a 32k dense
// layer instead of 1,720.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
    return d;
}
// *word = x in CTA `rank` of the cluster (word: the shared-memory address in this CTA)
__device__ __forceinline__ void st_cluster(uint32_t word, uint32_t rank, uint32_t x)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(word, rank)), "r"(x) : "memory");
}
// All threads of the cluster's CTAs.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
// Announce `bytes` to come on the barrier; CG = 2: a barrier of either CTA (shared::cluster address),
// relaxed, as nothing of this thread's is handed over.
template <int CG>
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    if constexpr (CG == 1)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    else
        asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                     : "memory");
}
// Waits acquire at the scope of those who arrive: the cluster's two CTAs and their copies (CG = 2). TMEM:
// what is waited for is tensor memory that products read or wrote, which the tcgen05 fence after the
// wait orders; relaxed, at the same scope.
template <int CG, bool TMEM = false>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if constexpr (CG == 2 && TMEM)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    else if constexpr (CG == 1)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    return ok != 0;
}
// Bounded wait for asynchronous work already issued (copies or products): about 2^31 cycles at most,
// whatever other CTAs reported.
template <int CG>
__device__ __forceinline__ bool mbar_wait_own(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    while (!mbar_try_wait<CG>(bar, parity))
        if (clock64() - t0 > (1LL << 31)) return false;
    return true;
}

// Whether the phase has completed by now: asked ahead of the wait, so that a completed one costs
// no round trip to the barrier at the point of use
template <int CG, bool TMEM = false>
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if constexpr (CG == 2 && TMEM)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    else if constexpr (CG == 1)
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    return ok != 0;
}

// Bounded wait (`limit` cycles, about 2^31 unless a test lowers it); false if the phase did
// not complete in time or another CTA already gave up.
template <int CG, bool TMEM = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit)
{
    if (mbar_try_wait<CG, TMEM>(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait<CG, TMEM>(bar, parity)) {
        if (clock64() - t0 > limit) return false;
        if (*reinterpret_cast<volatile unsigned int *>(&g_ris_tile_error) != 0u) return false;
    }
    return true;
}

// Copy a box into this CTA's shared memory. CG = 2: complete on a barrier of either CTA of the pair.
template <int CG>
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar)
{
    if constexpr (CG == 2)
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
        "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
    else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// ---- tcgen05 helpers
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptors, K-major or MN-major, 128-byte swizzle, version 1: the high
// word (stride byte offset 1024) is the same for all of them, the low word holds the address and
// the leading byte offset.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo)
{
    return ((addr >> 4) & 0x3FFFu) | ((lbo >> 4) << 16);
}
// What an offset of `bytes` (a multiple of 16; no carry out of the 14-bit address field, which
// covers all of shared memory) adds to a descriptor's low word.
__device__ __forceinline__ constexpr uint32_t dstep(int bytes) { return (uint32_t)bytes >> 4; }

// True in one lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xFFFFFFFF;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// Instruction descriptor, kind::f16: fp16 x fp16 -> f32, dense.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool b_mn_major)
{
    return (1u << 4)                      // D format f32 (A and B format 0: fp16)
           | ((b_mn_major ? 1u : 0u) << 16)
           | ((uint32_t)(N >> 3) << 17)
           | ((uint32_t)(M >> 4) << 24);
}

// Instruction descriptor, kind::f16: bf16 x bf16 -> f32, dense.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool b_mn_major)
{
    return (1u << 4)                      // D format f32
           | (1u << 7)                    // A bf16
           | (1u << 10)                   // B bf16
           | ((b_mn_major ? 1u : 0u) << 16)
           | ((uint32_t)(N >> 3) << 17)
           | ((uint32_t)(M >> 4) << 24);
}

// A operand from TMEM (rows in lanes, 16-bit values packed two per column), B from shared memory.
template <int CG>
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b, uint32_t idesc, uint32_t acc)
{
    if constexpr (CG == 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
    else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// kind::f8f6f4 (e4m3 x e4m3 with the instruction descriptor's format fields 0), A and B from
// shared memory.
template <int CG>
__device__ __forceinline__ void tc_mma_ss_f8(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc)
{
    if constexpr (CG == 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
    else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// A and B from shared memory, 16-bit values.
template <int CG>
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc)
{
    if constexpr (CG == 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
    else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// kind::f16 accumulating onto D scaled by 2^-12 on entry: D = A B + 2^-12 D.
template <int CG>
__device__ __forceinline__ void tc_mma_ss_scaled12(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc)
{
    if constexpr (CG == 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p, 12;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(1u), "n"(kDescHi)
        : "memory");
    else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p, 12;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(1u), "n"(kDescHi)
        : "memory");
}

// Arrive on the barrier (CG = 2: of both CTAs) once this thread's products so far are done.
template <int CG>
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if constexpr (CG == 1)
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                     "h"((uint16_t)3)
                     : "memory");
}
template <int CG>
__device__ __forceinline__ void tmem_alloc(uint32_t dst)
{
    if constexpr (CG == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
}
template <int CG>
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem)
{
    if constexpr (CG == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread t of the warp gets lane (base + t).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 lanes x 64 consecutive 32-bit columns, not waited for: tmem_wait_ld, then pin64 on the
// destination (an empty statement that redefines the registers, so that no use of them is
// scheduled before the wait).
__device__ __forceinline__ void tmem_issue64(uint32_t taddr, uint32_t *v)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]), "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39]), "=r"(v[40]), "=r"(v[41]), "=r"(v[42]), "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]), "=r"(v[48]), "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]), "=r"(v[54]), "=r"(v[55]), "=r"(v[56]), "=r"(v[57]), "=r"(v[58]), "=r"(v[59]), "=r"(v[60]), "=r"(v[61]), "=r"(v[62]), "=r"(v[63])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void pin64(uint32_t *v)
{
#pragma unroll
    for (int i = 0; i < 64; i += 8)
        asm volatile("" : "+r"(v[i]), "+r"(v[i + 1]), "+r"(v[i + 2]), "+r"(v[i + 3]), "+r"(v[i + 4]), "+r"(v[i + 5]),
                     "+r"(v[i + 6]), "+r"(v[i + 7]));
}

// 32 columns, not waited for (tmem_wait_st).
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t *v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// max of three floats in one instruction
__device__ __forceinline__ float fmax3(float x, float y, float z)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(x), "f"(y), "f"(z));
    return d;
}

// 2^x by the SFU (ex2.approx, relative error about 2^-22, subnormal results flushed to 0);
// 2^-inf = 0.
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a + b of an fp16 b, both exact operands of one fp32 addition
__device__ __forceinline__ float add_f16(float a, __half b)
{
    float r;
    asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(r) : "h"(__half_as_ushort(b)), "f"(a));
    return r;
}

// x = -infinity unless the word has the bit: a predicated move, which unlike a selection of two
// registers need not run on the integer pipe that the test is on
__device__ __forceinline__ void drop_unless(float &x, uint32_t word, uint32_t bit)
{
    asm("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
        "and.b32 t, %1, %2;\n\tsetp.eq.u32 p, t, 0;\n\t@p mov.b32 %0, 0xFF800000;\n\t}"
        : "+f"(x)
        : "r"(word), "r"(bit));
}

// Two fp32 values in one 64-bit register, and their packed fused multiply-add (each half
// rounded as the scalar operation).
__device__ __forceinline__ uint64_t f2_pack(float x, float y)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &x, float &y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Named barriers between the two warps of 32 query rows (one of each group). All of them are
// passed the same number of times by both warps whatever happens (a warp whose wait gave up only
// skips the work between them), so none can be left waiting.
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("barrier.cta.arrive.aligned %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_sync(int id) { asm volatile("barrier.cta.sync.aligned %0, 64;" ::"r"(id) : "memory"); }
// true if either warp passes flag
__device__ __forceinline__ bool pair_or(int id, bool flag)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %2, 0;\n\t"
        "barrier.cta.red.or.aligned.pred p, %1, 64, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(id), "r"((uint32_t)flag)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ int64_t row_word_offset(int64_t i)
{
    const int64_t a = i >> 5, b = i & 31;
    return i + 16 * a * (a - 1) + a * b;
}

// 16 bytes of outputs (four fp32 or eight bf16 values)
template <typename TOut>
__device__ __forceinline__ void store16(void *dst, const float *x);
template <>
__device__ __forceinline__ void store16<float>(void *dst, const float *x)
{
    *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
}
template <>
__device__ __forceinline__ void store16<__nv_bfloat16>(void *dst, const float *x)
{
    uint4 w;
    w.x = pack_bf16(x[0], x[1]);
    w.y = pack_bf16(x[2], x[3]);
    w.z = pack_bf16(x[4], x[5]);
    w.w = pack_bf16(x[6], x[7]);
    *reinterpret_cast<uint4 *>(dst) = w;
}

struct TileMaps {
    CUtensorMap qh, ql, kh, kl, v;
};

template <int DT, bool SPLIT, bool DENSE, bool SUFFIX, typename TOut>
__global__ void __launch_bounds__(kThreads, 1)
    k_attn_tile(const AttnArgs a, const __grid_constant__ TileMaps maps)
{
    static_assert(DT == 128 || DT == 64, "head dim 64 or 128");
    using L = Lay<DT>;
    constexpr int CG = L::CG, NSK = L::NSK, NSV = L::NSV, NB = L::NB;
    // no static shared memory: the dynamic block starts where the CTA's window does
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *const bars = reinterpret_cast<uint64_t *>(smem + L::OFF_BARS);
    uint32_t &tmem_base_sh = *reinterpret_cast<uint32_t *>(smem + L::OFF_TMEM);
    float *const m_sh = reinterpret_cast<float *>(smem + L::OFF_M);
    float2(*const ml_sh)[BM] = reinterpret_cast<float2(*)[BM]>(smem + L::OFF_ML);
    volatile ClosingNotes *const notes = reinterpret_cast<ClosingNotes *>(smem + L::OFF_END);
    const uint32_t sbase = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // ---- tile of this CTA (tiles covering rows row0 .. row1-1): heavier (later) tiles first. The
    // two CTAs of a cluster take two heads of a KV group at the same query tile or, where a group
    // has an odd number of heads, two consecutive query tiles of a head; either way the same key
    // tiles. A query tile outside the row range (the second of an odd last one) has no rows.
    const int qt_end = (int)((a.row1 + BM - 1) / BM), qt_first = (int)(a.row0 / BM);
    const int rank = CG == 2 ? (int)(blockIdx.x & 1) : 0;
    const bool head_pair = CG == 2 && (a.G & 1) == 0;
    const unsigned n_h = (unsigned)(head_pair ? a.Hq / 2 : a.Hq);
    const unsigned b = blockIdx.x / CG, r2 = b / n_h;
    const int h = head_pair ? 2 * (int)(b - r2 * n_h) + rank : (int)(b - r2 * n_h);
    const int s = (int)(r2 % (unsigned)a.n_sets), qp = (int)(r2 / (unsigned)a.n_sets);
    const int qt_hi = CG == 2 && !head_pair ? qt_end - 1 - 2 * qp : qt_end - 1 - qp;
    const int qt_lo = CG == 2 && !head_pair ? qt_hi - 1 : qt_hi;
    const int64_t q0 = (int64_t)(rank == 0 ? qt_hi : CG == 2 && !head_pair ? qt_lo : qt_hi) * BM;
    const int g = h / a.G;
    const int mask_id = s * a.heads_keyed + (a.heads_keyed > 1 ? g : 0);
    const int64_t last_row = min((int64_t)qt_hi * BM + BM - 1, a.row1 - 1);
    // causal: key tiles kt0 .. last_row / BN (kt0 = 0, or the tile of the first row's dense
    // suffix start, the earliest of the cluster's rows)
    const int kt0 = SUFFIX ? (int)(dense_suffix_start(a, (int64_t)max(qt_lo, qt_first) * BM) / BN) : 0;
    const int n_kt = (int)(last_row / BN) + 1 - kt0;

    constexpr auto BAR = [](int i) { return (uint32_t)(L::OFF_BARS + 8 * i); };
    const bool first_loads = a.debug_no_loads == 0 && (sbase & 1023u) == 0u;
    if (warp == kTmaWarp) {
        static_assert(L::NBAR <= 32, "a lane per barrier");
        if (lane < L::NBAR) {
            // S_GO, P_GO: the group's warps of each CTA and the relay; S_FULL, PV_DONE: the commit; the
            // copies' barriers: the loader of each CTA
            const bool go = (lane >= L::B_S_GO && lane < L::B_S_GO + NSK) || (lane >= L::B_P_GO && lane < L::B_P_GO + NSV);
            const bool done = (lane >= L::B_S_FULL && lane < L::B_S_FULL + NSK) || lane >= L::B_PV_DONE;
            mbar_init(smem_u32(&bars[lane]), go ? kGroupWarps * CG + 1 : done ? 1 : CG);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        if (lane < (int)(sizeof(ClosingNotes) / 4)) reinterpret_cast<volatile uint32_t *>(smem + L::OFF_END)[lane] = 0u;
        __syncwarp();
        // The barriers of both CTAs are initialised once this cluster barrier is passed. (That the other CTA's
        // tensor memory is allocated before a product writes to it follows from its softmax warps'
        // first arrivals.)
        if constexpr (CG == 2) cluster_sync();
        // the query tile and the first keys at once, under the rest of the start-up (about 2,000 cycles, the
        // TMEM allocation most of them). In this warp's branch: in the code of all warps the compiler spills
        // around it, N = 8192 230 instead of 226 us.
        if (lane == 0 && first_loads) {
            const uint32_t lead = CG == 2 ? cluster_addr(sbase, 0) : sbase;
            const uint32_t bq = lead + BAR(L::B_Q_FULL), bk = lead + BAR(L::B_K_FULL);
            const int key = kt0 * BN + L::KROWS * rank, row = (int)(q0 - a.q_first);
            mbar_arrive_expect_tx<CG>(bq, (SPLIT ? 2 : 1) * L::Q_ARR);
            mbar_arrive_expect_tx<CG>(bk, (SPLIT ? 2 : 1) * L::K_ARR);
            for (int blk = 0; blk < NB; ++blk) {
                tma_load_3d<CG>(sbase + L::OFF_Q + blk * L::Q_BLK, &maps.qh, 64 * blk, h, row, bq);
                if (SPLIT) tma_load_3d<CG>(sbase + L::OFF_Q + L::Q_ARR + blk * L::Q_BLK, &maps.ql, 64 * blk, h, row, bq);
                tma_load_3d<CG>(sbase + L::OFF_K + blk * L::K_BLK, &maps.kh, 64 * blk, g, key, bk);
                if (SPLIT) tma_load_3d<CG>(sbase + L::OFF_K + L::K_ARR + blk * L::K_BLK, &maps.kl, 64 * blk, g, key, bk);
            }
        }
    } else {
        if constexpr (CG == 2) cluster_arrive();
        if (warp == kScoreWarp) tmem_alloc<CG>(smem_u32(&tmem_base_sh));  // by one full warp (of each CTA)
        if constexpr (CG == 2) cluster_wait();
    }
    const uint32_t lead = CG == 2 ? cluster_addr(sbase, 0) : sbase;  // the issuing CTA's shared memory
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // all 512 columns: the allocation starts at TMEM address 0, so every address below is a
    // constant (anything else ends the CTA as a failed wait does, below)
    constexpr uint32_t T_S0 = 0, T_O = T_S0 + 2 * BN, T_P0 = T_O + DT;
    static_assert(T_P0 + BN <= kTmemCols, "TMEM columns");
    const uint32_t tmem = tmem_base_sh;
    auto arrive_lead = [&](int bar) {
        if constexpr (CG == 2)
            mbar_arrive_cluster(lead + BAR(bar));
        else
            mbar_arrive(sbase + BAR(bar));
    };
    const long long wl = a.wait_limit > 0 ? (long long)a.wait_limit : (1LL << 31);
    bool ok = tmem == 0u && (sbase & 1023u) == 0u;  // (the swizzled boxes need the alignment)

    if (warp >= kSoftmaxWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (warp == kTmaWarp) {
        // =============================== TMA producer
        if (lane == 0 && first_loads) {
            // (The query tile and the first keys were requested above.) Keys of tile j once the score
            // products of tile j - NSK are done, values of tile j once the value product of tile j - NSV is: the loader
            // waits on the barriers that announce those products (S_FULL, PV_DONE) instead of on
            // barriers of its own, which saves the tensor pipe two commits per tile. The score
            // products of tile t + 1 finish before the value product of tile t, so in this order no
            // wait holds up a load that could go before it.
            int nk = 1, nv = 0;  // tiles whose keys / values were requested
            auto load_k = [&](int j) -> bool {
                if (j >= n_kt) return true;
                const int st = j % NSK;
                if (j >= NSK && !mbar_wait<CG>(sbase + BAR(L::B_S_FULL + st), (j / NSK - 1) & 1, wl)) return false;
                const uint32_t bk = lead + BAR(L::B_K_FULL + st);
                const uint32_t dk = sbase + L::OFF_K + st * L::K_STAGE;
                const int key = (kt0 + j) * BN + L::KROWS * rank;
                mbar_arrive_expect_tx<CG>(bk, (SPLIT ? 2 : 1) * L::K_ARR);
                for (int blk = 0; blk < NB; ++blk) {
                    tma_load_3d<CG>(dk + blk * L::K_BLK, &maps.kh, 64 * blk, g, key, bk);
                    if (SPLIT) tma_load_3d<CG>(dk + L::K_ARR + blk * L::K_BLK, &maps.kl, 64 * blk, g, key, bk);
                }
                nk = j + 1;
                return true;
            };
            auto load_v = [&](int j) -> bool {
                if (j >= n_kt) return true;
                const int st = j % NSV;
                if (j >= NSV && !mbar_wait<CG>(sbase + BAR(L::B_PV_DONE + st), (j / NSV - 1) & 1, wl)) return false;
                const uint32_t bv = lead + BAR(L::B_V_FULL + st);
                const uint32_t dv = sbase + L::OFF_V + st * L::V_STAGE;
                mbar_arrive_expect_tx<CG>(bv, L::V_STAGE);
                for (int blk = 0; blk < NB / CG; ++blk)
                    tma_load_3d<CG>(dv + blk * L::V_BLK, &maps.v, 64 * (blk + rank), g, (kt0 + j) * BN, bv);
                nv = j + 1;
                return true;
            };
            ok = ok && load_v(0) && load_k(1) && load_v(1) && load_k(2) && load_k(3) && load_k(4);
            for (int t = 0; t < n_kt && ok; ++t) ok = load_k(t + 5) && load_v(t + 2);
            // (that the copies requested last have landed before a CTA leaves: see the end)
            st_cluster(sbase + L::OFF_END + offsetof(ClosingNotes, keys) + 4 * rank, 0, (uint32_t)nk);
            st_cluster(sbase + L::OFF_END + offsetof(ClosingNotes, values) + 4 * rank, 0, (uint32_t)nv);
            static_assert(NSK == 4 && NSV == 2, "the order of the loads and of the relay");
        }
    } else if (!ok || rank != 0) {
        // an unexpected base: straight to the common end; and the second CTA has nothing to issue
    } else if (warp == kRelayWarp) {
        // =============================== relay: what has landed, to the barriers that the issuing
        // warps wait on, in the order of the loads; so each of them waits on one barrier per tile
        if (lane == 0) {
            auto relay_k = [&](int j) -> bool {
                if (j >= n_kt) return true;
                if (!mbar_wait<CG>(sbase + BAR(L::B_K_FULL + j % NSK), (j / NSK) & 1, wl)) return false;
                mbar_arrive(sbase + BAR(L::B_S_GO + j % NSK));
                return true;
            };
            auto relay_v = [&](int j) -> bool {
                if (j >= n_kt) return true;
                if (!mbar_wait<CG>(sbase + BAR(L::B_V_FULL + j % NSV), (j / NSV) & 1, wl)) return false;
                mbar_arrive(sbase + BAR(L::B_P_GO + j % NSV));
                return true;
            };
            ok = mbar_wait<CG>(sbase + BAR(L::B_Q_FULL), 0, wl) && relay_k(0) && relay_v(0) && relay_k(1) && relay_v(1) &&
                 relay_k(2) && relay_k(3) && relay_k(4);
            for (int t = 0; t < n_kt && ok; ++t) ok = relay_k(t + 5) && relay_v(t + 2);
        }
    } else {
        // =============================== product issuers (of the cluster's first CTA, for both): one
        // warp for the scores, one for the value products, so that neither's waits (about 100
        // cycles each even on a completed phase) leave the tensor pipe without queued work.
        // The whole warp runs this code, so that every operand is warp-uniform, and one elected
        // lane issues: inside a branch on the lane the compiler moves each of a product's operands
        // (two descriptors, two TMEM addresses, the instruction descriptor) into uniform registers
        // one by one, about 60 cycles per product, as long as a 128 x 128 x 16 product itself.
        constexpr uint32_t ID_S = idesc_bf16(CG * BM, BN, false);  // S[128 x 128] = Q K^T, both K-major
        constexpr uint32_t ID_SH = idesc_f16(CG * BM, BN, false);  // fp16 x fp16 (and e4m3 x e4m3 for kind::f8f6f4)
        constexpr uint32_t ID_O = idesc_f16(CG * BM, DT, true);  // O[128 x DT] += P V, fp16, V MN-major
        // fp8-correction scores (rotated q / k at head dim 128, operands written by
        // launch_fp8_prep when the bounds allow): the same bytes in the same places as the
        // bf16 pair, read as fp16 hi parts and, in the place of the low parts (Q_ARR, K_ARR on),
        // e4m3 corrections, one 64-column block of hi parts and one of lo parts
        int ea = 0, eb = 0;
        const bool use8 = DT == 128 && SPLIT && a.qk_bound != nullptr &&
                          __any_sync(0xFFFFFFFFu, fp8_score_scales(a.qk_bound[0], a.qk_bound[1], ea, eb));
        // score products of a tile of ring stage ST: A = the query tile, B = the keys, both K-major in
        // shared memory, a k-step of 16 (e4m3: 32) columns 32 B further in a 128 B row
        auto issue_s = [&](auto st_c) {
            constexpr int ST = decltype(st_c)::value;
            const uint32_t kd = desc_lo(sbase + L::OFF_K + ST * L::K_STAGE, 16);  // K hi; K lo K_ARR on
            const uint32_t qd = desc_lo(sbase + L::OFF_Q, 16);                     // Q hi; Q lo Q_ARR on
            constexpr uint32_t dt = T_S0 + (ST & 1) * BN;
            if (elect_one()) {
                if (use8) {
                    // 2^12 (q_h8 k_l8 + q_l8 k_h8): two e4m3 products of 4 k-steps of 32
#pragma unroll
                    for (int ks = 0; ks < DT / 32; ++ks)
                        tc_mma_ss_f8<CG>(dt, qd + dstep(L::Q_ARR + ks * 32), kd + dstep(L::K_ARR + L::K_BLK + ks * 32), ID_SH, ks > 0);
#pragma unroll
                    for (int ks = 0; ks < DT / 32; ++ks)
                        tc_mma_ss_f8<CG>(dt, qd + dstep(L::Q_ARR + L::Q_BLK + ks * 32), kd + dstep(L::K_ARR + ks * 32), ID_SH, 1u);
                    // + q_h k_h in fp16, the corrections brought back by 2^-12 on the first k-step
#pragma unroll
                    for (int ks = 0; ks < DT / 16; ++ks) {
                        const uint32_t ad = qd + dstep((ks >> 2) * L::Q_BLK + (ks & 3) * 32);
                        const uint32_t bd = kd + dstep((ks >> 2) * L::K_BLK + (ks & 3) * 32);
                        if (ks == 0)
                            tc_mma_ss_scaled12<CG>(dt, ad, bd, ID_SH);
                        else
                            tc_mma_ss<CG>(dt, ad, bd, ID_SH, 1u);
                    }
                } else {
                    // (A, B) pairs: (Q hi, K hi), (Q lo, K hi), (Q hi, K lo)
#pragma unroll
                    for (int prod = 0; prod < (SPLIT ? 3 : 1); ++prod)
#pragma unroll
                        for (int ks = 0; ks < DT / 16; ++ks)
                            tc_mma_ss<CG>(dt, qd + dstep((prod == 1 ? L::Q_ARR : 0) + (ks >> 2) * L::Q_BLK + (ks & 3) * 32),
                                          kd + dstep((prod == 2 ? L::K_ARR : 0) + (ks >> 2) * L::K_BLK + (ks & 3) * 32), ID_S,
                                          prod > 0 || ks > 0);
                }
                tc_commit<CG>(sbase + BAR(L::B_S_FULL + ST));
            }
            __syncwarp();
        };
        // value product of a tile of ring stage ST: P (in TMEM, the buffer of the tile's parity), 128
        // keys of fp16 values packed two per column, times V, 128 keys x 128 B rows per block: 16 keys = two
        // 8-row atoms (SBO 1024); the second 64-column block of head dim is LBO = 16 KB away
        auto issue_o = [&](auto st_c, uint32_t acc) {
            constexpr int ST = decltype(st_c)::value;
            const uint32_t vd = desc_lo(sbase + L::OFF_V + ST * L::V_STAGE, L::V_BLK);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < BN / 16; ++ks)
                    tc_mma_ts<CG>(T_O, T_P0 + ST * (BN / 2) + 8 * ks, vd + dstep(ks * 2048), ID_O, ks > 0 ? 1u : acc);
                tc_commit<CG>(sbase + BAR(L::B_PV_DONE + ST));
            }
            __syncwarp();
        };
        auto wait_all = [&](int bar, int parity) -> bool {
            const bool got = __all_sync(0xFFFFFFFFu, mbar_wait<CG>(sbase + BAR(bar), parity, wl));
            tc_fence_after();
            return got;
        };
        int issued = 0;  // tiles whose products this warp committed
        // the scores of tile j, as soon as those of tile j - 2 have been read out: they are there
        // when the group of tile j comes for them
        auto score_step = [&](auto st_c, int j) {
            if (!ok || j >= n_kt) return;
            ok = wait_all(L::B_S_GO + decltype(st_c)::value, (j / NSK) & 1);
            if (!ok) return;
            issue_s(st_c);
            issued = j + 1;
        };
        auto value_step = [&](auto st_c, int j) {
            if (!ok || j >= n_kt) return;
            ok = wait_all(L::B_P_GO + decltype(st_c)::value, (j / NSV) & 1);
            if (!ok) return;
            issue_o(st_c, j > 0 ? 1u : 0u);
            issued = j + 1;
        };
        using I0 = std::integral_constant<int, 0>;
        using I1 = std::integral_constant<int, 1>;
        using I2 = std::integral_constant<int, 2>;
        using I3 = std::integral_constant<int, 3>;
        if (warp == kScoreWarp) {
            for (int j = 0; j < n_kt && ok; j += 4) {
                score_step(I0{}, j);
                score_step(I1{}, j + 1);
                score_step(I2{}, j + 2);
                score_step(I3{}, j + 3);
            }
        } else {
            for (int j = 0; j < n_kt && ok; j += 2) {
                value_step(I0{}, j);
                value_step(I1{}, j + 1);
            }
        }
        if (lane < CG) {
            const int off = L::OFF_END + (warp == kValueWarp ? offsetof(ClosingNotes, valued) : offsetof(ClosingNotes, scored));
            st_cluster(sbase + off, lane, (uint32_t)issued);
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
        // =============================== softmax: group grp of four warps takes the tiles of parity
        // grp, one thread per query row q0 + r; at the start and the end a thread owns half of its
        // row's head dim, columns OC grp .. OC grp + OC - 1
        constexpr int OC = DT / 2;
        const int wq = warp & 3, grp = warp >> 2;
        const int r = wq * 32 + lane;  // TMEM lane
        const int64_t i = q0 + r;
        const bool row_ok = i >= a.row0 && i < a.row1;
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        const float sc = a.scale_log2;
        const float v_absmax = *a.v_absmax;
        // the group's score buffer is free for its first tile
        if (lane == 0 && grp < n_kt) arrive_lead(L::B_S_GO + grp);
        // kept keys of word e of tile j (keys 128 (kt0 + j) + 32 e .. +31): the bitmap's word, or
        // the range suffix_lo .. i (dense: 0 .. i)
        constexpr bool kRange = DENSE || SUFFIX;
        constexpr int NW = BN / 32;
        const uint32_t *bm = kRange ? nullptr
                                    : a.bitmap + (int64_t)mask_id * a.words_per_mask + (row_ok ? row_word_offset(i) : 0);
        const int n_words = row_ok ? (int)(i >> 5) + 1 : 0;
        const int row_in = row_ok ? (int)(i - (int64_t)kt0 * BN) : -1;  // the row's own key, from the first tile's start
        const int suffix_in = SUFFIX ? (int)(dense_suffix_start(a, i) - (int64_t)kt0 * BN) : 0;
        auto mask_words = [&](int j, uint32_t(&w)[NW]) {
#pragma unroll
            for (int e = 0; e < NW; ++e) {
                if (kRange) {
                    const int k0 = j * BN + 32 * e;
                    const int lim = min(31, max(-1, row_in - k0));  // last kept key of the word
                    w[e] = lim < 0 ? 0u : 0xFFFFFFFFu >> (31 - lim);
                    if (SUFFIX) {
                        const int lo = suffix_in - k0;
                        if (lo > 31)
                            w[e] = 0u;
                        else if (lo > 0)
                            w[e] &= 0xFFFFFFFFu << lo;
                    }
                } else {
                    const int wd = (kt0 + j) * NW + e;
                    w[e] = wd < n_words ? bm[wd] : 0u;
                }
            }
        };
        // bitmap words fetched two of the group's tiles (four tiles) ahead of their use, past a
        // DRAM miss
        uint32_t cw[NW], nw[NW], nnw[NW];
        if (!kRange) {
            mask_words(grp, cw);
            mask_words(grp + 2, nw);
        }
        const uint64_t sc2 = f2_pack(sc, sc);
        float l = 0.f, m_own = -INFINITY;  // row sum over this thread's tiles, relative to 2^m_own
        bool s_full = false;  // seen at the end of the last tile: a poll takes 200 cycles even if it succeeds
        for (int j = grp; j < n_kt; j += 2) {
            if (!kRange) mask_words(j + 4, nnw);
            if (ok) {
                const uint32_t bar = sbase + BAR(L::B_S_FULL + j % NSK);
                ok = __all_sync(0xFFFFFFFFu, s_full || mbar_wait<CG, true>(bar, (j / NSK) & 1, wl));
            }
            tc_fence_after();
            uint32_t su[2][64];
            tmem_issue64(T_S0 + grp * BN + lane_off, su[0]);
            tmem_issue64(T_S0 + grp * BN + lane_off + 64, su[1]);
            bool whole = false;  // every pair of this warp's rows and this tile is kept
            if (kRange) {
                mask_words(j, cw);
                whole = __all_sync(0xFFFFFFFFu, (cw[0] & cw[1] & cw[2] & cw[3]) == 0xFFFFFFFFu);
            }
            tmem_wait_ld();
            pin64(su[0]);
            pin64(su[1]);
            tc_fence_before();
            __syncwarp();
            tc_fence_before();
            if (lane == 0 && j + 2 < n_kt) arrive_lead(L::B_S_GO + (j + 2) % NSK);
            float sv[BN];
#pragma unroll
            for (int c = 0; c < BN; ++c) sv[c] = __uint_as_float(su[c >> 6][c & 63]);
            if (!whole) {
#pragma unroll
                for (int c = 0; c < BN; ++c) drop_unless(sv[c], cw[c >> 5], 1u << (c & 31));
            }
            if (!kRange) {
#pragma unroll
                for (int e = 0; e < NW; ++e) {
                    cw[e] = nw[e];
                    nw[e] = nnw[e];
                }
            }
            // row max as a tree (the scale is positive: it is applied to the max and folded into
            // the exponent of P)
            float mx8[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                mx8[e] = fmaxf(sv[e], sv[e + 8]);
#pragma unroll
                for (int c = 16; c < BN; c += 16) mx8[e] = fmax3(mx8[e], sv[c + e], sv[c + 8 + e]);
            }
            const float mx =
                fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) * sc;
            // The row's reference maximum moves on from tile to tile, handed to the other group. Lazy
            // rescale: it moves, and O is rescaled, only when the row max grows by more than
            // kLazyLog2. The TMEM loads / stores are warp-collective
            // (.sync.aligned), so the whole warp runs them when any of its rows needs it; the
            // other rows multiply by 1.
            float m_prev = -INFINITY;
            if (j > 0) {
                pair_sync(1 + 2 * wq + (grp ^ 1));
                m_prev = m_sh[r];
            }
            const bool upd = mx > m_prev + kLazyLog2;
            const float m_ref = upd ? mx : m_prev;
            // the value product of tile t is done (t < 0: nothing to wait for)
            auto pv_done = [&](int t) -> bool {
                const uint32_t bar = sbase + BAR(L::B_PV_DONE + t % NSV);
                return t < 0 || __all_sync(0xFFFFFFFFu, mbar_wait<CG, true>(bar, (t / NSV) & 1, wl));
            };
            const bool scale_o = upd && m_prev != -INFINITY;
            const bool any_scale = __any_sync(0xFFFFFFFFu, scale_o);
            const float al = scale_o ? exp2f(m_prev - m_ref) : 1.f;
            if (m_ref != m_own) {
                l *= m_own == -INFINITY ? 0.f : exp2f(m_own - m_ref);
                m_own = m_ref;
            }
            const float mu = (m_ref == -INFINITY) ? 0.f : m_ref;
            // P = exp2(s - m_ref) as the A operand of the value product, packed two keys per
            // column. The row sum adds P as rounded, so that the rounding of each weight moves the
            // output by at most 2^-11 of the weight times |v_j - o| (a normalised average of the
            // values with slightly perturbed weights). The additions take the fp16 halves as they are:
            // this loop alone, two warps of a scheduler, 690 cycles a tile with conversions and packed
            // additions, 600 so, 540 for the exponentials and their arguments only.
            float lsum[4] = {};
            const uint64_t nmu2 = f2_pack(-mu, -mu);
            uint32_t hw[BN / 2];
#pragma unroll
            for (int w = 0; w < BN / 2; ++w) {
                float x0, x1;
                f2_unpack(f2_fma(f2_pack(sv[2 * w], sv[2 * w + 1]), sc2, nmu2), x0, x1);
                const __half2 hp = __floats2half2_rn(ex2(x0), ex2(x1));
                lsum[2 * (w & 1)] = add_f16(lsum[2 * (w & 1)], __low2half(hp));
                lsum[2 * (w & 1) + 1] = add_f16(lsum[2 * (w & 1) + 1], __high2half(hp));
                hw[w] = *reinterpret_cast<const uint32_t *>(&hp);
            }
            // Only now on to the other group: its exponentials (the other warp of this scheduler) run
            // while this warp stores P and takes the next tile's scores and maximum, and not
            // against this warp's own
            if (j + 1 < n_kt) {
                m_sh[r] = m_ref;
                __threadfence_block();
                pair_arrive(1 + 2 * wq + grp);
            }
            if (!ok) continue;
            ok = pv_done(j - 2);  // P's buffer is free
            if (!ok) continue;
            tc_fence_after();
            if (any_scale) {
                // O has settled once the value product of tile j - 1 is done (that of tile j - 2 first,
                // above, so that the barrier is not polled a phase early); nothing adds to it before
                // this warp's P is announced below, and the other group's warp of these rows scales it next
                // only after that product. Here and not ahead of the exponentials, where the wait held
                // up the other group as well.
                ok = pv_done(j - 1);
                if (!ok) continue;
                tc_fence_after();
#pragma unroll 1
                for (int c0 = 0; c0 < DT; c0 += 32) {
                    float ov[32];
                    uint32_t ow[32];
                    tmem_ld32(T_O + lane_off + c0, ov);
#pragma unroll
                    for (int c = 0; c < 32; ++c) ow[c] = __float_as_uint(ov[c] * al);
                    tmem_st32(T_O + lane_off + c0, ow);
                }
                tmem_wait_st();
            }
            const uint32_t tp = T_P0 + grp * (BN / 2) + lane_off;
            tmem_st32(tp, hw);
            tmem_st32(tp + 32, hw + 32);
            s_full = j + 2 < n_kt && mbar_test<CG, true>(sbase + BAR(L::B_S_FULL + (j + 2) % NSK), ((j + 2) / NSK) & 1);
            l += (lsum[0] + lsum[2]) + (lsum[1] + lsum[3]);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            tc_fence_before();
            if (lane == 0) arrive_lead(L::B_P_GO + grp);
        }
        // the row's maximum and sum from both threads
        ml_sh[grp][r] = make_float2(m_own, l);
        ok = !pair_or(9 + wq, !ok);
        for (int t = max(0, n_kt - 2); t < n_kt && ok; ++t)  // in order, as above
            ok = __all_sync(0xFFFFFFFFu, mbar_wait<CG>(sbase + BAR(L::B_PV_DONE + t % NSV), (t / NSV) & 1, wl));
        if (ok) {
            tc_fence_after();
            const float2 ma = ml_sh[0][r], mb = ml_sh[1][r];
            // the group of the last tile holds the final maximum; a group without tiles has l = 0
            const float m_fin = ((n_kt - 1) & 1) ? mb.x : ma.x;
            const float lt = (ma.x == m_fin ? ma.y : ma.y * exp2f(ma.x - m_fin)) +
                             (mb.x == m_fin ? mb.y : mb.y * exp2f(mb.x - m_fin));
            // fp16 values were scaled by 2^-E for the value product
            const float vs = __uint_as_float((uint32_t)(127 + v_scale_exp(v_absmax)) << 23);
            const float inv = lt > 0.f ? vs / lt : 0.f;
            // O, normalised, through shared memory (the ring is free: every load was consumed) so that
            // neighbouring lanes store neighbouring pieces of a row: stores of 16 bytes per lane and
            // row took 4,000 cycles of a CTA. A warp's part: its 32 rows x OC columns, 16-byte
            // pieces swizzled by the row.
            constexpr int RB = OC * (int)sizeof(TOut), NP = RB / 16;  // bytes and pieces of a row's part
            unsigned char *stage = smem + warp * (32 * RB);
#pragma unroll
            for (int c0 = 0; c0 < OC; c0 += 32) {
                float ov[32];
                tmem_ld32(T_O + lane_off + OC * grp + c0, ov);
#pragma unroll
                for (int c = 0; c < 32; ++c) ov[c] *= inv;
#pragma unroll
                for (int e = 0; e < 32 * (int)sizeof(TOut) / 16; ++e) {
                    const int piece = c0 * (int)sizeof(TOut) / 16 + e;
                    store16<TOut>(stage + lane * RB + ((piece ^ (lane & (NP - 1))) << 4), ov + e * (16 / (int)sizeof(TOut)));
                }
            }
            __syncwarp();
            const int64_t w0 = q0 + 32 * wq;  // the warp's first row
            TOut *out = (SUFFIX ? reinterpret_cast<TOut *>(a.part_o) : reinterpret_cast<TOut *>(a.out) + (int64_t)s * a.N * a.Hq * DT) +
                        (int64_t)h * DT + OC * grp;
#pragma unroll
            for (int e = 0; e < NP; ++e) {
                const int rr = e * (32 / NP) + lane / NP, piece = lane & (NP - 1);
                const uint4 x = *reinterpret_cast<const uint4 *>(stage + rr * RB + ((piece ^ (rr & (NP - 1))) << 4));
                if (w0 + rr >= a.row0 && w0 + rr < a.row1)
                    *reinterpret_cast<uint4 *>(out + (w0 + rr) * a.Hq * DT + piece * (16 / (int)sizeof(TOut))) = x;
            }
            if (SUFFIX) {
                if (row_ok && grp == 0) a.part_lse[i * a.Hq + h] = m_fin + __log2f(lt);
            } else if (row_ok && grp == 0 && a.lse != nullptr) {
                a.lse[((int64_t)s * a.Hq + h) * a.lse_ld + i] = (m_fin + __log2f(lt)) * kLn2;
            }
        }
    }

    if (!ok) {
        atomicOr(&g_ris_tile_error, 2u);
        for (int c = 0; c < CG; ++c) st_cluster(sbase + L::OFF_END + offsetof(ClosingNotes, bad), c, 1u);
    }
    __syncwarp();
    tc_fence_before();
    // Neither CTA of a cluster may leave, or release TMEM, while a product is running or anything can
    // still reach its shared memory. The softmax warps of each CTA have seen, in their own
    // barriers, every commit (S_FULL of every tile, PV_DONE of every tile), and so the end of every copy:
    // nothing is under way unless a wait gave up. Then the copies and commits still to come, as the
    // loaders and the issuing warps counted them, are waited for before both CTAs leave. (What one
    // loader requested and the other did not is announced here in its place. A tile is requested only
    // after the products on its stage's last tile, so no count is behind by more than the ring, and no
    // barrier by more than one phase.)
    if constexpr (CG == 2) cluster_sync();
    __syncthreads();
    tc_fence_after();
    if (notes->bad != 0u) {
        if (warp == kTmaWarp && lane == 0) {
            auto landed = [&](int bar, int stages, int n0, int n1) {
                const int n = max(n0, n1);
                for (int j = max(0, n - stages); j < n; ++j) {
                    if (j >= min(n0, n1)) mbar_arrive(sbase + BAR(bar + j % stages));
                    mbar_wait_own<CG>(sbase + BAR(bar + j % stages), (j / stages) & 1);
                }
            };
            if (rank == 0) {
                constexpr int R1 = CG - 1;
                if (notes->keys[0] > 0u) mbar_wait_own<CG>(sbase + BAR(L::B_Q_FULL), 0);
                landed(L::B_K_FULL, NSK, (int)notes->keys[0], (int)notes->keys[R1]);
                landed(L::B_V_FULL, NSV, (int)notes->values[0], (int)notes->values[R1]);
            }
            const int ns = (int)notes->scored, nv = (int)notes->valued;
            for (int j = max(0, ns - NSK); j < ns; ++j) mbar_wait_own<CG>(sbase + BAR(L::B_S_FULL + j % NSK), (j / NSK) & 1);
            for (int j = max(0, nv - NSV); j < nv; ++j) mbar_wait_own<CG>(sbase + BAR(L::B_PV_DONE + j % NSV), (j / NSV) & 1);
        }
        __syncwarp();
        if constexpr (CG == 2) cluster_sync();
        __syncthreads();
        tc_fence_after();
    }
    if (warp == kScoreWarp) tmem_dealloc<CG>(tmem);
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// [N][H][DT] 16-bit values (bf16, or fp16 with f16 set) viewed as 3D (d, head, token); box =
// 64 d x 1 head x `rows` tokens.
bool make_map3(CUtensorMap *m, const void *base, int64_t N, int H, int rows, int DT, bool f16 = false)
{
    auto fn = encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[3] = {(cuuint64_t)DT, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[2] = {(cuuint64_t)DT * 2, (cuuint64_t)H * DT * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)rows};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base),
              dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DT, bool SPLIT, bool DENSE, typename TOut, bool SUFFIX = false>
cudaError_t launch_t(const AttnArgs &a, const TileMaps &maps, cudaStream_t s)
{
    auto kern = k_attn_tile<DT, SPLIT, DENSE, SUFFIX, TOut>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        if (e != cudaSuccess) return e;
        // the softmax threads' setmaxnreg would wait for registers that a smaller launch lacks
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, kern);
        if (e != cudaSuccess) return e;
        if (fa.numRegs < kRegs) return cudaErrorInvalidConfiguration;
        attr = true;
    }
    constexpr int CG = Lay<DT>::CG;
    const int64_t n_qt = (a.row1 + BM - 1) / BM - a.row0 / BM;  // tiles covering rows row0 .. row1-1
    const bool tile_pair = CG == 2 && (a.G & 1) != 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((tile_pair ? (n_qt + 1) / 2 * 2 : n_qt) * a.Hq * a.n_sets));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CG;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a, maps);
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

}  // namespace

bool tile_design_available() { return encode_fn() != nullptr; }


// Read and clear this kernel's device error word (the caller has synchronised).
cudaError_t read_tile_error(unsigned int *out)
{
    cudaError_t e = cudaMemcpyFromSymbol(out, g_ris_tile_error, sizeof(unsigned int));
    if (e != cudaSuccess || *out == 0u) return e;
    const unsigned int zero = 0u;
    return cudaMemcpyToSymbol(g_ris_tile_error, &zero, sizeof(unsigned int));
}

// Q / K / V tensor maps of a call (the low parts only with split queries and keys; the values
// as fp16). q_hi, q_lo: moved back by a.q_first rows, as the kernels' other row pointers.
bool make_maps(TileMaps &maps, const AttnArgs &a, const void *q_hi, const void *q_lo, int D)
{
    const bool split = q_lo != nullptr;
    if (a.v16 == nullptr || a.v_absmax == nullptr) return false;
    const int krows = D == 128 ? Lay<128>::KROWS : Lay<64>::KROWS;  // keys of a box
    if (!make_map3(&maps.kh, a.k, a.N, a.Hkv, krows, D) || !make_map3(&maps.v, a.v16, a.N, a.Hkv, BN, D, true)) return false;
    const size_t back = (size_t)a.q_first * a.Hq * D * 2;
    auto q_map = [&](CUtensorMap *m, const void *q) {
        return make_map3(m, static_cast<const char *>(q) + back, a.q_rows, a.Hq, BM, D);
    };
    if (!q_map(&maps.qh, q_hi)) return false;
    if (split) return q_map(&maps.ql, q_lo) && make_map3(&maps.kl, a.k_lo, a.N, a.Hkv, krows, D);
    maps.kl = maps.kh;
    maps.ql = maps.qh;
    return true;
}

template <int DT>
cudaError_t launch_tile_d(const AttnArgs &a, const TileMaps &maps, bool split, int out_dtype, bool dense, cudaStream_t s)
{
    if (out_dtype == RIS_F32) {
        if (split) return dense ? launch_t<DT, true, true, float>(a, maps, s) : launch_t<DT, true, false, float>(a, maps, s);
        return dense ? launch_t<DT, false, true, float>(a, maps, s) : launch_t<DT, false, false, float>(a, maps, s);
    }
    if (split)
        return dense ? launch_t<DT, true, true, __nv_bfloat16>(a, maps, s)
                     : launch_t<DT, true, false, __nv_bfloat16>(a, maps, s);
    return dense ? launch_t<DT, false, true, __nv_bfloat16>(a, maps, s)
                 : launch_t<DT, false, false, __nv_bfloat16>(a, maps, s);
}

// q_hi / q_lo: queries as a bf16 pair [N][Hq][D] (q_lo null: exact bf16 queries and keys,
// one score product); a.k / a.k_lo: keys as a pair; a.v: values. Head dim 128 or 64.
cudaError_t launch_attention_tile(const AttnArgs &a, int D, const void *q_hi, const void *q_lo, int out_dtype,
                                  bool dense, cudaStream_t s)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    if (D != 128 && D != 64) return cudaErrorInvalidValue;
    alignas(64) TileMaps maps;
    if (!make_maps(maps, a, q_hi, q_lo, D)) return cudaErrorInvalidValue;
    return D == 128 ? launch_tile_d<128>(a, maps, q_lo != nullptr, out_dtype, dense, s)
                    : launch_tile_d<64>(a, maps, q_lo != nullptr, out_dtype, dense, s);
}

cudaError_t launch_attention_tile_suffix(const AttnArgs &a, int D, const void *q_hi, const void *q_lo, cudaStream_t s)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    if (a.part_o == nullptr || a.part_lse == nullptr || a.n_sets != 1 || (D != 128 && D != 64))
        return cudaErrorInvalidValue;
    const bool split = q_lo != nullptr;
    alignas(64) TileMaps maps;
    if (!make_maps(maps, a, q_hi, q_lo, D)) return cudaErrorInvalidValue;
    if (D == 128)
        return split ? launch_t<128, true, false, float, true>(a, maps, s)
                     : launch_t<128, false, false, float, true>(a, maps, s);
    return split ? launch_t<64, true, false, float, true>(a, maps, s)
                 : launch_t<64, false, false, float, true>(a, maps, s);
}

}  // namespace ris
