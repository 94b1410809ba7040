// RIS sparse attention, masked dense-tile design on the 5th-generation tensor cores
// (paper, Methods, "Hybrid Anchor and Pre-Fusion Unified Softmax (PFUS)"; the dense causal
// upper bound of Table tab:results_32k is the same kernel with every causal pair kept).
//
// Where the master mask keeps a large share of the causal pairs (union densities of tens of
// percent, and the dense mode) a dense 128 x 128 score tile with the mask applied as -inf
// beats gathering rows pair by pair. One CTA owns one (128-query tile, query head, set):
//
//   warp 8 (TMA)   streams 128-key tiles of the keys (64 KB: hi parts and corrections) and of
//                  the values (fp16, 32 KB) in 128-byte swizzled boxes into two two-stage
//                  shared-memory rings: a key stage is refilled as soon as its score products
//                  are done, a value stage once its value product is; it also waits for each
//                  tile's values to land and then arrives on that tile's P_FULL barrier, so
//                  that the MMA warp waits once per value product;
//   warp 9 (MMA)   issues tcgen05.mma: the score tile S (A = the query tile: its hi part in TMEM,
//                  its low part in shared memory) into a double-buffered TMEM score tile, and
//                  O += P V (A = P as fp16 in TMEM) into the TMEM output tile, committing each
//                  step to an mbarrier; TMEM holds S twice (2 x 128 columns), O (128), the
//                  query's hi part (64) and P (64), all 512 columns. P has columns of its own, so
//                  the scores of tile j + 2 start as soon as those of tile j have been read;
//   warps 0-7      two groups of four warps, one thread per query row in each, taking alternate
//                  tiles: write the query tile, then per tile tcgen05.ld the row's 128 scores,
//                  apply the bitmap (words fetched four tiles ahead) or the causal cut, take the
//                  row max, pass the row's reference maximum on to the other group, fp32 online
//                  softmax with lazy rescaling of O in TMEM (only when the row max grows by more
//                  than 2^8), write P into TMEM, and at the end normalise O (and undo the values'
//                  power-of-two scale) and store the row.
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
// e4m3 corrections at twice the rate, 8 fp16 value products), 1,536 cycles of the tensor pipe.
// Measured per tile with clock64() stamps in the longest CTA of a 32k dense / 64k 10% layer:
//   2,485 / 2,650 cycles  P over the score columns, one lane issuing inside a branch, two threads
//                         per row in lockstep: each product cost the issuing lane about 60 cycles of
//                         operand moves, as long as the product, plus its waits;
//   2,055 / 2,400         operands warp-uniform and issued by an elected lane: the softmax, its two
//                         threads per row meeting in every tile, set the pace;
//   1,860 / 2,040         the two groups on alternate tiles, half a period apart (this form): the
//                         rest is the L2 latency of the keys, requested only when the ring's
//                         two stages allow, and the issuer's waits.
// Layer calls, before -> now: N = 8192 305 -> 279 us, 32k dense 3.73 -> 3.32 ms, 64k 14.0 -> 12.6 ms.
// A separate issuing warp for the value products ran no faster (its products interleave with the
// next scores, whose keys then arrive later still).
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
constexpr int kSoftmaxThreads = 32 * kSoftmaxWarps;
constexpr int kTmaWarp = kSoftmaxWarps, kMmaWarp = kSoftmaxWarps + 1;
constexpr int kThreads = 32 * (kSoftmaxWarps + 4);
// registers per thread: at launch, then after setmaxnreg of a softmax and of a loader / MMA thread
constexpr int kRegs = 168, kSoftmaxRegs = 200, kOtherRegs = 104;
static_assert(2 * kSoftmaxRegs + kOtherRegs == 3 * kRegs, "the shares of the three warpgroups add up to the launch's");
constexpr uint32_t kTmemCols = 512;  // S[2] (2 x 128) + O (128) + Q hi (64) + P (64)

// shared-memory map (bytes, from a 1024-aligned base) for head dim DT (128 or 64): the K ring,
// the V ring, the low part of the query tile, then the barriers, the TMEM base and what the two
// threads of a row hand to each other: the row's reference maximum after each tile, and at the
// end each thread's row sum and the maximum it refers to
constexpr int KV_BLK = BN * 128;            // 16 KB: one 64-column block
constexpr int kStages = 2;                  // stages of each ring
template <int DT>
struct Smem {
    static constexpr int KV_ARR = BN * DT * 2;  // 32 KB at DT = 128: one of K hi / K lo / V / Q lo
    static constexpr int K_STAGE = 2 * KV_ARR;  // K hi, K lo
    static constexpr int V_STAGE = KV_ARR;
    static constexpr int OFF_K = 0;
    static constexpr int OFF_V = kStages * K_STAGE;
    static constexpr int OFF_Q = OFF_V + kStages * V_STAGE;
    static constexpr int OFF_BARS = OFF_Q + KV_ARR;
    static constexpr int OFF_TMEM = OFF_BARS + 120;  // after the NBAR barriers
    static constexpr int OFF_M = OFF_BARS + 128;     // float [BM]
    static constexpr int OFF_ML = OFF_M + BM * 4;    // float2 [2][BM]
    static constexpr int BYTES = OFF_ML + 2 * BM * 8;
    static_assert(BYTES <= 232448, "shared memory of a CTA");
};
// the head-dim-128 layout (232,064 of the 232,448 bytes a CTA can have) is requested at either
// head dim: it keeps one CTA per SM, as the CTA holds all 512 TMEM columns
constexpr int SMEM_BYTES = Smem<128>::BYTES;

// S_FULL, S_READ, P_FULL and PV_DONE have one barrier per tile parity, so that no waiter can
// fall two phases behind a barrier it polls by parity.
enum Bar {
    B_Q = 0, B_K_FULL = 1, B_V_FULL = 3, B_S_FULL = 5, B_S_READ = 7, B_P_FULL = 9, B_PV_DONE = 11, B_END = 13,
    NBAR = 14
};
static_assert(NBAR * 8 <= 120, "barriers below the TMEM base word");

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait for this CTA's own asynchronous work (copies or products already issued):
// about 2^31 cycles at most, whatever other CTAs reported.
__device__ __forceinline__ bool mbar_wait_own(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > (1LL << 31)) return false;
    return true;
}

// Bounded wait (`limit` cycles, about 2^31 unless a test lowers it); false if the phase did
// not complete in time or another CTA already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) return false;
        if (*reinterpret_cast<volatile unsigned int *>(&g_ris_tile_error) != 0u) return false;
    }
    return true;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar)
{
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
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// kind::f8f6f4 (e4m3 x e4m3 with the instruction descriptor's format fields 0), A and B from
// shared memory.
__device__ __forceinline__ void tc_mma_ss_f8(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// A and B from shared memory, 16-bit values.
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %5};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a), "r"(b), "r"(idesc), "r"(acc), "n"(kDescHi)
        : "memory");
}

// kind::f16 accumulating onto D scaled by 2^-12 on entry: D = A B + 2^-12 D.
__device__ __forceinline__ void tc_mma_ts_scaled12(uint32_t d_tmem, uint32_t a_tmem, uint32_t b, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p, 12;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b), "r"(idesc), "r"(1u), "n"(kDescHi)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
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

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t *v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
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

// 32 lanes x 16 consecutive 32-bit columns, loaded and waited for in one statement.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

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

// Two fp32 values in one 64-bit register, and their packed fused multiply-add and sum (each
// half rounded as the scalar operation).
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
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
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

template <typename TOut>
__device__ __forceinline__ void store8(TOut *dst, const float *x);
template <>
__device__ __forceinline__ void store8<float>(float *dst, const float *x)
{
    reinterpret_cast<float4 *>(dst)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4 *>(dst)[1] = make_float4(x[4], x[5], x[6], x[7]);
}
template <>
__device__ __forceinline__ void store8<__nv_bfloat16>(__nv_bfloat16 *dst, const float *x)
{
    uint4 w;
    w.x = pack_bf16(x[0], x[1]);
    w.y = pack_bf16(x[2], x[3]);
    w.z = pack_bf16(x[4], x[5]);
    w.w = pack_bf16(x[6], x[7]);
    *reinterpret_cast<uint4 *>(dst) = w;
}

struct TileMaps {
    CUtensorMap kh, kl, v;
};

template <int DT, bool SPLIT, bool DENSE, bool SUFFIX, typename TOut>
__global__ void __launch_bounds__(kThreads, 1)
    k_attn_tile(const AttnArgs a, const __grid_constant__ TileMaps maps, const void *q_hi, const void *q_lo)
{
    static_assert(DT == 128 || DT == 64, "head dim 64 or 128");
    constexpr int KV_ARR = Smem<DT>::KV_ARR, K_STAGE = Smem<DT>::K_STAGE, V_STAGE = Smem<DT>::V_STAGE;
    constexpr int OFF_K = Smem<DT>::OFF_K, OFF_V = Smem<DT>::OFF_V, OFF_Q = Smem<DT>::OFF_Q;
    constexpr int NB = DT / 64;  // 64-column blocks of a row
    // no static shared memory: the dynamic block starts where the CTA's window does
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *const bars = reinterpret_cast<uint64_t *>(smem + Smem<DT>::OFF_BARS);
    uint32_t &tmem_base_sh = *reinterpret_cast<uint32_t *>(smem + Smem<DT>::OFF_TMEM);
    float *const m_sh = reinterpret_cast<float *>(smem + Smem<DT>::OFF_M);
    float2(*const ml_sh)[BM] = reinterpret_cast<float2(*)[BM]>(smem + Smem<DT>::OFF_ML);
    const uint32_t sbase = smem_u32(smem);
    if ((sbase & 1023u) != 0u) {  // the swizzled boxes need it; the same for every thread
        if (threadIdx.x == 0) atomicOr(&g_ris_tile_error, 2u);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // ---- tile of this CTA (tiles covering rows row0 .. row1-1): heavier (later) tiles first
    const int qt_end = (int)((a.row1 + BM - 1) / BM);
    const int64_t b = blockIdx.x;
    const int h = (int)(b % a.Hq);
    const int64_t r2 = b / a.Hq;
    const int s = (int)(r2 % a.n_sets);
    const int qt = qt_end - 1 - (int)(r2 / a.n_sets);
    const int64_t q0 = (int64_t)qt * BM;
    const int g = h / a.G;
    const int mask_id = s * a.heads_keyed + (a.heads_keyed > 1 ? g : 0);
    const int64_t last_row = (q0 + BM - 1 < a.row1 - 1) ? q0 + BM - 1 : a.row1 - 1;
    // causal: key tiles kt0 .. last_row / BN (kt0 = 0, or the tile of the first row's dense
    // suffix start, the earliest of the tile's rows)
    const int kt0 = SUFFIX ? (int)(dense_suffix_start(a, q0) / BN) : 0;
    const int n_kt = (int)(last_row / BN) + 1 - kt0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBAR; ++i) {
            uint32_t cnt = 1;
            if (i == B_Q) cnt = kSoftmaxThreads;
            if (i == B_S_READ || i == B_S_READ + 1) cnt = kGroupWarps;
            if (i == B_P_FULL || i == B_P_FULL + 1) cnt = kGroupWarps + 1;  // + the loader's relay
            mbar_init(smem_u32(&bars[i]), cnt);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kMmaWarp) {  // TMEM allocation by one full warp
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // all 512 columns: the allocation starts at TMEM address 0, so every address below is a
    // constant (anything else ends the CTA as a failed wait does, below)
    constexpr uint32_t T_S0 = 0, T_O = T_S0 + 2 * BN, T_Q = T_O + DT, T_P = T_Q + DT / 2;
    static_assert(T_P + BN / 2 <= kTmemCols, "TMEM columns");
    const uint32_t tmem = tmem_base_sh;
    constexpr auto BAR = [](int i) { return (uint32_t)(Smem<DT>::OFF_BARS + 8 * i); };
    const long long wl = a.wait_limit > 0 ? (long long)a.wait_limit : (1LL << 31);
    bool ok = tmem == 0u;

    if (warp >= kSoftmaxWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (!ok) {
        // unexpected TMEM base: straight to the common end
    } else if (warp == kTmaWarp) {
        // =============================== TMA producer
        if (lane == 0 && a.debug_no_loads == 0) {
            // Keys of tile j once the score products of tile j - 2 are done, values of tile j once the
            // value product of tile j - 2 is. The ring stages and the score buffers are both
            // indexed by tile parity, so the loader waits on the barriers that announce those
            // products (S_FULL, PV_DONE) instead of on barriers of its own, which saves the tensor
            // pipe two commits per tile. The keys are requested ahead of the values: the score
            // products of tile t + 1 finish before the value product of tile t - 2, so in this
            // order no wait holds up a load that could go before it.
            // The loader also waits for each tile's values to land and then arrives on that tile's
            // P_FULL (which counts the softmax warps and this one), so that the MMA warp waits
            // once before a value product instead of twice.
            static_assert(kStages == 2, "ring stages share the parity of the score buffers");
            int nk = 0, nv = 0, nr = 0;  // tiles whose keys / values were requested; values relayed
            auto load_k = [&](int j) {
                const uint32_t bk = smem_u32(&bars[B_K_FULL + j % kStages]);
                const uint32_t dk = sbase + OFF_K + (j % kStages) * K_STAGE;
                mbar_arrive_expect_tx(bk, (SPLIT ? 2 : 1) * KV_ARR);
                for (int blk = 0; blk < NB; ++blk) {
                    tma_load_3d(dk + blk * KV_BLK, &maps.kh, 64 * blk, g, (kt0 + j) * BN, bk);
                    if (SPLIT) tma_load_3d(dk + KV_ARR + blk * KV_BLK, &maps.kl, 64 * blk, g, (kt0 + j) * BN, bk);
                }
                nk = j + 1;
            };
            auto load_v = [&](int j) {
                const uint32_t bv = smem_u32(&bars[B_V_FULL + j % kStages]);
                const uint32_t dv = sbase + OFF_V + (j % kStages) * V_STAGE;
                mbar_arrive_expect_tx(bv, KV_ARR);
                for (int blk = 0; blk < NB; ++blk) tma_load_3d(dv + blk * KV_BLK, &maps.v, 64 * blk, g, (kt0 + j) * BN, bv);
                nv = j + 1;
            };
            auto relay = [&](int jv) -> bool {
                if (!mbar_wait(smem_u32(&bars[B_V_FULL + jv % kStages]), (jv / kStages) & 1, wl)) return false;
                mbar_arrive(smem_u32(&bars[B_P_FULL + (jv & 1)]));
                nr = jv + 1;
                return true;
            };
            for (int j = 0; j < kStages && j < n_kt; ++j) {
                load_k(j);
                load_v(j);
            }
            auto next_k = [&](int j) -> bool {  // into the stage that tile j - 2 leaves
                if (j >= n_kt) return true;
                if (!mbar_wait(smem_u32(&bars[B_S_FULL + (j & 1)]), ((j - kStages) >> 1) & 1, wl)) return false;
                load_k(j);
                return true;
            };
            ok = next_k(kStages);
            for (int t = 0; t < n_kt && ok; ++t) {
                ok = next_k(t + kStages + 1);
                if (ok && t >= 1) ok = relay(t - 1);
                if (!ok) break;
                if (t >= kStages) {
                    ok = mbar_wait(smem_u32(&bars[B_PV_DONE + (t & 1)]), ((t - kStages) >> 1) & 1, wl);
                    if (!ok) break;
                    load_v(t);
                }
            }
            if (ok && nr < n_kt) ok = relay(n_kt - 1);
            // let the copies requested last into each stage land before the CTA can leave
            // (earlier ones were consumed before their stage was refilled)
            for (int j = nk - kStages; j < nk; ++j)
                if (j >= 0) mbar_wait_own(smem_u32(&bars[B_K_FULL + j % kStages]), (j / kStages) & 1);
            for (int j = nv - kStages; j < nv; ++j)
                if (j >= 0) mbar_wait_own(smem_u32(&bars[B_V_FULL + j % kStages]), (j / kStages) & 1);
        }
    } else if (warp == kMmaWarp) {
        // =============================== MMA issuer
        // The whole warp runs this code, so that every operand is warp-uniform, and one elected
        // lane issues: inside a branch on the lane the compiler moves each of a product's operands
        // (two descriptors, two TMEM addresses, the instruction descriptor) into uniform registers
        // one by one, about 60 cycles per product, as long as a 128 x 128 x 16 product itself.
        constexpr uint32_t ID_S = idesc_bf16(BM, BN, false);  // S[128 x 128] = Q K^T, both K-major
        constexpr uint32_t ID_SH = idesc_f16(BM, BN, false);  // fp16 x fp16 (and e4m3 x e4m3 for kind::f8f6f4)
        constexpr uint32_t ID_O = idesc_f16(BM, DT, true);    // O[128 x DT] += P V, fp16, V MN-major
        // fp8-correction scores (rotated q / k at head dim 128, operands written by
        // launch_fp8_prep when the bounds allow): the same bytes in the same places as the
        // bf16 pair, read as fp16 hi parts (query in TMEM, key bytes 0-255 of a row) and e4m3
        // corrections (the 64-column blocks of the query's low part in shared memory and of
        // the key's at KV_ARR: hi parts, then lo parts)
        int ea = 0, eb = 0;
        const bool use8 = DT == 128 && SPLIT && a.qk_bound != nullptr &&
                          __any_sync(0xFFFFFFFFu, fp8_score_scales(a.qk_bound[0], a.qk_bound[1], ea, eb));
        // score products of a tile whose parity (ring stage and score buffer) is ST
        auto issue_s = [&](auto st_c) {
            constexpr int ST = decltype(st_c)::value;
            const uint32_t kd = desc_lo(sbase + OFF_K + ST * K_STAGE, 16);  // K hi; K lo KV_ARR on
            const uint32_t qd = desc_lo(sbase + OFF_Q, 16);                  // Q lo
            constexpr uint32_t dt = T_S0 + ST * BN;
            if (elect_one()) {
                if (use8) {
                    // 2^12 (q_h8 k_l8 + q_l8 k_h8): two e4m3 products of 4 k-steps of 32
#pragma unroll
                    for (int ks = 0; ks < DT / 32; ++ks)
                        tc_mma_ss_f8(dt, qd + dstep(ks * 32), kd + dstep(KV_ARR + KV_BLK + ks * 32), ID_SH, ks > 0);
#pragma unroll
                    for (int ks = 0; ks < DT / 32; ++ks)
                        tc_mma_ss_f8(dt, qd + dstep(KV_BLK + ks * 32), kd + dstep(KV_ARR + ks * 32), ID_SH, 1u);
                    // + q_h k_h in fp16, the corrections brought back by 2^-12 on the first k-step
#pragma unroll
                    for (int ks = 0; ks < DT / 16; ++ks) {
                        const uint32_t bd = kd + dstep((ks >> 2) * KV_BLK + (ks & 3) * 32);
                        if (ks == 0)
                            tc_mma_ts_scaled12(dt, T_Q, bd, ID_SH);
                        else
                            tc_mma_ts(dt, T_Q + 8 * ks, bd, ID_SH, 1u);
                    }
                } else {
                    // (A, B) pairs: (Q hi, K hi), (Q lo, K hi), (Q hi, K lo); k-steps of 16 over D,
                    // 16 columns = 32 B inside a 128 B row. The query's high part lives in TMEM
                    // (16-bit values packed two per column), its low part in shared memory
#pragma unroll
                    for (int prod = 0; prod < (SPLIT ? 3 : 1); ++prod)
#pragma unroll
                        for (int ks = 0; ks < DT / 16; ++ks) {
                            const int koff = (ks >> 2) * KV_BLK + (ks & 3) * 32;
                            const uint32_t bd = kd + dstep((prod == 2 ? KV_ARR : 0) + koff);
                            if (prod == 1)
                                tc_mma_ss(dt, qd + dstep(koff), bd, ID_S, 1u);
                            else
                                tc_mma_ts(dt, T_Q + 8 * ks, bd, ID_S, prod > 0 || ks > 0);
                        }
                }
                tc_commit(sbase + BAR(B_S_FULL + ST));
            }
            __syncwarp();
        };
        // value product of a tile of parity ST: P, 128 keys of fp16 values packed two per column,
        // times V, 64 keys x 128 B rows per block: 16 keys = two 8-row atoms (SBO 1024); the
        // second 64-column block of head dim is LBO = 16 KB away
        auto issue_o = [&](auto st_c, uint32_t acc) {
            constexpr int ST = decltype(st_c)::value;
            const uint32_t vd = desc_lo(sbase + OFF_V + ST * V_STAGE, KV_BLK);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < BN / 16; ++ks)
                    tc_mma_ts(T_O, T_P + 8 * ks, vd + dstep(ks * 2048), ID_O, ks > 0 ? 1u : acc);
                tc_commit(sbase + BAR(B_PV_DONE + ST));
            }
            __syncwarp();
        };
        auto wait_all = [&](int bar, int parity) -> bool {
            const bool got = __all_sync(0xFFFFFFFFu, mbar_wait(sbase + BAR(bar), parity, wl));
            tc_fence_after();
            return got;
        };
        // score products of tile j (parity ST) into the buffer that tile j - 2 has been read out of
        auto next_s = [&](auto st_c, int j) -> bool {
            constexpr int ST = decltype(st_c)::value;
            const int par = (j >> 1) & 1;
            if (!wait_all(B_K_FULL + ST, par)) return false;
            if (j >= 2 && !wait_all(B_S_READ + ST, par ^ 1)) return false;
            issue_s(st_c);
            return true;
        };
        // Tile j, parity ST: the scores of tile j + 3 (the other group reads tile j + 1 out while
        // this one forms P of tile j), so that scores are always there when a group comes for
        // them; then, with P of tile j written and its values landed (relayed by the loader), its
        // value product.
        auto tile_step = [&](auto st_c, auto other_c, int j) {
            constexpr int ST = decltype(st_c)::value;
            if (j + 3 < n_kt) ok = next_s(other_c, j + 3);
            if (!ok) return;
            ok = wait_all(B_P_FULL + ST, (j >> 1) & 1);
            if (ok) issue_o(st_c, j > 0 ? 1u : 0u);
        };
        constexpr std::integral_constant<int, 0> even{};
        constexpr std::integral_constant<int, 1> odd{};
        ok = wait_all(B_Q, 0) && next_s(even, 0);
        if (ok && n_kt > 1) ok = next_s(odd, 1);
        if (ok && n_kt > 2) ok = next_s(even, 2);
        for (int j = 0; j < n_kt && ok; j += 2) {
            tile_step(even, odd, j);
            if (ok && j + 1 < n_kt) tile_step(odd, even, j + 1);
        }
        // every product issued has to finish before TMEM is released
        if (elect_one()) tc_commit(sbase + BAR(B_END));
        __syncwarp();
        mbar_wait_own(sbase + BAR(B_END), 0);
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
        // this thread's half of the query row: the high part into TMEM (OC / 2 packed columns)
        {
            const int64_t qrow = ((row_ok ? i : 0) * a.Hq + h) * DT + OC * grp;
            const uint4 *src = reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(q_hi) + qrow);
            uint32_t qw[OC / 2];
#pragma unroll
            for (int u = 0; u < OC / 8; ++u) {
                const uint4 x = row_ok ? src[u] : make_uint4(0u, 0u, 0u, 0u);
                qw[4 * u] = x.x;
                qw[4 * u + 1] = x.y;
                qw[4 * u + 2] = x.z;
                qw[4 * u + 3] = x.w;
            }
            const uint32_t tq = T_Q + lane_off + (OC / 2) * grp;
#pragma unroll
            for (int c = 0; c < OC / 2; c += 16) tmem_st16(tq + c, qw + c);
            if (SPLIT) {
                // the low part as the K-major A operand in shared memory: 64-column blocks of 128
                // rows of 128 bytes, 16-byte pieces swizzled by the row
                src = reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(q_lo) + qrow);
#pragma unroll
                for (int u = 0; u < OC / 8; ++u) {
                    const int piece = (OC / 8) * grp + u;
                    *reinterpret_cast<uint4 *>(smem + OFF_Q + (piece >> 3) * KV_BLK + r * 128 +
                                               (((piece & 7) ^ (r & 7)) << 4)) =
                        row_ok ? src[u] : make_uint4(0u, 0u, 0u, 0u);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&bars[B_Q]));
        }
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
        for (int j = grp; j < n_kt; j += 2) {
            const int par = (j >> 1) & 1;
            if (!kRange) mask_words(j + 4, nnw);
            if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&bars[B_S_FULL + grp]), par, wl));
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
            if (lane == 0) mbar_arrive(smem_u32(&bars[B_S_READ + grp]));
            float sv[BN];
#pragma unroll
            for (int c = 0; c < BN; ++c) sv[c] = __uint_as_float(su[c >> 6][c & 63]);
            if (!whole) {
#pragma unroll
                for (int c = 0; c < BN; ++c) sv[c] = ((cw[c >> 5] >> (c & 31)) & 1u) ? sv[c] : -INFINITY;
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
            // The row's reference maximum moves on from tile to tile, handed to the other group as
            // soon as it is known. Lazy rescale: it moves, and O is rescaled, only when the row max
            // grows by more than 2^8. The TMEM loads / stores are warp-collective
            // (.sync.aligned), so the whole warp runs them when any of its rows needs it; the
            // other rows multiply by 1.
            float m_prev = -INFINITY;
            if (j > 0) {
                pair_sync(1 + 2 * wq + (grp ^ 1));
                m_prev = m_sh[r];
            }
            const bool upd = mx > m_prev + 8.f;
            const float m_ref = upd ? mx : m_prev;
            if (j + 1 < n_kt) {
                m_sh[r] = m_ref;
                __threadfence_block();
                pair_arrive(1 + 2 * wq + grp);
            }
            if (!ok) continue;
            // the value product of tile j - 1 is done: O has settled, and P may be written over
            auto pv_done = [&]() -> bool {
                return j == 0 || __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&bars[B_PV_DONE + (grp ^ 1)]),
                                                                   ((j - 1) >> 1) & 1, wl));
            };
            const bool scale_o = upd && m_prev != -INFINITY;
            if (__any_sync(0xFFFFFFFFu, scale_o)) {
                ok = pv_done();
                if (!ok) continue;
                tc_fence_after();
                const float al = scale_o ? exp2f(m_prev - m_ref) : 1.f;
#pragma unroll 1
                for (int c0 = 0; c0 < DT; c0 += 16) {
                    float ov[16];
                    uint32_t ow[16];
                    tmem_ld16(T_O + lane_off + c0, ov);
#pragma unroll
                    for (int c = 0; c < 16; ++c) ow[c] = __float_as_uint(ov[c] * al);
                    tmem_st16(T_O + lane_off + c0, ow);
                }
            }
            if (m_ref != m_own) {
                l *= m_own == -INFINITY ? 0.f : exp2f(m_own - m_ref);
                m_own = m_ref;
            }
            const float mu = (m_ref == -INFINITY) ? 0.f : m_ref;
            // P = exp2(s - m_ref) as the A operand of the value product, packed two keys per
            // column. The row sum adds P as rounded, so that the rounding of each weight moves the
            // output by at most 2^-11 of the weight times |v_j - o| (a normalised average of the
            // values with slightly perturbed weights).
            uint64_t lsum[2] = {0ull, 0ull};
            const uint64_t nmu2 = f2_pack(-mu, -mu);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t hw[BN / 4];
#pragma unroll
                for (int w = 0; w < BN / 4; ++w) {
                    const int c = (BN / 2) * half + 2 * w;
                    float x0, x1;
                    f2_unpack(f2_fma(f2_pack(sv[c], sv[c + 1]), sc2, nmu2), x0, x1);
                    const __half2 hp = __floats2half2_rn(ex2(x0), ex2(x1));
                    const float2 pr = __half22float2(hp);
                    lsum[w & 1] = f2_add(lsum[w & 1], f2_pack(pr.x, pr.y));
                    hw[w] = *reinterpret_cast<const uint32_t *>(&hp);
                }
                if (half == 0) {
                    ok = pv_done();
                    if (!ok) break;
                    tc_fence_after();
                }
                tmem_st32(T_P + lane_off + (BN / 4) * half, hw);
            }
            if (!ok) continue;
            float la, lb;
            f2_unpack(f2_add(lsum[0], lsum[1]), la, lb);
            l += la + lb;
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars[B_P_FULL + grp]));
        }
        // the row's maximum and sum from both threads
        ml_sh[grp][r] = make_float2(m_own, l);
        ok = !pair_or(9 + wq, !ok);
        if (ok)
            ok = __all_sync(0xFFFFFFFFu,
                            mbar_wait(smem_u32(&bars[B_PV_DONE + ((n_kt - 1) & 1)]), ((n_kt - 1) >> 1) & 1, wl));
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
            TOut *out = SUFFIX ? reinterpret_cast<TOut *>(a.part_o + ((row_ok ? i : 0) * a.Hq + h) * DT + OC * grp)
                               : reinterpret_cast<TOut *>(a.out) + (((int64_t)s * a.N + (row_ok ? i : 0)) * a.Hq + h) * DT +
                                     OC * grp;
#pragma unroll
            for (int c0 = 0; c0 < OC; c0 += 32) {
                float ov[32];
                tmem_ld32(T_O + lane_off + OC * grp + c0, ov);
                if (row_ok) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) ov[c] *= inv;
#pragma unroll
                    for (int e = 0; e < 4; ++e) store8<TOut>(out + c0 + 8 * e, ov + 8 * e);
                }
            }
            if (SUFFIX) {
                if (row_ok && grp == 0) a.part_lse[i * a.Hq + h] = m_fin + __log2f(lt);
            } else if (row_ok && grp == 0 && a.lse != nullptr) {
                a.lse[((int64_t)s * a.Hq + h) * a.lse_ld + i] = (m_fin + __log2f(lt)) * kLn2;
            }
        }
    }

    if (!ok) atomicOr(&g_ris_tile_error, 2u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
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
cudaError_t launch_t(const AttnArgs &a, const TileMaps &maps, const void *q_hi, const void *q_lo, cudaStream_t s)
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
    const int64_t n_qt = (a.row1 + BM - 1) / BM - a.row0 / BM;  // tiles covering rows row0 .. row1-1
    const unsigned grid = (unsigned)(n_qt * a.Hq * a.n_sets);
    kern<<<grid, kThreads, SMEM_BYTES, s>>>(a, maps, q_hi, q_lo);
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

// K / V tensor maps of a call (the key low part only with split queries and keys; the values
// as fp16).
bool make_maps(TileMaps &maps, const AttnArgs &a, bool split, int D)
{
    if (a.v16 == nullptr || a.v_absmax == nullptr) return false;
    if (!make_map3(&maps.kh, a.k, a.N, a.Hkv, BN, D) || !make_map3(&maps.v, a.v16, a.N, a.Hkv, BN, D, true)) return false;
    if (split) return make_map3(&maps.kl, a.k_lo, a.N, a.Hkv, BN, D);
    maps.kl = maps.kh;
    return true;
}

template <int DT>
cudaError_t launch_tile_d(const AttnArgs &a, const TileMaps &maps, const void *q_hi, const void *q_lo, int out_dtype,
                          bool dense, cudaStream_t s)
{
    const bool split = q_lo != nullptr;
    if (out_dtype == RIS_F32) {
        if (split) return dense ? launch_t<DT, true, true, float>(a, maps, q_hi, q_lo, s) : launch_t<DT, true, false, float>(a, maps, q_hi, q_lo, s);
        return dense ? launch_t<DT, false, true, float>(a, maps, q_hi, q_lo, s) : launch_t<DT, false, false, float>(a, maps, q_hi, q_lo, s);
    }
    if (split)
        return dense ? launch_t<DT, true, true, __nv_bfloat16>(a, maps, q_hi, q_lo, s)
                     : launch_t<DT, true, false, __nv_bfloat16>(a, maps, q_hi, q_lo, s);
    return dense ? launch_t<DT, false, true, __nv_bfloat16>(a, maps, q_hi, q_lo, s)
                 : launch_t<DT, false, false, __nv_bfloat16>(a, maps, q_hi, q_lo, s);
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
    if (!make_maps(maps, a, q_lo != nullptr, D)) return cudaErrorInvalidValue;
    return D == 128 ? launch_tile_d<128>(a, maps, q_hi, q_lo, out_dtype, dense, s)
                    : launch_tile_d<64>(a, maps, q_hi, q_lo, out_dtype, dense, s);
}

cudaError_t launch_attention_tile_suffix(const AttnArgs &a, int D, const void *q_hi, const void *q_lo, cudaStream_t s)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    if (a.part_o == nullptr || a.part_lse == nullptr || a.n_sets != 1 || (D != 128 && D != 64))
        return cudaErrorInvalidValue;
    const bool split = q_lo != nullptr;
    alignas(64) TileMaps maps;
    if (!make_maps(maps, a, split, D)) return cudaErrorInvalidValue;
    if (D == 128)
        return split ? launch_t<128, true, false, float, true>(a, maps, q_hi, q_lo, s)
                     : launch_t<128, false, false, float, true>(a, maps, q_hi, q_lo, s);
    return split ? launch_t<64, true, false, float, true>(a, maps, q_hi, q_lo, s)
                 : launch_t<64, false, false, float, true>(a, maps, q_hi, q_lo, s);
}

}  // namespace ris
