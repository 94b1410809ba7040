// RIS sparse attention, fp32 inputs (paper, Methods, "Pre-Fusion Unified Softmax"): fp32
// FFMA throughout, no TF32, for the fp32 configuration whose bar is 1e-5 relative L2.
//
// One warp owns one task (row i, KV head g, output set s) and takes the row's keys 16 at a time:
//   scores   eight lanes share a key row (its 16-byte pieces interleaved over them, so that every
//            load reads whole 128-byte lines) and hold their D/8 elements of four keys, all in
//            flight at once; each lane multiplies them with all heads' queries (shared memory,
//            one 16-byte read per four keys), and a splitting butterfly over the eight lanes
//            leaves each lane the score of one head;
//   softmax  a lane holds four scores of its head; the probabilities go to shared memory, twice
//            each, as operands of the packed multiply-add;
//   values   every lane owns D/32 channels of all heads and adds p v key by key (coalesced rows,
//            four keys' loads in flight before they are used).
// Products and sums run as packed pairs of fp32 (fma.rn.f32x2, rounded as the scalar operation):
// half the issue slots. Bound by the L2 rows (2 D 4 B per pair and KV head) and the FFMA pipe
// alike; residency hides the load latency: three CTAs of four warps per SM, four with one or two
// heads in a group. (With six heads at N = 6007 two CTAs were 8% slower, four, which spill, 38%; one head at
// N = 2048 is 6% faster with four.) A lane per key row instead, 32 lines per load and groups padded to
// eight heads, took 492 us for 12 / 2 heads of 128, N = 6007, 4.9% of the pairs, and 50 us for one head,
// N = 2048, 5%; these layer calls take 249 and 28-31 us.
#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "attn_common.cuh"

namespace ris {
namespace {

__device__ __forceinline__ float2 f2_unpack(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ ulonglong2 ldg2x2(const float *p) { return __ldg(reinterpret_cast<const ulonglong2 *>(p)); }

// NG: compile-time bound on the query heads per KV head. The key lists (16 or 32 bits, or none
// for a dense mask) and the output type are looked at per step and per row: template parameters
// for them would multiply the kernels and save nothing.
template <int D, int NG>
__global__ void __launch_bounds__(kAttnWarps * 32, NG <= 2 ? 4 : 3) k_attn_f32(const AttnArgs a, int col_bytes, bool dense, bool out_bf16)
{
    constexpr int H = NG > 4 ? 8 : NG > 2 ? 4 : NG;  // heads of the butterfly: a power of two
    constexpr int KP = D / 32;                       // 16-byte pieces of a key row per lane
    constexpr int DL = D / 32;                       // channels per lane in the value sum
    __shared__ __align__(16) float qs[kAttnWarps][NG][D];
    __shared__ __align__(16) float2 ps[kAttnWarps][16][H];  // (p, p) of a key and head
    __shared__ __align__(16) float2 as[kAttnWarps][H];      // (al, al): rescale of a head's output

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l8 = lane & 7, kg = lane >> 3;
    const int64_t tid = (int64_t)blockIdx.x * kAttnWarps + warp;
    if (tid >= a.n_tasks) return;
    const Task t = decode_task(a, tid);
    int64_t beg, n64;
    if (dense)
        key_range<true>(a, t, beg, n64);
    else
        key_range<false>(a, t, beg, n64);
    const int n = (int)n64;  // a row holds fewer than 2^31 keys
    const uint16_t *col2 = reinterpret_cast<const uint16_t *>(a.col) + (dense ? 0 : beg);
    const uint32_t *col4 = reinterpret_cast<const uint32_t *>(a.col) + (dense ? 0 : beg);

    // the heads' queries; a lane reads elements 4 (8 u + l8) + [0, 4), u < KP
    const float *qg = reinterpret_cast<const float *>(a.q) + (t.i * a.Hq + (int64_t)t.g * a.G) * D;
    for (int e = 4 * lane; e < NG * D; e += 128)
        *reinterpret_cast<ulonglong2 *>(&qs[warp][0][0] + e) = e < a.G * D ? ldg2x2(qg + e) : make_ulonglong2(0ull, 0ull);

    const float *kbase = reinterpret_cast<const float *>(a.k) + (int64_t)t.g * D + 4 * l8;
    const float *vbase = reinterpret_cast<const float *>(a.v) + (int64_t)t.g * D + lane * DL;
    const int64_t rs = (int64_t)a.Hkv * D;
    // the head whose scores this lane ends up with (several lanes the same one when H < 8)
    const int my_h = l8 / (8 / H);
    uint64_t o[NG][DL / 2];
#pragma unroll
    for (int h = 0; h < NG; ++h)
#pragma unroll
        for (int e = 0; e < DL / 2; ++e) o[h][e] = 0ull;
    float m = -INFINITY, l = 0.f;

    auto key = [&](int pos) -> int {  // slots past the row read the row itself
        if (pos >= n) return (int)t.i;
        return dense ? pos : col_bytes == 2 ? (int)col2[pos] : (int)col4[pos];
    };
    int idx = key(lane & 15);
    // 16 keys from the row's position base on, fewer at the end of a row (FULL false)
    auto step = [&](auto full, int base) {
        constexpr bool FULL = decltype(full)::value;
        const int cnt = n - base;  // keys left
        const int next = key(base + 16 + (lane & 15));
        // scores of keys 4 r + kg at this lane's head
        float s[4];
        __syncwarp();  // the queries are there; the probabilities of the step before have been taken
        {
            ulonglong2 kb[4][KP];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float *kr = kbase + (int64_t)__shfl_sync(0xFFFFFFFFu, idx, 4 * r + kg) * rs;
#pragma unroll
                for (int u = 0; u < KP; ++u) kb[r][u] = ldg2x2(kr + 32 * u);
            }
            float sh[4][H];
#pragma unroll
            for (int h = 0; h < H; ++h) {
                if (h >= NG) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) sh[r][h] = 0.f;
                    continue;
                }
                uint64_t acc[4][2];
#pragma unroll
                for (int u = 0; u < KP; ++u) {
                    const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(&qs[warp][h][32 * u + 4 * l8]);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        acc[r][0] = u == 0 ? f2_mul(kb[r][u].x, q.x) : f2_fma(kb[r][u].x, q.x, acc[r][0]);
                        acc[r][1] = u == 0 ? f2_mul(kb[r][u].y, q.y) : f2_fma(kb[r][u].y, q.y, acc[r][1]);
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 x = f2_unpack(acc[r][0]), y = f2_unpack(acc[r][1]);
                    sh[r][h] = (x.x + x.y) + (y.x + y.y);
                }
            }
            // sums over the eight lanes of the row: while more than one head is left, a lane passes
            // half of its heads on and keeps the other half
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                int lanes = 4;
#pragma unroll
                for (int w = H; w > 1; w >>= 1) {
                    const bool hi = (lane & lanes) != 0;
#pragma unroll
                    for (int e = 0; e < w / 2; ++e) {
                        const float send = hi ? sh[r][e] : sh[r][e + w / 2], keep = hi ? sh[r][e + w / 2] : sh[r][e];
                        sh[r][e] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, lanes);
                    }
                    lanes >>= 1;
                }
#pragma unroll
                for (int w = 8 / H; w > 1; w >>= 1) {
                    sh[r][0] += __shfl_xor_sync(0xFFFFFFFFu, sh[r][0], lanes);
                    lanes >>= 1;
                }
                s[r] = FULL || 4 * r + kg < cnt ? sh[r][0] * a.scale_log2 : -INFINITY;
            }
        }

        // online softmax of this lane's head over the 16 keys (four here, four key groups)
        float mx = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 16));
        const float mn = fmaxf(m, mx);
        const float mu = (mn == -INFINITY) ? 0.f : mn;
        const float al = exp2f(m - mu);
        const bool moved = mn > m;
        m = mn;
        float sum = 0.f;
        const bool writer = (l8 & (8 / H - 1)) == 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float p = exp2f(s[r] - mu);
            sum += p;
            if (writer) ps[warp][4 * r + kg][my_h] = make_float2(p, p);
        }
        l = l * al + sum;
        if (writer && kg == 0) as[warp][my_h] = make_float2(al, al);
        __syncwarp();
        if (__any_sync(0xFFFFFFFFu, moved)) {
#pragma unroll
            for (int h = 0; h < NG; ++h) {
                const uint64_t f = *reinterpret_cast<const uint64_t *>(&as[warp][h]);
#pragma unroll
                for (int e = 0; e < DL / 2; ++e) o[h][e] = f2_mul(o[h][e], f);
            }
        }

        // values, four keys at a time
        uint64_t vb[2][4][DL / 2];
        auto load_v = [&](int r, uint64_t(&dst)[4][DL / 2]) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float *vr = vbase + (int64_t)__shfl_sync(0xFFFFFFFFu, idx, 4 * r + x) * rs;
                if constexpr (DL == 4) {
                    const ulonglong2 y = ldg2x2(vr);
                    dst[x][0] = y.x;
                    dst[x][1] = y.y;
                } else {
                    dst[x][0] = __ldg(reinterpret_cast<const unsigned long long *>(vr));
                }
            }
        };
        load_v(0, vb[0]);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (!FULL && 4 * r >= cnt) break;
            if (r + 1 < 4 && (FULL || 4 * (r + 1) < cnt)) load_v(r + 1, vb[(r + 1) & 1]);
            if (!FULL) {
                // slots past the row hold the row's own values, which may be infinite: p = 0 is not enough
#pragma unroll
                for (int x = 1; x < 4; ++x)
#pragma unroll
                    for (int e = 0; e < DL / 2; ++e)
                        if (4 * r + x >= cnt) vb[r & 1][x][e] = 0ull;
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int h = 0; h < NG; ++h) {
                    const uint64_t p = *reinterpret_cast<const uint64_t *>(&ps[warp][4 * r + x][h]);
#pragma unroll
                    for (int e = 0; e < DL / 2; ++e) o[h][e] = f2_fma(p, vb[r & 1][x][e], o[h][e]);
                }
        }
        idx = next;
    };
    // The full steps have a body of their own: setting aside the slots past the row in a common one takes the larger
    // groups 5% (12 / 2 heads, N = 6007: 274 us without, 288-292 with, 249 with two bodies); the
    // smaller ones are 1 us faster with one (one head, N = 2048: 29.4 against 31-32 us).
    int base = 0;
    if constexpr (NG > 2) {
#pragma unroll 1
        for (; base + 16 <= n; base += 16) step(std::true_type{}, base);
        if (base < n) step(std::false_type{}, base);
    } else {
#pragma unroll 1
        for (; base < n; base += 16) step(std::false_type{}, base);
    }

    // row sums over the key groups, normalise, store
    l += __shfl_xor_sync(0xFFFFFFFFu, l, 8);
    l += __shfl_xor_sync(0xFFFFFFFFu, l, 16);
    const int64_t orow = (((int64_t)t.s * a.N + t.i) * a.Hq + (int64_t)t.g * a.G) * D + lane * DL;
#pragma unroll
    for (int h = 0; h < NG; ++h) {
        if (h >= a.G) break;
        const float inv = 1.f / __shfl_sync(0xFFFFFFFFu, l, h * (8 / H));
        float x[DL];
#pragma unroll
        for (int e = 0; e < DL / 2; ++e) {
            const float2 y = f2_unpack(o[h][e]);
            x[2 * e] = y.x * inv;
            x[2 * e + 1] = y.y * inv;
        }
        const int64_t at = orow + (int64_t)h * D;
        if (out_bf16) {
            __nv_bfloat162 w[DL / 2];
#pragma unroll
            for (int e = 0; e < DL / 2; ++e) w[e] = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
            __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(a.out) + at;
            if constexpr (DL == 4)
                *reinterpret_cast<uint2 *>(dst) = *reinterpret_cast<const uint2 *>(w);
            else
                *reinterpret_cast<uint32_t *>(dst) = *reinterpret_cast<const uint32_t *>(w);
        } else {
            float *dst = reinterpret_cast<float *>(a.out) + at;
            if constexpr (DL == 4)
                *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
            else
                *reinterpret_cast<float2 *>(dst) = make_float2(x[0], x[1]);
        }
    }
    if (a.lse != nullptr && kg == 0 && (l8 & (8 / H - 1)) == 0 && my_h < a.G)
        a.lse[((int64_t)t.s * a.Hq + (int64_t)t.g * a.G + my_h) * a.lse_ld + t.i] = (m + log2f(l)) * kLn2;
}

template <int D>
cudaError_t launch_d(const AttnArgs &a, int out_dtype, int col_bytes, bool dense, cudaStream_t s)
{
    const unsigned grid = (unsigned)((a.n_tasks + kAttnWarps - 1) / kAttnWarps);
    const dim3 block(kAttnWarps * 32);
    const bool bf = out_dtype == RIS_BF16;
    if (a.G == 1)
        k_attn_f32<D, 1><<<grid, block, 0, s>>>(a, col_bytes, dense, bf);
    else if (a.G == 2)
        k_attn_f32<D, 2><<<grid, block, 0, s>>>(a, col_bytes, dense, bf);
    else if (a.G <= 4)
        k_attn_f32<D, 4><<<grid, block, 0, s>>>(a, col_bytes, dense, bf);
    else if (a.G <= 6)
        k_attn_f32<D, 6><<<grid, block, 0, s>>>(a, col_bytes, dense, bf);
    else
        k_attn_f32<D, 8><<<grid, block, 0, s>>>(a, col_bytes, dense, bf);
    note_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_attention_f32(const AttnArgs &a, int D, int out_dtype, int col_bytes, bool dense,
                                 cudaStream_t s)
{
    return D == 64 ? launch_d<64>(a, out_dtype, col_bytes, dense, s) : launch_d<128>(a, out_dtype, col_bytes, dense, s);
}

}  // namespace ris
