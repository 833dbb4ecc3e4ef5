// FP64-grade complex products of D >= 64 matrices on the digit products (pm_digits.cuh) with tcgen05: the 5th-generation
// tensor cores multiply f16 digits four times as fast as mma.sync, asynchronously, and keep the sums in tensor memory.
//
// Per 64 x 64 output block one chain of M = 128, K = 16 MMAs forms Re and Im at once,
//   [[Ar, -Ai], [Ai, Ar]] [Br; Bi]:  tensor-memory lanes 0..63 the rows of Re C, 64..127 those of Im C,
// with one f32 accumulator of 64 columns for each diagonal i + j = t of digit pairs (t = 0..7: all 512 columns).
// Up to 128 real terms (64 complex k) the sums are integers below 2^24, hence exact; longer products are read back
// every 64 k.  All warps convert a panel of 16 k of both operands to fixed point and store its digits as f16 in the
// canonical no-swizzle K-major layout (A: planes -Ai, Ar, Ai per digit, so both halves of the embedding are 128 consecutive
// rows; B: Br of every digit, then Bi) beside the MMAs of the panel before, which thread 0 issued (24 of them); then all
// warps read the accumulators back, add the diagonals in 64-bit integers and round.
//
// Bound by the integer instructions that split the operands and sum the diagonals, not by the MMAs (64 x 64 x 64: 96 MMAs,
// 8.7 k cycles at 4096 multiply-adds per cycle).  Blocks of 64 x 64 because the eight diagonals fill the tensor memory at
// 64 columns.  Measured (d = 40, N = 4000 / d = 128, N = 608; on the FP64 pipe 61 / 86 ms, mma.sync products of pm_fxl.cuh
// 7.0 / 13.4 ms): one MMA per digit pair, eight warps, doubles in and out 5.2 / 8.9 ms; sixteen warps 4.6 / 7.8 ms; up to
// four pairs per MMA (one thread issued 68 per panel, now 24) 3.9 / 7.2 ms; fixed-point operands and results
// (large_body_fx) 2.73 / 5.49 ms; the next panel converted by all warps beside the MMAs 2.70 / 5.28 ms.  At D = 32 an M = 128 tile would be half padding: pm_fxl.cuh stays there, in the trees and
// in the batched kernel (whose tensor memory belongs to its 3xTF32 products).
//
// Entries must be below 2 in magnitude; a NaN, an infinity or a larger entry makes the output block NaN.  Waits are
// bounded (pm_umma.cuh): once one gave up, the products leave their output as it was, and the callers turn the leaf or the
// gradient into NaN beside the status bit.
#pragma once

#include "pm_fxl.cuh"
#include "pm_umma.cuh"

namespace pm {
namespace fxu {

using fx::i64;
using fx::ND;

constexpr int BM = 64, KP = 16, KMAX = 64;                // output block, complex k per panel and per read-back
constexpr int PLANE = BM * KP * 2;                        // one digit of one part of 64 rows
constexpr int AB = 3 * PLANE, BB = 2 * PLANE;             // bytes per digit of A and of B
constexpr int STAGE = ND * (AB + BB);                     // 70 KB
constexpr int ITEMS = 2 * (BM * KP / 2);                  // pairs of a panel (A, then B)
constexpr int CROW = BM * 16 + 16;                        // row of the output in shared memory, padded
constexpr size_t BYTES = 2 * (size_t)STAGE;
static_assert(BM * CROW <= (int)BYTES, "the output fits in the stages");
static_assert(umma::Fmt<umma::kBF16x3>::SBO == 256 && umma::kLBO == 128 && umma::KC == KP, "descriptor of a 16-bit panel");

// f16 operands, f32 accumulators, M = 128
__device__ __forceinline__ uint32_t idesc(int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | (8u << 24); }

// sum of the diagonals in units of 2^-60; the accumulators hold plain integers, below 2^22 for t <= 2 (read from the
// bits after adding 1.5 2^23), below 2^24 for the others (converted)
__device__ __forceinline__ i64 collect(const float (&v)[fx::NA][8], int c) {
    constexpr uint32_t B = 0x4B400000u;
    const int32_t v0 = (int32_t)(__float_as_uint(v[0][c] + fx::kBias) - B);
    const int32_t v1 = (int32_t)(__float_as_uint(v[1][c] + fx::kBias) - B);
    const int32_t v2 = (int32_t)(__float_as_uint(v[2][c] + fx::kBias) - B);
    const int32_t v3 = __float2int_rn(v[3][c]), v4 = __float2int_rn(v[4][c]), v5 = __float2int_rn(v[5][c]);
    const int32_t v6 = __float2int_rn(fmaf(v[7][c], 0.00390625f, v[6][c]) * 0.0625f);  // units 2^-60
    i64 q = (i64)v5 * 16 + v6;
    q += (i64)v4 * 4096;
    q += (i64)v3 * (1 << 20);
    q += (i64)v2 * (1 << 28);
    return q + (i64)((unsigned long long)(long long)(v1 + v0 * 256) << 36);
}

__device__ __forceinline__ void ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// matrices of doubles, or of fixed-point numbers x = q 2^-56 (longlong2)
__device__ __forceinline__ i64 fixed(double v, bool &bad) { return fxl::to_fixed(v, bad); }
__device__ __forceinline__ i64 fixed(i64 v, bool &) { return v; }
__device__ __forceinline__ void result(i64 q, bool bad, double &v) { v = bad ? nan("") : fx::to_double<fx::FC>(q); }
__device__ __forceinline__ void result(i64 q, bool, i64 &v) { v = (q + 7 + ((q >> 4) & 1)) >> 4; }  // ties to even

// C = A B for one block of rows x cols (multiples of 16, at most 64), K a multiple of 16; add: C holds an earlier part of
// the sum over k.  All NT threads (256 or 512); starts after the caller's barrier and ends with one.
template <int NT, typename E>
__device__ __forceinline__ void block_mm(const E *A, int lda, const E *B, int ldb, E *C, int ldc, int K,
                                         int rows, int cols, unsigned char *smem, umma::Ctx &cx) {
    constexpr int PER = ITEMS / NT;   // pairs per thread and panel
    constexpr int W = 64 * 128 / NT;  // accumulator columns per warp
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (*(volatile int *)cx.abort) return;  // uniform: set before the last block barrier
    bool bad = false, any = false;
    // item w < 512: word w of the A planes (row 8 (w / 64) + (w / 4) % 8, k = 8 ((w / 32) % 2) + 2 (w % 4) and + 1), else the
    // same word of the B planes (column, k): a warp stores 32 consecutive words of every plane
    E v[PER][2];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int it = tid + NT * i, w = it & 511;
            const int r = 8 * (w >> 6) + ((w >> 2) & 7), k = k0 + 8 * ((w >> 5) & 1) + 2 * (w & 3);
            if (it < 512) {
                if (r < rows) {
                    v[i][0] = A[(size_t)r * lda + k];
                    v[i][1] = A[(size_t)r * lda + k + 1];
                }
            } else if (r < cols) {
                v[i][0] = B[(size_t)k * ldb + r];
                v[i][1] = B[(size_t)(k + 1) * ldb + r];
            }
        }
    };
    auto store = [&](int buf) {
        unsigned char *st = smem + (size_t)buf * STAGE;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int it = tid + NT * i, w = it & 511, r = 8 * (w >> 6) + ((w >> 2) & 7);
            if (r >= (it < 512 ? rows : cols)) continue;
            uint32_t re[ND], im[ND];
            fx::split_pair(fixed(v[i][0].x, bad), fixed(v[i][1].x, bad), re);
            fx::split_pair(fixed(v[i][0].y, bad), fixed(v[i][1].y, bad), im);
            if (it < 512) {
                uint32_t *p = (uint32_t *)st + w;
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    p[d * (AB / 4)] = fx::neg2(im[d]);
                    p[d * (AB / 4) + PLANE / 4] = re[d];
                    p[d * (AB / 4) + 2 * (PLANE / 4)] = im[d];
                }
            } else {
                uint32_t *p = (uint32_t *)(st + ND * AB) + w;
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    p[d * (PLANE / 4)] = re[d];
                    p[(ND + d) * (PLANE / 4)] = im[d];
                }
            }
        }
    };
    // One digit i of A against up to four consecutive digits of B: their planes are consecutive rows, and the accumulators of
    // the diagonals i + j, i + j + 1, ... consecutive columns, so one MMA of N = 256 takes four digit pairs.  Diagonal 7
    // starts with the pair (1, 6), the others with i = 0.
    auto issue = [&](int buf, bool fresh) {
        const uint32_t sa = umma::smem_u32(smem + (size_t)buf * STAGE), sb = sa + ND * AB;
        auto group = [&](int h, int i, int j, int n, bool first) {  // h: [Ar; Ai] Br, then [-Ai; Ar] Bi
            umma::mma<umma::kBF16x3>(cx.tmem + (uint32_t)(BM * (i + j)),
                                     umma::desc<umma::kBF16x3>(sa + i * AB + (h ? 0 : PLANE)),
                                     umma::desc<umma::kBF16x3>(sb + (h * ND + j) * PLANE), idesc(BM * n), first ? 0u : 1u);
        };
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                const bool f = fresh && h == 0;
                const int n = fx::last_digit(i) + 1, m = i == 1 ? n - 1 : n;  // i = 1: the pair (1, 6) by itself
#pragma unroll
                for (int j = 0; j < m; j += 4) group(h, i, j, m - j < 4 ? m - j : 4, f && i == 0);
                if (i == 1) group(h, 1, ND - 1, 1, f);
            }
    };

    const int row = (warp & 3) * 32 + lane;  // tensor-memory lane: Re row, or 64 + Im row
    const int r = row & 63, part = row >> 6, ch = (warp >> 2) * W;
    i64 o[W];
#pragma unroll
    for (int c = 0; c < W; ++c) o[c] = 0;

    const int np = K / KP;
    uint32_t used[2] = {cx.cnt[umma::kBarDone], cx.cnt[umma::kBarDone + 1]};  // completions before panel p of each stage
    auto stage = [&](int p) {  // panel p into its stage, panel p + 1 on its way
        store(p & 1);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        if (p + 1 < np) load((p + 1) * KP);
    };
    load(0);
    stage(0);
    any = __syncthreads_or(bad);
    for (int p = 0; p < np; ++p) {
        const int buf = p & 1;
        if (tid == 0) {
            umma::fence_after();
            issue(buf, (p * KP) % KMAX == 0);
            umma::commit(cx.bar + umma::kBarDone + buf);
        }
        __syncwarp();
        if (p + 1 < np) {  // beside the MMAs of panel p, once those of panel p - 1 have left the stage
            if (p >= 1) umma::wait_idx(cx, umma::kBarDone + (buf ^ 1), used[buf ^ 1] + (p - 1) / 2);
            stage(p + 1);
        }
        if (p + 1 == np || ((p + 1) * KP) % KMAX == 0) {  // read back
            umma::wait_idx(cx, umma::kBarDone + buf, used[buf] + p / 2);
            umma::fence_after();
            if (!__any_sync(0xffffffffu, *(volatile int *)cx.abort)) {
                const uint32_t tl = cx.tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
                for (int g = 0; g < W; g += 8) {
                    if (ch + g >= cols) break;
                    float x[fx::NA][8];
#pragma unroll
                    for (int t = 0; t < fx::NA; ++t) ld8(tl + (uint32_t)(64 * t + ch + g), x[t]);
                    umma::wait_ld();
#pragma unroll
                    for (int c = 0; c < 8; ++c) o[g + c] += collect(x, c);
                }
            }
            umma::fence_before();
        }
        any = __syncthreads_or(bad) || any;  // panel p + 1 is staged, and every accumulator read before a next part starts
    }
    cx.cnt[umma::kBarDone] += (np + 1) / 2;
    cx.cnt[umma::kBarDone + 1] += np / 2;
    // out through the idle stages (every MMA has completed), coalesced
    if (!__syncthreads_or(*(volatile int *)cx.abort)) {
        auto *dst = &reinterpret_cast<E *>(smem + (size_t)r * CROW)->x + part;
#pragma unroll
        for (int c = 0; c < W; ++c) result(o[c], any, dst[2 * (ch + c)]);
        __syncthreads();
        for (int i = tid >> 4; i < rows; i += NT / 16)
            for (int j = tid & 15; j < cols; j += 16)
                C[(size_t)i * ldc + j] = *reinterpret_cast<const E *>(smem + (size_t)i * CROW + j * 16);
    }
    __syncthreads();
}

// C = A B for D x D matrices (row stride D) of true dimension d by the whole block (fxl::cta_mm's contract)
template <int D, int NT, typename E>
__device__ __noinline__ void cta_mm(const E *A, const E *B, E *C, unsigned char *smem, int d, umma::Ctx &cx) {
    const int n = fxl::extent(d);
#pragma unroll 1
    for (int i = 0; i < n; i += BM)
#pragma unroll 1
        for (int j = 0; j < n; j += BM)
            block_mm<NT, E>(A + (size_t)i * D, D, B + j, D, C + (size_t)i * D + j, D, n, min(BM, n - i), min(BM, n - j), smem, cx);
}

}  // namespace fxu
}  // namespace pm
