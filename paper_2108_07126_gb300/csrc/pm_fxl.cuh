// FP64-grade complex products of D >= 32 matrices by a thread block, on the digit products of pm_digits.cuh:
// the matrices stay doubles in global memory, a k-panel of both operands is converted to fixed point and split
// into digits while it is staged in shared memory, the warps multiply the digits with mma.sync and keep the
// output in 64-bit integers (collected once per panel of 16 complex k, the bound under which the f32 sums are
// exact), and the result is rounded to doubles at the end.
//
// Entries must be below 2 in magnitude (exponents, polynomials and propagators are); a NaN, an infinity or a
// larger entry in an operand makes the whole output block NaN.
//
// Bound by the tensor pipe: a 64 x 64 product is 17 408 MMAs (34.8 k cycles at one m16n8k16 per two cycles and SM)
// against 0.6 M cycles for its 10^6 multiply-adds on the FP64 pipe.  The staging (conversion and split of the next panel) is
// spread between the MMA tiles.  Used at D = 32, in the trees and scans, and by the batched kernel; single calls with
// D >= 64 run their slices on tcgen05 (pm_fxu.cuh).  d = 23 gradient, N = 1000: 11.0 -> 2.7 ms with these products.
#pragma once

#include "pm_fx.cuh"

namespace pm {
namespace fxl {

using fx::i64;
using fx::ND;
using fx::u64;

constexpr int kThreads = 256;
constexpr int KP = 16;  // complex k per panel

// Output block BM x BM of a product, eight warps: RB row blocks of 16 rows, the other warps share the columns.
template <int BM> struct G {
    static constexpr int RB = BM / 16, NT = BM / 8;
    static constexpr int WC = 8 / RB;       // column warps
    static constexpr int NTW = NT / WC;     // column tiles of eight per warp
    static constexpr int AW = RB * 2 * ND * 32 * 4, BW = NT * 2 * ND * 32 * 2;  // words of a staged panel
    static constexpr int IA = RB * 128 / kThreads, IB = NT * 64 / kThreads;     // pairs per thread and panel
    static constexpr size_t BYTES = (size_t)2 * (AW + BW) * 4;                    // double-buffered
};
template <int D> __host__ __device__ constexpr int block_of() { return D >= 64 ? 64 : 32; }
template <int D> __host__ __device__ constexpr size_t mm_bytes() { return G<block_of<D>()>::BYTES; }

__device__ __forceinline__ i64 to_fixed(double v, bool &bad) {
    const u64 b = (u64)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    bad = bad || e >= 1024;
    const u64 m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = e - 1075 + fx::F;  // <= 4 for |v| < 2
    const u64 q = sh >= 0 ? m << (sh & 7) : (sh > -60 ? fx::round_even(m, -sh) : 0ull);
    return (i64)b < 0 ? -(i64)q : (i64)q;
}

// COMPACT: fewer registers (one part of A at a time, the parts in a loop).  For the batched FP32 kernel: with the full form in its
// tree, ptxas spilled in the items of small d (64 instances, d = 4, N = 10 000: 385 -> 568 us, with this one 410 us).
// C = A B for one block of at most BM x BM: A is rows x K (row stride lda), B is K x cols (ldb), C (ldc) must not
// alias them; rows, cols and K are multiples of 16 (BM = 32: rows and cols full).  All 256 threads; smem:
// G<BM>::BYTES.  Starts after the caller's barrier and ends with one.
template <int BM, bool COMPACT = false>
__device__ __forceinline__ void block_mm(const double2 *A, int lda, const double2 *B, int ldb, double2 *C, int ldc, int K,
                                         unsigned char *smem, int rows = BM, int cols = BM) {
    using g = G<BM>;
    constexpr int NTW = g::NTW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rb = warp % g::RB, cw = warp / g::RB;
    const int nrb = BM == 32 ? g::RB : rows / 16, ntw = BM == 32 ? NTW : cols / 16;  // active row blocks, tiles per warp
    uint32_t *st = (uint32_t *)smem;
    bool bad = false;

    // staging: thread word w of A is register reg of lane l2 of row block w / 128 (rows l2 / 4 + 8 (reg & 1), k =
    // 2 (l2 & 3) + 8 (reg >> 1) and + 1), so that a warp stores 32 consecutive words of every digit plane
    double2 va[g::IA][2], vb[g::IB][2];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < g::IA; ++i) {
            const int w = tid + kThreads * i, l2 = (w & 127) >> 2, reg = w & 3;
            if ((w >> 7) >= nrb) continue;
            const int r = 16 * (w >> 7) + (l2 >> 2) + 8 * (reg & 1), k = k0 + 2 * (l2 & 3) + 8 * (reg >> 1);
            va[i][0] = A[(size_t)r * lda + k];
            va[i][1] = A[(size_t)r * lda + k + 1];
        }
#pragma unroll
        for (int i = 0; i < g::IB; ++i) {
            const int w = tid + kThreads * i, l2 = (w & 63) >> 1, reg = w & 1;
            if ((w >> 6) >= g::WC * ntw) continue;
            const int n = 8 * (w >> 6) + (l2 >> 2), k = k0 + 2 * (l2 & 3) + 8 * reg;
            vb[i][0] = B[(size_t)k * ldb + n];
            vb[i][1] = B[(size_t)(k + 1) * ldb + n];
        }
    };
    auto put = [&](uint32_t *s, int stride, const double2 (&v)[2]) {
        uint32_t d[ND];
        fx::split_pair(to_fixed(v[0].x, bad), to_fixed(v[1].x, bad), d);
#pragma unroll
        for (int i = 0; i < ND; ++i) s[2 * i * stride] = d[i];
        fx::split_pair(to_fixed(v[0].y, bad), to_fixed(v[1].y, bad), d);
#pragma unroll
        for (int i = 0; i < ND; ++i) s[(2 * i + 1) * stride] = d[i];
    };
    // piece k of a panel: the thread's k-th pair of A, then of B
    constexpr int PIECES = g::IA + g::IB;
    auto store_piece = [&](int buf, int k) {
        uint32_t *sa = st + buf * (g::AW + g::BW), *sb = sa + g::AW;
        const int w = tid + kThreads * (k < g::IA ? k : k - g::IA);
        if (k < g::IA) {
            if ((w >> 7) < nrb) put(sa + (w >> 7) * (2 * ND * 128) + (w & 127), 128, va[k < g::IA ? k : 0]);
        } else if ((w >> 6) < g::WC * ntw) {
            put(sb + (w >> 6) * (2 * ND * 64) + (w & 63), 64, vb[k < g::IA ? 0 : k - g::IA]);
        }
    };

    i64 o[NTW][2][4];
#pragma unroll
    for (int t = 0; t < NTW; ++t)
#pragma unroll
        for (int pt = 0; pt < 2; ++pt)
#pragma unroll
            for (int u = 0; u < 4; ++u) o[t][pt][u] = 0;

    load(0);
#pragma unroll
    for (int k = 0; k < PIECES; ++k) store_piece(0, k);
    bool any = __syncthreads_or(bad);
    for (int kp = 0; kp < K / KP; ++kp) {
        const bool more = kp + 1 < K / KP;
        if (more) load((kp + 1) * KP);
        const uint32_t *sa = st + (kp & 1) * (g::AW + g::BW), *sb = sa + g::AW;
        fx::Digits<16> a;
        if constexpr (!COMPACT) {
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const uint4 x = *reinterpret_cast<const uint4 *>(sa + rb * (2 * ND * 128) + 2 * i * 128 + lane * 4);
            const uint4 y = *reinterpret_cast<const uint4 *>(sa + rb * (2 * ND * 128) + (2 * i + 1) * 128 + lane * 4);
            a.re[i][0] = x.x; a.re[i][1] = x.y; a.re[i][2] = x.z; a.re[i][3] = x.w;
            a.im[i][0] = y.x; a.im[i][1] = y.y; a.im[i][2] = y.z; a.im[i][3] = y.w;
        }
        }
#pragma unroll
        for (int t = 0; t < NTW; ++t) {
            // the next panel is converted and stored piece by piece between the tiles, beside the MMAs
            if (more) {
#pragma unroll
                for (int k = t * PIECES / NTW; k < (t + 1) * PIECES / NTW; ++k) store_piece((kp + 1) & 1, k);
            }
            if (t >= ntw || rb >= nrb) continue;
            const uint32_t *sn = sb + (cw * ntw + t) * (2 * ND * 64) + lane * 2;
            if constexpr (COMPACT) {
#pragma unroll 2
                for (int pt = 0; pt < 2; ++pt) {
                    float acc[fx::NA][4];
                    fx::acc_init(acc);
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {  // Ar, then Ai
                        uint4 x[ND];
                        uint2 b[ND];
                        const uint32_t neg = h == 1 && pt == 0 ? 0x80008000u : 0u;
#pragma unroll
                        for (int i = 0; i < ND; ++i) x[i] = *reinterpret_cast<const uint4 *>(sa + rb * (2 * ND * 128) + (2 * i + h) * 128 + lane * 4);
#pragma unroll
                        for (int j = 0; j < ND; ++j) {
                            b[j] = *reinterpret_cast<const uint2 *>(sn + (2 * j + (h ^ pt)) * 64);
                            b[j].x ^= neg;
                            b[j].y ^= neg;
                        }
#pragma unroll
                        for (int i = 0; i < ND; ++i)
#pragma unroll
                            for (int j = 0; j <= fx::last_digit(i); ++j) fx::mma(acc[i + j], x[i].x, x[i].y, x[i].z, x[i].w, b[j].x, b[j].y);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[t][pt][u] += fx::collect_fine(acc, u);
                }
                continue;
            }
#pragma unroll
            for (int pt = 0; pt < 2; ++pt) {  // Re: Ar Br + Ai (-Bi); Im: Ar Bi + Ai Br
                float acc[fx::NA][4];
                uint2 b[ND];
#pragma unroll
                for (int j = 0; j < ND; ++j) b[j] = *reinterpret_cast<const uint2 *>(sn + (2 * j + pt) * 64);
#pragma unroll
                for (int i = 0; i < ND; ++i)
#pragma unroll
                    for (int j = 0; j <= fx::last_digit(i); ++j) {
                        if (fx::first_pair(i, j)) fx::mma_first(acc[i + j], a.re[i][0], a.re[i][1], a.re[i][2], a.re[i][3], b[j].x, b[j].y, fx::acc_start(i + j));
                        else fx::mma(acc[i + j], a.re[i][0], a.re[i][1], a.re[i][2], a.re[i][3], b[j].x, b[j].y);
                    }
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    b[j] = *reinterpret_cast<const uint2 *>(sn + (2 * j + 1 - pt) * 64);
                    if (pt == 0) {
                        b[j].x = fx::neg2(b[j].x);
                        b[j].y = fx::neg2(b[j].y);
                    }
                }
#pragma unroll
                for (int i = 0; i < ND; ++i)
#pragma unroll
                    for (int j = 0; j <= fx::last_digit(i); ++j)
                        fx::mma(acc[i + j], a.im[i][0], a.im[i][1], a.im[i][2], a.im[i][3], b[j].x, b[j].y);
#pragma unroll
                for (int u = 0; u < 4; ++u) o[t][pt][u] += fx::collect_fine(acc, u);
            }
        }
        any = __syncthreads_or(bad) || any;
    }
    const double nanv = any ? nan("") : 0.0;
#pragma unroll
    for (int t = 0; t < NTW; ++t)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (t >= ntw || rb >= nrb) continue;
            const int r = 16 * rb + (lane >> 2) + 8 * (u >> 1), c = 8 * (cw * ntw + t) + 2 * (lane & 3) + (u & 1);
            double2 v = make_double2(fx::to_double<fx::FC>(o[t][0][u]), fx::to_double<fx::FC>(o[t][1][u]));
            if (any) v = make_double2(nanv, nanv);
            C[(size_t)r * ldc + c] = v;
        }
    __syncthreads();
}

// C = A B for D x D matrices (row stride D) of true dimension d by the whole block (256 threads); C must not alias A
// or B; ends with a barrier.  Only the leading ceil(d / 16) * 16 rows, columns and k are read and written: d = 40 in
// its 64 x 64 frame takes 3 of 4 panels on 3 of 4 row blocks.
__device__ __forceinline__ int extent(int d) { return (d + 15) & ~15; }
template <int D, int BM = block_of<D>(), bool COMPACT = false>
__device__ __noinline__ void cta_mm(const double2 *A, const double2 *B, double2 *C, unsigned char *smem, int d) {
    const int n = D == 32 ? 32 : extent(d);
#pragma unroll 1
    for (int i = 0; i < n; i += BM)
#pragma unroll 1
        for (int j = 0; j < n; j += BM)
            block_mm<BM, COMPACT>(A + (size_t)i * D, D, B + j, D, C + (size_t)i * D + j, D, n, smem, min(BM, n - i), min(BM, n - j));
}

}  // namespace fxl
}  // namespace pm
