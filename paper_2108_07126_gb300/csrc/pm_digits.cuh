// FP64-grade complex matrix products of 8 x 8 and 16 x 16 matrices on the tensor cores, as exact sums
// of integer digits (the error-free splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication", 2012).
//
// Every matrix of the propagation is bounded: the scaled exponent X = -i G / 2^s has norm < 0.4, its
// Taylor polynomial norm < 1.5, slice propagators and their products are unitary.  So the entries
// are kept as 64-bit fixed-point numbers x = q 2^-56 (absolute rounding 2^-57, less than the rounding of a
// double near 1/4), and a product needs no scaling:
//   * q is split into seven balanced base-256 digits (the top one has 10 bits, |x| < 2), each an exact f16;
//   * digit products are summed by mma.sync m16n8k16 (f16 in, f32 accumulate), one accumulator per diagonal
//     i + j = t.  The sums are integers below 2^22 (worst case over 32 real terms), so every f32 accumulation is
//     exact; with the accumulator started at 1.5 2^23 the integer can be read from the bits of the float;
//   * the diagonal sums t = 0 .. 7 (34 digit pairs) are added in 64-bit integers.  The dropped ones (t >= 8) are below
//     2^-62; without t = 7 (28 pairs) a 16 x 16 product was off by 2^-56, a 128 x 128 one by 2^-54, more than on the FP64
//     pipe.
// The FP64 pipe of GB300 runs about two multiply-adds per clock and SM, mma.sync 1024: one 16 x 16 complex
// product takes 9.7 k SM cycles on the FP64 pipe and 272 MMAs (550 cycles) here.
//
// Register layout (one warp per matrix).  Lane 4 g + t holds, for D = 16, the pairs of entries
// (row g + 8 r, columns 8 h + 2 t, + 1), pair index 2 h + r, and for D = 8 the pair (row g, columns 2 t, + 1):
// the layout of the A operand and of the accumulator of m16n8k16 at once, so a product's output is the next
// product's left operand without any exchange.  The right operand B is needed as the same layout of B^T:
// X^T = -conj(X) and (X^2)^T = conj(X^2) (X is anti-Hermitian) only flip signs, the leaf product is kept
// transposed (R^T <- R^T U^T, whose right operand is U in its own layout), and squarings transpose the
// digits with movmatrix.
// D = 8 runs as one real 16 x 16 by 16 x 8 product, [[Ar, -Ai], [Ai, Ar]] [Br; Bi]: one MMA per digit pair.
#pragma once

#include <cstdint>

#include "pm_common.cuh"

namespace pm {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

constexpr int F = 56;     // fraction bits
constexpr int ND = 7;     // digits
constexpr int NA = 8;     // diagonals i + j of digit pairs that are summed (0 .. 7)
constexpr float kBias = 12582912.f;             // 1.5 * 2^23: floats in [2^23, 2^24) have integer spacing
constexpr u64 kSplitBias = 0x0200808080808080ull;  // makes every digit field non-negative

// round(m 2^-sh), 0 < sh < 60, ties to even.  Ties are common -- a double in [2^-5, 2^-4) is an odd multiple of half a unit
// every other time -- and rounding them away from zero scaled a whole matrix by 1 + 2^-54 at every conversion.
__device__ __forceinline__ u64 round_even(u64 m, int sh) { return (m + (1ull << (sh - 1)) - 1 + ((m >> sh) & 1)) >> sh; }
__device__ __forceinline__ i64 from_double(double v, int s) {  // round(v 2^(F - s)), |v| 2^-s < 2
    const i64 b = __double_as_longlong(v);
    const u64 m = ((u64)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = (int)((b >> 52) & 0x7ff) - 1075 + F - s;  // value = m 2^sh; zero and subnormals shift out
    u64 q;
    if (sh >= 0) q = m << min(sh, 10);
    else q = sh > -60 ? round_even(m, -sh) : 0ull;
    return b < 0 ? -(i64)q : (i64)q;
}
// q 2^-FR rounded to a double, in integer arithmetic (the conversion instruction runs on the FP64 pipe, 16 cycles a warp)
template <int FR = F> __device__ __forceinline__ double to_double(i64 q) {
    const u64 a = q < 0 ? (u64)-q : (u64)q;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const u64 m = a << lz;
    // 53 bits (the leading one adds to the exponent), ties to even
    const u64 mant = (m >> 11) + (((uint32_t)m & 0x7ffu) + ((uint32_t)(m >> 11) & 1u) > 0x400u ? 1 : 0);
    const u64 bits = ((u64)(1023 + 63 - FR - 1 - lz) << 52) + mant;
    return __longlong_as_double((long long)(bits | ((u64)q & 0x8000000000000000ull)));
}

// x * c rounded, c = ch 2^-32 + cl 2^-64 in [0, 1/4) (cl signed)
struct Coef {
    int32_t ch, cl;
    int32_t ns, sh;  // c = ns 2^(-sh - 24), ns in [2^30, 2^31)
};
__device__ __forceinline__ i64 mulc(i64 x, const Coef c) {
    const int32_t xh = (int32_t)(x >> 32);
    const uint32_t xl = (uint32_t)x;
    i64 t = (i64)((u64)xl * (uint32_t)c.ch) + 0x80000000ll;
    t += (i64)xh * c.cl;
    return (i64)xh * c.ch + (t >> 32);
}

// x * c to 31 bits of c and an absolute 2^-34 of x (|x| < 1/2): enough where the result is multiplied by
// X^6 or more afterwards
__device__ __forceinline__ i64 mulc_short(i64 x, const Coef c) {
    return ((i64)(int32_t)((x + (1ll << 23)) >> 24) * c.ns) >> c.sh;
}

// x / 2, ties to even: X^2 / 2 is on the diagonal of every slice propagator, and rounding its ties one way made
// the norm of U grow by 2^-58 a slice
__device__ __forceinline__ i64 halve(i64 x) { return (x + ((x >> 1) & 1)) >> 1; }

__device__ __forceinline__ uint32_t digit_pair(uint32_t w, uint32_t sub) {
    uint32_t d;
    asm("sub.f16x2 %0, %1, %2;" : "=r"(d) : "r"(w), "r"(sub));
    return d;
}

template <int D> struct L {
    static constexpr int NP = D == 16 ? 4 : 1;  // pairs per lane
    static constexpr int NE = 2 * NP;           // entries per lane
    __device__ static __forceinline__ int row(int lane, int e) { return (lane >> 2) + (D == 16 ? 8 * ((e >> 1) & 1) : 0); }
    __device__ static __forceinline__ int col(int lane, int e) {
        return 2 * (lane & 3) + (e & 1) + (D == 16 ? 8 * (e >> 2) : 0);
    }
};

template <int D> struct Tile {
    i64 re[L<D>::NE], im[L<D>::NE];
};
template <int D> struct Digits {
    uint32_t re[ND][L<D>::NP], im[ND][L<D>::NP];
};

// digits 0 (top) .. 6 of a pair of entries
__device__ __forceinline__ void split_pair(i64 a, i64 b, uint32_t (&d)[ND]) {
    const u64 x = (u64)a + kSplitBias, y = (u64)b + kSplitBias;
    const uint32_t xl = (uint32_t)x, xh = (uint32_t)(x >> 32), yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
    d[0] = digit_pair((__byte_perm(xh, yh, 0x7632) & 0x03FF03FFu) | 0x64006400u, 0x66006600u);
    d[1] = digit_pair((__byte_perm(xh, yh, 0x0501) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    d[2] = digit_pair((__byte_perm(xh, yh, 0x0400) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    d[3] = digit_pair((__byte_perm(xl, yl, 0x0703) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    d[4] = digit_pair((__byte_perm(xl, yl, 0x0602) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    d[5] = digit_pair((__byte_perm(xl, yl, 0x0501) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    d[6] = digit_pair((__byte_perm(xl, yl, 0x0400) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
}

template <int D> __device__ __forceinline__ void split(const Tile<D> &t, Digits<D> &d) {
#pragma unroll
    for (int p = 0; p < L<D>::NP; ++p) {
        uint32_t w[ND];
        split_pair(t.re[2 * p], t.re[2 * p + 1], w);
#pragma unroll
        for (int i = 0; i < ND; ++i) d.re[i][p] = w[i];
        split_pair(t.im[2 * p], t.im[2 * p + 1], w);
#pragma unroll
        for (int i = 0; i < ND; ++i) d.im[i][p] = w[i];
    }
}

__device__ __forceinline__ uint32_t neg2(uint32_t w) { return w ^ 0x80008000u; }
__device__ __forceinline__ uint32_t transpose8(uint32_t w) {
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(w));
    return r;
}

// The right operand of a product, as the digits of its transpose, in shared memory that is private to the
// lane: word (digit, part, pair) at ((digit * 2 + part) * NP + pair) * 32 + lane.
constexpr int kPlain = 0, kAntiHerm = 1, kHerm = 2, kTrans = 3;
template <int D> __host__ __device__ constexpr int rhs_words() { return ND * 2 * L<D>::NP * 32; }

// digits of M (own layout) -> right operand: kPlain: M^T as B; kAntiHerm: M^T = -conj(M); kHerm: M^T = conj(M);
// kTrans: transposed through movmatrix
template <int D> __device__ __forceinline__ void put_rhs(uint32_t *rhs, int lane, const Digits<D> &d, int mode) {
    constexpr int NP = L<D>::NP;
    const uint32_t fr = mode == kAntiHerm ? 0x80008000u : 0u, fi = mode == kHerm ? 0x80008000u : 0u;
#pragma unroll
    for (int i = 0; i < ND; ++i)
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            uint32_t a, b;
            if (mode == kTrans) {
                // pair 2 h + r is the 8 x 8 block (row block r, column block h); its transpose is the block (h, r)
                const int q = NP == 4 ? ((p & 1) << 1) | (p >> 1) : 0;
                a = transpose8(d.re[i][q]);
                b = transpose8(d.im[i][q]);
            } else {
                a = d.re[i][p] ^ fr;
                b = d.im[i][p] ^ fi;
            }
            rhs[((i * 2 + 0) * NP + p) * 32 + lane] = a;
            rhs[((i * 2 + 1) * NP + p) * 32 + lane] = b;
        }
}

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                    uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the first MMA of an accumulator: starts from s
__device__ __forceinline__ void mma_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1, float s) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(s));
}

__host__ __device__ constexpr float acc_start(int t) { return t < 6 ? kBias : 0.f; }
// last digit j paired with digit i
__host__ __device__ constexpr int last_digit(int i) { return NA - 1 - i < ND - 1 ? NA - 1 - i : ND - 1; }
// whether the pair (i, j) is the first on its diagonal in the loops over i, then j
__host__ __device__ constexpr bool first_pair(int i, int j) { return i == 0 || (j == ND - 1 && i + j < NA); }

__device__ __forceinline__ void acc_init(float (&acc)[NA][4]) {
#pragma unroll
    for (int t = 0; t < NA; ++t)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[t][u] = acc_start(t);
}

// sum_t v_t 2^(40 - 8 t) of the diagonal sums v_t; v_0 .. v_5 biased, v_6 and v_7 plain (rounded to 2^-56)
__device__ __forceinline__ i64 collect(const float (&acc)[NA][4], int u) {
    constexpr uint32_t B = 0x4B400000u, C = 257u * B;  // 256 B + B mod 2^32
    // v_5 + round((v_6 + v_7 / 256) / 256), biased
    const uint32_t w5 = __float_as_uint(fmaf(fmaf(acc[7][u], 0.00390625f, acc[6][u]), 0.00390625f, acc[5][u]));
    const int32_t lo = (int32_t)(__float_as_uint(acc[4][u]) * 256u + w5 - C);
    const int32_t mid = (int32_t)(__float_as_uint(acc[2][u]) * 256u + __float_as_uint(acc[3][u]) - C);
    const uint32_t hi = __float_as_uint(acc[0][u]) * 256u + __float_as_uint(acc[1][u]) - C;
    return (i64)mid * 65536 + (i64)lo + (i64)((u64)hi << 32);
}

// the same sum rounded to 2^-60: for outputs that are collected panel by panel
constexpr int FC = 60;
__device__ __forceinline__ i64 collect_fine(const float (&acc)[NA][4], int u) {
    constexpr uint32_t B = 0x4B400000u, C = 257u * B;
    const uint32_t b6 = __float_as_uint(fmaf(acc[7][u], 0.00390625f, acc[6][u]) + kBias);
    const int32_t l = (int32_t)(__float_as_uint(acc[5][u]) * 256u + b6 - C);
    const int32_t m = (int32_t)(__float_as_uint(acc[3][u]) * 256u + __float_as_uint(acc[4][u]) - C);
    const int32_t h = (int32_t)(__float_as_uint(acc[1][u]) * 256u + __float_as_uint(acc[2][u]) - C);
    const uint32_t t = __float_as_uint(acc[0][u]) - B;
    // ties to even: rounding half up leaves a mean of 2^-65 in every entry, which as a matrix of constants has norm
    // d 2^-65 and the same sign in every slice (d = 40, N = 4000: error 1.5e-13 instead of 4e-14)
    return (i64)((l + 7 + ((l >> 4) & 1)) >> 4) + (i64)m * 4096 + (i64)h * (1 << 28) + (i64)((u64)t << 44);
}

// one quarter of a 16 x 16 product: n-tile nt (columns 8 nt ..), part 0 = Re, 1 = Im -> o[2 r + c]
__device__ __forceinline__ void mul16_quarter(const Digits<16> &a, const uint32_t *rhs, int lane, int nt, int part,
                                              i64 (&o)[4]) {
    float acc[NA][4];
    // Re: Ar Br + Ai (-Bi); Im: Ar Bi + Ai Br
    const uint32_t f2 = part ? 0u : 0x80008000u;
    {
        uint32_t b[ND][2];
#pragma unroll
        for (int j = 0; j < ND; ++j) {
            b[j][0] = rhs[((j * 2 + part) * 4 + nt) * 32 + lane];
            b[j][1] = rhs[((j * 2 + part) * 4 + 2 + nt) * 32 + lane];
        }
#pragma unroll
        for (int i = 0; i < ND; ++i)
#pragma unroll
            for (int j = 0; j <= last_digit(i); ++j) {
                if (first_pair(i, j)) mma_first(acc[i + j], a.re[i][0], a.re[i][1], a.re[i][2], a.re[i][3], b[j][0], b[j][1], acc_start(i + j));
                else mma(acc[i + j], a.re[i][0], a.re[i][1], a.re[i][2], a.re[i][3], b[j][0], b[j][1]);
            }
    }
    {
        uint32_t b[ND][2];
#pragma unroll
        for (int j = 0; j < ND; ++j) {
            b[j][0] = rhs[((j * 2 + 1 - part) * 4 + nt) * 32 + lane] ^ f2;
            b[j][1] = rhs[((j * 2 + 1 - part) * 4 + 2 + nt) * 32 + lane] ^ f2;
        }
#pragma unroll
        for (int i = 0; i < ND; ++i)
#pragma unroll
            for (int j = 0; j <= last_digit(i); ++j)
                mma(acc[i + j], a.im[i][0], a.im[i][1], a.im[i][2], a.im[i][3], b[j][0], b[j][1]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) o[u] = collect(acc, u);
}

__device__ __forceinline__ void mul(const Digits<16> &a, const uint32_t *rhs, int lane, Tile<16> &o) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        i64 v[4];
        mul16_quarter(a, rhs, lane, nt, 0, v);
#pragma unroll
        for (int u = 0; u < 4; ++u) o.re[4 * nt + u] = v[u];
        mul16_quarter(a, rhs, lane, nt, 1, v);
#pragma unroll
        for (int u = 0; u < 4; ++u) o.im[4 * nt + u] = v[u];
    }
}
__device__ __forceinline__ void mul(const Digits<8> &a, const uint32_t *rhs, int lane, Tile<8> &o) {
    float acc[NA][4];
    uint32_t b[ND][2];
#pragma unroll
    for (int j = 0; j < ND; ++j) {
        b[j][0] = rhs[(j * 2 + 0) * 32 + lane];
        b[j][1] = rhs[(j * 2 + 1) * 32 + lane];
    }
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        const uint32_t n = neg2(a.im[i][0]);
#pragma unroll
        for (int j = 0; j <= last_digit(i); ++j) {
            if (first_pair(i, j)) mma_first(acc[i + j], a.re[i][0], a.im[i][0], n, a.re[i][0], b[j][0], b[j][1], acc_start(i + j));
            else mma(acc[i + j], a.re[i][0], a.im[i][0], n, a.re[i][0], b[j][0], b[j][1]);
        }
    }
    o.re[0] = collect(acc, 0);
    o.re[1] = collect(acc, 1);
    o.im[0] = collect(acc, 2);
    o.im[1] = collect(acc, 3);
}

// o = a1 B1 + a2 B2
__device__ __forceinline__ void mul_sum(const Digits<16> &a1, const uint32_t *rhs1, const Digits<16> &a2, const uint32_t *rhs2,
                                        int lane, Tile<16> &o) {
    mul(a1, rhs1, lane, o);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            i64 v[4];
            mul16_quarter(a2, rhs2, lane, nt, part, v);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (part) o.im[4 * nt + u] += v[u];
                else o.re[4 * nt + u] += v[u];
            }
        }
}
// (D = 8: both products in one set of accumulators, 32 real terms as in one 16 x 16 product)
__device__ __forceinline__ void mul_sum(const Digits<8> &a1, const uint32_t *rhs1, const Digits<8> &a2, const uint32_t *rhs2,
                                        int lane, Tile<8> &o) {
    float acc[NA][4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const Digits<8> &a = k ? a2 : a1;
        const uint32_t *rhs = k ? rhs2 : rhs1;
        uint32_t b[ND][2];
#pragma unroll
        for (int j = 0; j < ND; ++j) {
            b[j][0] = rhs[(j * 2 + 0) * 32 + lane];
            b[j][1] = rhs[(j * 2 + 1) * 32 + lane];
        }
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const uint32_t n = neg2(a.im[i][0]);
#pragma unroll
            for (int j = 0; j <= last_digit(i); ++j) {
                if (k == 0 && first_pair(i, j)) mma_first(acc[i + j], a.re[i][0], a.im[i][0], n, a.re[i][0], b[j][0], b[j][1], acc_start(i + j));
                else mma(acc[i + j], a.re[i][0], a.im[i][0], n, a.re[i][0], b[j][0], b[j][1]);
            }
        }
    }
    o.re[0] = collect(acc, 0);
    o.re[1] = collect(acc, 1);
    o.im[0] = collect(acc, 2);
    o.im[1] = collect(acc, 3);
}

// tile <-> shared memory private to the lane: entry e at e * 32 + lane (16 bytes)
template <int D> __device__ __forceinline__ void st_priv(longlong2 *S, int lane, const Tile<D> &t) {
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e) S[e * 32 + lane] = make_longlong2(t.re[e], t.im[e]);
}
template <int D> __device__ __forceinline__ void ld_priv(const longlong2 *S, int lane, Tile<D> &t) {
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e) {
        const longlong2 v = S[e * 32 + lane];
        t.re[e] = v.x;
        t.im[e] = v.y;
    }
}

}  // namespace fx
}  // namespace pm
