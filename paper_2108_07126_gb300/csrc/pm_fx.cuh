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

#include "pm_fused.cuh"

namespace pm {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

constexpr int F = 56;     // fraction bits
constexpr int ND = 7;     // digits
constexpr int NA = 8;     // diagonals i + j of digit pairs that are summed (0 .. 7)
constexpr float kBias = 12582912.f;             // 1.5 * 2^23: floats in [2^23, 2^24) have integer spacing
constexpr u64 kSplitBias = 0x0200808080808080ull;  // makes every digit field non-negative

__device__ __forceinline__ i64 from_double(double v, int s) {  // round(v 2^(F - s)), |v| 2^-s < 2
    const i64 b = __double_as_longlong(v);
    const u64 m = ((u64)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = (int)((b >> 52) & 0x7ff) - 1075 + F - s;  // value = m 2^sh; zero and subnormals shift out
    u64 q;
    if (sh >= 0) q = m << min(sh, 10);
    else q = sh > -60 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
    return b < 0 ? -(i64)q : (i64)q;
}
// q 2^-FR rounded to a double, in integer arithmetic (the conversion instruction runs on the FP64 pipe, 16 cycles a warp)
template <int FR = F> __device__ __forceinline__ double to_double(i64 q) {
    const u64 a = q < 0 ? (u64)-q : (u64)q;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const u64 m = a << lz;
    const u64 mant = (m >> 11) + ((m >> 10) & 1);  // 53 bits, the leading one adds to the exponent
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
    return (i64)((l + 8) >> 4) + (i64)m * 4096 + (i64)h * (1 << 28) + (i64)((u64)t << 44);
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

// ---------------------------------------------------------------- the propagation kernel

constexpr int kGT = 16;  // slices whose coefficients are prepared together

template <int D> struct Cfg {
    static constexpr int MAXW = D == 16 ? 8 : 16;             // warps per block (D = 16: 255 registers)
    static constexpr int TILE = L<D>::NE * 32 * 16;             // bytes of a lane-private tile
    static constexpr int RHS = rhs_words<D>() * 4;              // bytes of a right operand
    static constexpr size_t LEAF_BYTES = (size_t)kGT * D * D * 8;  // packed exponents of a tile in global memory
    static constexpr int PS = D + 1;                            // row stride of the packed exponent (8 bytes)
    static_assert(D * PS * 8 <= RHS, "the packed exponent fits in the right operand's space");
};
template <int D> __host__ __device__ inline size_t warp_bytes(int nb) {
    // X, X^2, R^T, right operand (its space holds the coefficient tile and the packed exponent before), class tile
    const size_t gam = (size_t)nb * kGT * 8;
    return (size_t)3 * Cfg<D>::TILE + (gam > Cfg<D>::RHS ? gam : Cfg<D>::RHS) + 64;
}
template <int D> __host__ __device__ inline size_t smem_bytes(int nb, int warps) {
    return (size_t)warps * warp_bytes<D>(nb) + (((size_t)nb * 8 + 15) & ~(size_t)15);
}

// 1 / k! as multipliers and as fixed-point constants
constexpr u64 fact(int k) { return k <= 1 ? 1ull : (u64)k * fact(k - 1); }
constexpr Coef inv_fact(int k) {
    const u64 n = fact(k < 3 ? 3 : k);  // 2^64 / n = ch 2^32 + cl, |cl| <= 2^31
    const u64 c = 0ull - n;             // 2^64 - n
    const u64 v = c / n + 1;            // floor(2^64 / n)
    const u64 h = (v + 0x80000000ull) >> 32;
    int up = 0;
    while ((v << up) < (1ull << 62)) ++up;  // v 2^up in [2^62, 2^63)
    return Coef{(int32_t)h, (int32_t)(i64)(v - (h << 32)), (int32_t)(((v << up) + (1ull << 31)) >> 32), 32 + up - 24};
}
constexpr i64 inv_fact_fx(int k) { return (i64)(((1ull << F) + fact(k) / 2) / fact(k)); }
static __constant__ Coef c_inv[kMaxDegree + 1] = {inv_fact(0), inv_fact(1), inv_fact(2), inv_fact(3), inv_fact(4),
                                                   inv_fact(5), inv_fact(6), inv_fact(7), inv_fact(8), inv_fact(9),
                                                   inv_fact(10), inv_fact(11), inv_fact(12)};
static __constant__ i64 c_inv_fx[kMaxDegree + 1] = {
    inv_fact_fx(0), inv_fact_fx(1), inv_fact_fx(2), inv_fact_fx(3), inv_fact_fx(4),  inv_fact_fx(5),  inv_fact_fx(6),
    inv_fact_fx(7), inv_fact_fx(8), inv_fact_fx(9), inv_fact_fx(10), inv_fact_fx(11), inv_fact_fx(12)};

// digits of a basis matrix entry: B 2^-E with 2^E > ||B||_1
__host__ __device__ constexpr int ksteps(int nb) { return nb > 0 ? (nb + 15) / 16 : 1; }
template <int D> __host__ __device__ constexpr size_t basis_digit_bytes(int nb) {
    return (size_t)ksteps(nb) * (D * D / 8) * ND * 32 * sizeof(uint2);
}
__device__ __forceinline__ int basis_exp(double norm) { return norm > 0.0 ? ilogb(norm) + 1 : 0; }

// The packed basis as the right operand of the assembly's MMAs: word pair (kstep, entry tile, digit, lane)
// holds the digits of matrices 16 ks + 2 t, + 1 and + 8, + 9 at entry 8 nt + g.
template <int D>
__global__ void __launch_bounds__(32) basis_digits_kernel(const double *packed, const double *bnorm, int nb, uint2 *out) {
    constexpr int DD = D * D, NT = DD / 8;
    const int lane = threadIdx.x, nt = blockIdx.x, ks = blockIdx.y, n = 8 * nt + (lane >> 2);
    uint32_t w[2][ND];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        i64 v[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int e = 16 * ks + 8 * h + 2 * (lane & 3) + c;
            v[c] = e < nb ? from_double(packed[(size_t)e * DD + n], basis_exp(bnorm[e])) : 0;
        }
        split_pair(v[0], v[1], w[h]);
    }
#pragma unroll
    for (int i = 0; i < ND; ++i) out[(((size_t)ks * NT + nt) * ND + i) * 32 + lane] = make_uint2(w[0][i], w[1][i]);
}

// The packed exponents of a tile of up to 16 slices, scaled by 2^-s, into g [16][D D]: one GEMM
// [slices x basis matrices] [basis matrices x entries] on the digit products (the coefficients are scaled by
// 2^(E - s), so |gamma| <= norm bound / 2^s).  On the FP64 pipe the same sum costs 2.4 k SM cycles per slice
// for 16 basis matrices at D = 16, here 56 MMAs (112 cycles).  Sums over more than 32 matrices are collected
// every 32 (the exactness bound).
template <int D>
__device__ __forceinline__ void assemble_tile(const uint2 *bd, int nb, const double *gam, int s0, int s1,
                                              const double *bnorm, int lane, i64 *g) {
    constexpr int DD = D * D, NT = DD / 8;
    const int gr = lane >> 2, t4 = lane & 3;  // the lane's rows: slices gr and gr + 8, squarings s0 and s1
    for (int k0 = 0; k0 < 16 * ksteps(nb); k0 += 32) {
        uint32_t a[2][4][ND];
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                i64 v[2][2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int e = k0 + 16 * ks + 8 * h + 2 * t4 + c;
                    const int E = e < nb ? basis_exp(bnorm[e]) : 0;
                    v[0][c] = e < nb ? from_double(gam[e * kGT + gr], s0 - E) : 0;
                    v[1][c] = e < nb ? from_double(gam[e * kGT + gr + 8], s1 - E) : 0;
                }
                split_pair(v[0][0], v[0][1], a[ks][2 * h]);
                split_pair(v[1][0], v[1][1], a[ks][2 * h + 1]);
            }
        const int nks = min(2, ksteps(nb) - k0 / 16);
        const uint2 *bk = bd + (size_t)(k0 / 16) * NT * ND * 32 + lane;
        uint2 b[ND];  // the digits of the next step's entries, loaded one step ahead
#pragma unroll
        for (int j = 0; j < ND; ++j) b[j] = __ldg(bk + j * 32);
#pragma unroll 1
        for (int nt = 0; nt < NT; ++nt) {
            float acc[NA][4];
            uint2 c[ND];
            const int last = (nt + 1 < NT ? nt + 1 : nt) * ND * 32;
#pragma unroll
            for (int j = 0; j < ND; ++j) c[j] = __ldg(bk + (nks == 2 ? ((size_t)NT + nt) * ND * 32 : last) + j * 32);
#pragma unroll
            for (int i = 0; i < ND; ++i)
#pragma unroll
                for (int j = 0; j <= last_digit(i); ++j) {
                    if (first_pair(i, j)) mma_first(acc[i + j], a[0][0][i], a[0][1][i], a[0][2][i], a[0][3][i], b[j].x, b[j].y, acc_start(i + j));
                    else mma(acc[i + j], a[0][0][i], a[0][1][i], a[0][2][i], a[0][3][i], b[j].x, b[j].y);
                }
#pragma unroll
            for (int j = 0; j < ND; ++j) b[j] = c[j];
            if (nks == 2) {
#pragma unroll
                for (int j = 0; j < ND; ++j) b[j] = __ldg(bk + last + j * 32);
#pragma unroll
                for (int i = 0; i < ND; ++i)
#pragma unroll
                    for (int j = 0; j <= last_digit(i); ++j)
                        mma(acc[i + j], a[1][0][i], a[1][1][i], a[1][2][i], a[1][3][i], c[j].x, c[j].y);
            }
            i64 o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) o[u] = collect(acc, u);
            longlong2 *d0 = reinterpret_cast<longlong2 *>(g + gr * DD + 8 * nt + 2 * t4);
            longlong2 *d1 = reinterpret_cast<longlong2 *>(g + (gr + 8) * DD + 8 * nt + 2 * t4);
            if (k0 > 0) {
                const longlong2 x = *d0, y = *d1;
                o[0] += x.x;
                o[1] += x.y;
                o[2] += y.x;
                o[3] += y.y;
            }
            *d0 = make_longlong2(o[0], o[1]);
            *d1 = make_longlong2(o[2], o[3]);
        }
    }
}

// One propagation (TRAJ: the output pass of a trajectory), one warp per leaf: the steps of fused_body
// (pm_fused.cuh) with the matrices in fixed point.  The partial products between blocks stay in fixed
// point in p.partials; leaf_out and block_out get doubles.  A slice whose norm bound is not finite or
// above the table poisons the results with NaN (fixed point has none).
template <int D, int INTEG, bool TRAJ>
__global__ void __launch_bounds__(Cfg<D>::MAXW * 32, 1) fx_kernel(const FusedParams p) {
    constexpr int NE = L<D>::NE, DD = D * D, PS = Cfg<D>::PS, EPL = DD / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_second;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int nb = p.n_basis, blk = blockIdx.x, nblk = gridDim.x;
    const size_t wb = warp_bytes<D>(nb);
    unsigned char *wbase = smem + (size_t)warp * wb;
    const int64_t n_leaves = (int64_t)nblk * W, leaf = (int64_t)blk * W + warp;
    i64 *gbuf = (i64 *)((unsigned char *)p.fx_g + (size_t)leaf * Cfg<D>::LEAF_BYTES);
    longlong2 *SX = (longlong2 *)wbase, *SX2 = SX + NE * 32;
    longlong2 *SRT = SX2 + NE * 32;
    uint32_t *rhs = (uint32_t *)(SRT + NE * 32);
    i64 *xpk = (i64 *)rhs;  // packed exponent, dead before the right operand is written
    double *gam = (double *)rhs;  // coefficients of a tile, dead once its exponents are assembled
    int *cls = (int *)(wbase + wb - 64);
    double *bnorm = (double *)(smem + (size_t)W * wb);
    for (int i = tid; i < nb; i += blockDim.x) bnorm[i] = p.bnorm1[i];

    const int64_t j0 = p.n_steps * leaf / n_leaves;
    const int len = (int)(p.n_steps * (leaf + 1) / n_leaves - j0);

    Tile<D> T;
#pragma unroll
    for (int e = 0; e < NE; ++e) {  // R^T = I, or the prefix of the leaf
        const int j = L<D>::row(lane, e), i = L<D>::col(lane, e);
        if constexpr (TRAJ) {
            const double2 v = p.traj_pin[(size_t)leaf * DD + i * D + j];
            T.re[e] = from_double(v.x, 0);
            T.im[e] = from_double(v.y, 0);
        } else {
            T.re[e] = i == j ? (i64)1 << F : 0;
            T.im[e] = 0;
        }
    }
    st_priv<D>(SRT, lane, T);
    __syncthreads();

    unsigned flags = 0;
    unsigned long long n_exp = 0;
    int m_max = 0, s_max = 0;

    for (int t0 = 0; t0 < len; t0 += kGT) {
        __syncwarp();
        if (lane < kGT) {
            const bool act = t0 + lane < len;
            double *gcol = gam + lane;
            slice_coefficients<double, INTEG, kGT>(p, j0 + t0 + lane, act, gcol);
            double nu = 0.0;
            for (int e = 0; e < nb; ++e) nu = fma(fabs(gcol[e * kGT]), bnorm[e], nu);
            cls[lane] = find_class(p, nu, &flags);
        }
        __syncwarp();
        const int nr = min(kGT, len - t0);
        assemble_tile<D>((const uint2 *)p.fx_basis, nb, gam, cls_s(p.cls_code[cls[lane >> 2]]) + p.extra_squarings,
                         cls_s(p.cls_code[cls[(lane >> 2) + 8]]) + p.extra_squarings, bnorm, lane, gbuf);
        __syncwarp();
        longlong2 gq[EPL / 2];  // the next slice's packed exponent
        auto fetch = [&](int rr) {
            const longlong2 *src = reinterpret_cast<const longlong2 *>(gbuf + (size_t)rr * DD) + lane;
#pragma unroll
            for (int t = 0; t < EPL / 2; ++t) gq[t] = src[32 * t];
        };
        fetch(0);
        for (int rr = 0; rr < nr; ++rr) {
            const int code = p.cls_code[cls[rr]];
            const int q = cls_q(code), rh = cls_r(code), s = cls_s(code) + p.extra_squarings;

            // packed exponent, two consecutive entries per lane and step
#pragma unroll
            for (int t = 0; t < EPL / 2; ++t) {
                const int pos = 2 * (lane + 32 * t);
                i64 *dst = xpk + (pos / D) * PS + (pos % D);
                dst[0] = gq[t].x;
                dst[1] = gq[t].y;
            }
            if (rr + 1 < nr) fetch(rr + 1);
            __syncwarp();
            // X = -i G / 2^s: Re X = Im G, Im X = -Re G (upper triangle: Re G, strict lower: Im G)
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                const int i = L<D>::row(lane, e), j = L<D>::col(lane, e);
                const i64 a = xpk[i * PS + j], b = xpk[j * PS + i];
                T.re[e] = i > j ? a : (i < j ? -b : 0);
                T.im[e] = -(i <= j ? a : b);
            }
            __syncwarp();
            st_priv<D>(SX, lane, T);

            // T += B_b = a_{q b} I + a_{q b + 1} X + a_{q b + 2} X^2 (as many terms as q), a_k = 1 / k!
            auto add_block = [&](int b) {
                const i64 a0 = c_inv_fx[q * b];
#pragma unroll
                for (int e = 0; e < NE; ++e)
                    if (L<D>::row(lane, e) == L<D>::col(lane, e)) T.re[e] += a0;
                if (q < 2) return;
                if (b == 0) {
#pragma unroll
                    for (int e = 0; e < NE; ++e) {
                        const longlong2 x = SX[e * 32 + lane];
                        T.re[e] += x.x;
                        T.im[e] += x.y;
                    }
                    if (q >= 3) {
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            const longlong2 x = SX2[e * 32 + lane];
                            T.re[e] += halve(x.x);
                            T.im[e] += halve(x.y);
                        }
                    }
                } else if (q * b >= 6) {  // X^6 or more follows: short multiplications
                    const Coef c1 = c_inv[q * b + 1], c2 = c_inv[q * b + 2];
#pragma unroll
                    for (int e = 0; e < NE; ++e) {
                        const longlong2 x = SX[e * 32 + lane], y = SX2[e * 32 + lane];
                        T.re[e] += mulc_short(x.x, c1) + mulc_short(y.x, c2);
                        T.im[e] += mulc_short(x.y, c1) + mulc_short(y.y, c2);
                    }
                } else {  // q b >= 2: every coefficient is at most 1 / 3!
                    const Coef c1 = c_inv[q * b + 1], c2 = c_inv[q * b + 2];
#pragma unroll
                    for (int e = 0; e < NE; ++e) {
                        const longlong2 x = SX[e * 32 + lane];
                        T.re[e] += mulc(x.x, c1);
                        T.im[e] += mulc(x.y, c1);
                    }
                    if (q >= 3) {
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            const longlong2 x = SX2[e * 32 + lane];
                            T.re[e] += mulc(x.x, c2);
                            T.im[e] += mulc(x.y, c2);
                        }
                    }
                }
            };
            auto start_horner = [&]() {  // T = X^q: a_{q rh} X^q + B_{rh - 1}
                if (q * rh == 2) {
#pragma unroll
                    for (int e = 0; e < NE; ++e) {
                        T.re[e] = halve(T.re[e]);
                        T.im[e] = halve(T.im[e]);
                    }
                } else if (q * rh > 2) {
                    const Coef c = c_inv[q * rh];
                    if (q * rh >= 9) {
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            T.re[e] = mulc_short(T.re[e], c);
                            T.im[e] = mulc_short(T.im[e], c);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            T.re[e] = mulc(T.re[e], c);
                            T.im[e] = mulc(T.im[e], c);
                        }
                    }
                }
                add_block(rh - 1);
            };
            // the products of the slice through one call site: powers, [X^q as the right operand], Horner
            // steps T <- T X^q (polynomials of X commute), squarings, [U as the right operand], R^T <- R^T U^T
            const int n_pow = q - 1, n_hor = rh - 1;
            const int e0 = n_pow, e1 = e0 + (n_hor > 0), e2 = e1 + n_hor, e3 = e2 + s, e4 = e3 + 1;
            int bl = rh - 1;
            if (n_pow == 0) start_horner();
            for (int op = 0; op <= e4; ++op) {
                Digits<D> d;
                split<D>(T, d);
                if (op < e0) {
                    if (op == 0) put_rhs<D>(rhs, lane, d, kAntiHerm);
                } else if (op < e1) {
                    put_rhs<D>(rhs, lane, d, q == 2 ? kHerm : kAntiHerm);
                    start_horner();
                    continue;
                } else if (op >= e2 && op < e3) {
                    put_rhs<D>(rhs, lane, d, kTrans);
                } else if (op == e3) {
                    put_rhs<D>(rhs, lane, d, kPlain);
                    ld_priv<D>(SRT, lane, T);
                    continue;
                }
                mul(d, rhs, lane, T);
                if (op < e0) {
                    if (op == 0 && q == 3) st_priv<D>(SX2, lane, T);
                    if (op == e0 - 1 && n_hor == 0) start_horner();
                } else if (op < e2) {
                    add_block(--bl);
                }
            }
            st_priv<D>(SRT, lane, T);

            if constexpr (TRAJ) {
                const int64_t j = j0 + t0 + rr;
                if ((j + 1) % p.traj_every == 0 || j + 1 == p.n_steps) {
                    const int64_t o = j / p.traj_every;
                    const int d = p.d_out;
                    const double bad = __any_sync(0xffffffffu, flags) ? nan("") : 0.0;
                    if (p.traj_psi0 == nullptr) {
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            const int jj = L<D>::row(lane, e), i = L<D>::col(lane, e);
                            if (i < d && jj < d) {
                                const size_t at = ((size_t)o * d + i) * d + jj;
                                const double re = to_double(T.re[e]) + bad, im = to_double(T.im[e]) + bad;
                                if (p.out_c128) ((double2 *)p.traj_out)[at] = make_double2(re, im);
                                else ((float2 *)p.traj_out)[at] = make_float2((float)re, (float)im);
                            }
                        }
                    } else {  // psi(t_n) = R psi_0: the lane's rows of R^T, then the eight lanes of a column
#pragma unroll
                        for (int h = 0; h < NE / (D == 16 ? 4 : 2); ++h)
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                double re = bad, im = bad;
#pragma unroll
                                for (int r = 0; r < (D == 16 ? 2 : 1); ++r) {
                                    const int e = D == 16 ? (2 * h + r) * 2 + c : c;
                                    const double2 b = p.traj_psi0[L<D>::row(lane, e)];
                                    const double ax = to_double(T.re[e]), ay = to_double(T.im[e]);
                                    re = fma(ax, b.x, fma(-ay, b.y, re));
                                    im = fma(ax, b.y, fma(ay, b.x, im));
                                }
#pragma unroll
                                for (int off = 4; off < 32; off <<= 1) {
                                    re += __shfl_xor_sync(0xffffffffu, re, off);
                                    im += __shfl_xor_sync(0xffffffffu, im, off);
                                }
                                const int i = 8 * h + 2 * (lane & 3) + c;
                                if (lane < 4 && i < d) {
                                    const size_t at = (size_t)o * d + i;
                                    if (p.out_c128) ((double2 *)p.traj_out)[at] = make_double2(re, im);
                                    else ((float2 *)p.traj_out)[at] = make_float2((float)re, (float)im);
                                }
                            }
                    }
                }
            }
            n_exp += (unsigned long long)((q - 1) + (rh - 1) + s);
            m_max = max(m_max, cls_m(code));
            s_max = max(s_max, s);
        }
    }
    flags = __reduce_or_sync(0xffffffffu, flags);
    if constexpr (TRAJ) return;  // the forward pass combined the leaves and recorded the statistics

    if (p.leaf_out) {
        ld_priv<D>(SRT, lane, T);
        const double bad = flags ? nan("") : 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e)
            p.leaf_out[(size_t)leaf * DD + L<D>::col(lane, e) * D + L<D>::row(lane, e)] =
                make_double2(to_double(T.re[e]) + bad, to_double(T.im[e]) + bad);
    }
    if (lane == 0 && len > 0) {
        atomicAdd(&p.counters[0], n_exp);
        atomicAdd(&p.counters[1], (unsigned long long)len);
        atomicMax(&p.counters[2], (unsigned long long)m_max);
        atomicMax(&p.counters[3], (unsigned long long)s_max);
    }
    if (lane == 0 && flags) atomicOr(&p.status[0], flags);

    // ---- pairwise tree over the leaves of the block: (R_late R_early)^T = R_early^T R_late^T
    const int any_bad = __syncthreads_or((int)flags);
    auto tile_of = [&](int w) { return (longlong2 *)(smem + (size_t)w * wb) + 2 * NE * 32; };
    for (int h = 1; h < W; h <<= 1) {
        const int left = warp * 2 * h;
        if (left + h < W) {
            Digits<D> d;
            ld_priv<D>(tile_of(left + h), lane, T);
            split<D>(T, d);
            put_rhs<D>(rhs, lane, d, kTrans);
            ld_priv<D>(tile_of(left), lane, T);
            split<D>(T, d);
            mul(d, rhs, lane, T);
        }
        __syncthreads();
        if (left + h < W) st_priv<D>(tile_of(left), lane, T);
        __syncthreads();
    }
    if (warp == 0) {
        ld_priv<D>(SRT, lane, T);
        longlong2 *dst = (longlong2 *)p.partials + (size_t)blk * DD;
        const double bad = any_bad ? nan("") : 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int at = L<D>::col(lane, e) * D + L<D>::row(lane, e);
            __stcg((longlong2 *)dst + at, make_longlong2(T.re[e], T.im[e]));
            if (p.block_out)
                p.block_out[(size_t)blk * DD + at] = make_double2(to_double(T.re[e]) + bad, to_double(T.im[e]) + bad);
        }
    }
    __threadfence();
    __syncthreads();

    // ---- pairwise tree over the blocks: the second arrival at a node multiplies, the first leaves
    int idx = blk, n = nblk, level = 0, toff = 0;
    while (n > 1) {
        const int parent = idx >> 1;
        if ((idx | 1) < n) {
            if (tid == 0) s_second = (atomicAdd(&p.tickets[toff + parent], 1u) != 0u);
            __syncthreads();
            if (!s_second) return;
            if (tid == 0) p.tickets[toff + parent] = 0u;  // ready for the next launch
            __threadfence();
            longlong2 *gL = (longlong2 *)p.partials + (size_t)((idx & ~1) << level) * DD;
            const longlong2 *gR = (const longlong2 *)p.partials + (size_t)((idx | 1) << level) * DD;
            // D = 16: four quarters of the product over the warps; each reads both factors first
            constexpr int NQ = D == 16 ? 4 : 1;
            i64 o[NE > 4 ? 4 : 1][4];
            int n_own = 0;
            for (int qt = warp; qt < NQ; qt += W, ++n_own) {
                Digits<D> d;
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    const longlong2 v = __ldcg(gL + L<D>::col(lane, e) * D + L<D>::row(lane, e));
                    T.re[e] = v.x;
                    T.im[e] = v.y;
                }
                split<D>(T, d);
                put_rhs<D>(rhs, lane, d, kPlain);
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    const longlong2 v = __ldcg(gR + L<D>::row(lane, e) * D + L<D>::col(lane, e));
                    T.re[e] = v.x;
                    T.im[e] = v.y;
                }
                split<D>(T, d);
                if constexpr (D == 16) {
                    i64 v[4];
                    mul16_quarter(d, rhs, lane, qt >> 1, qt & 1, v);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k == n_own) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) o[k][u] = v[u];
                        }
                } else {
                    mul(d, rhs, lane, T);
                }
            }
            __syncthreads();  // every factor is read before the left one is overwritten
            n_own = 0;
            for (int qt = warp; qt < NQ; qt += W, ++n_own) {
                if constexpr (D == 16) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k == n_own) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int i = (lane >> 2) + 8 * (u >> 1), j = 8 * (qt >> 1) + 2 * (lane & 3) + (u & 1);
                                __stcg((i64 *)(gL + i * D + j) + (qt & 1), o[k][u]);
                            }
                        }
                } else {
#pragma unroll
                    for (int e = 0; e < NE; ++e)
                        __stcg(gL + L<D>::row(lane, e) * D + L<D>::col(lane, e), make_longlong2(T.re[e], T.im[e]));
                }
            }
            __threadfence();
            __syncthreads();
        }
        idx = parent;
        n = (n + 1) >> 1;
        toff += n;
        ++level;
    }

    // ---- root: U(T), statistics snapshot
    if (tid == 0) {
        __threadfence();
        for (int i = 0; i < 4; ++i) p.counters[4 + i] = atomicExch(&p.counters[i], 0ull);
        const unsigned st = atomicExch(&p.status[0], 0u);
        p.status[1] = st;
        s_second = (int)st;
    }
    __syncthreads();
    const double bad = s_second ? nan("") : 0.0;
    const int d = p.d_out;
    for (int t = tid; t < d * d; t += blockDim.x) {
        const longlong2 v = __ldcg((const longlong2 *)p.partials + (t / d) * D + (t % d));
        const double re = to_double(v.x) + bad, im = to_double(v.y) + bad;
        if (p.out_c128) ((double2 *)p.U_out)[t] = make_double2(re, im);
        else ((float2 *)p.U_out)[t] = make_float2((float)re, (float)im);
    }
}

template <int D, int INTEG, bool TRAJ>
cudaError_t launch(const FusedParams &p, int grid, int warps, size_t smem, cudaStream_t st) {
    auto k = fx_kernel<D, INTEG, TRAJ>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, warps * 32, smem, st>>>(p);
    return cudaGetLastError();
}
template <int D>
cudaError_t basis_digits(const double *packed, const double *bnorm, int nb, void *out, cudaStream_t st) {
    basis_digits_kernel<D><<<dim3(D * D / 8, ksteps(nb)), 32, 0, st>>>(packed, bnorm, nb, (uint2 *)out);
    return cudaGetLastError();
}
template <int D, int INTEG, bool TRAJ> int max_blocks_per_sm(int warps, size_t smem) {
    int nb = 0;
    auto k = fx_kernel<D, INTEG, TRAJ>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, warps * 32, smem) != cudaSuccess) return 0;
    return nb;
}

}  // namespace fx
}  // namespace pm
