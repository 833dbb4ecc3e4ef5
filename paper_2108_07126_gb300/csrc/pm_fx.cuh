// The fused propagation kernel for D = 8 and 16 in FP64 on the digit products of pm_digits.cuh: one warp per leaf,
// matrices in fixed point, the steps of fused_body (pm_fused.cuh).
#pragma once

#include "pm_digits.cuh"
#include "pm_fused.cuh"

namespace pm {
namespace fx {

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
    unsigned bad_prefix = 0;  // a prefix with a NaN (fixed point has none): every output of the leaf is NaN
#pragma unroll
    for (int e = 0; e < NE; ++e) {  // R^T = I, or the prefix of the leaf
        const int j = L<D>::row(lane, e), i = L<D>::col(lane, e);
        if constexpr (TRAJ) {
            const double2 v = p.traj_pin[(size_t)leaf * DD + i * D + j];
            bad_prefix |= !(fabs(v.x) < 2.0) || !(fabs(v.y) < 2.0);
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
    // trajectory mode: the outputs of slices bad_from, bad_from + 1, ... of the leaf are NaN, those before it are valid
    int bad_from = TRAJ && __any_sync(0xffffffffu, bad_prefix) ? 0 : len;

    for (int t0 = 0; t0 < len; t0 += kGT) {
        __syncwarp();
        unsigned tile_flags = 0;
        if (lane < kGT) {
            const bool act = t0 + lane < len;
            double *gcol = gam + lane;
            slice_coefficients<double, INTEG, kGT>(p, j0 + t0 + lane, act, gcol);
            double nu = 0.0;
            for (int e = 0; e < nb; ++e) nu = fma(fabs(gcol[e * kGT]), bnorm[e], nu);
            cls[lane] = find_class(p, nu, &tile_flags);
            flags |= tile_flags;
        }
        if constexpr (TRAJ) {
            const unsigned m = __ballot_sync(0xffffffffu, tile_flags != 0);
            if (m) bad_from = min(bad_from, t0 + __ffs(m) - 1);
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
                    const double bad = t0 + rr >= bad_from ? nan("") : 0.0;
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
