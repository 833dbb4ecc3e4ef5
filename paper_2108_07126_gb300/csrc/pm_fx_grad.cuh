// Scans over the leaf products and the adjoint sweep of the gradient for D = 8 and 16 in FP64, on the digit
// products of pm_fx.cuh (the method and its formulas: pm_grad.cuh).
//
// Scans: groups of eight block products are multiplied first (fx_group_kernel); then one thread block per forward
// block and direction multiplies the group totals and blocks before (after) its own and combines the result with
// its leaves in a log-depth scan (fx_scan_kernel).  A sequential scan over 152 blocks costs 152 dependent
// products on one SM.
//
// Adjoint: one warp per leaf, backwards from the leaf's end.  With P_j = U_j ... U_1, W_j = V^dagger U_N ... U_{j+1}:
//   dz/dc = Tr(P_{j-1} W_j L_X(dX/dc)) = Tr(M dX/dc),  M = U_j^dagger M',
//   M' = the upper-right block of exp([[X, P_j W_j], [0, X]])
// (L_X(E) = int e^{sX} E e^{-sX} ds U_j, so the prefix after the slice enters instead of the one before), and
// P_{j-1} = U_j^dagger P_j.  So one sweep needs neither stored prefixes nor the forward exponentials a second time.
// The warp keeps the transposed matrices: Y = X^T (anti-Hermitian like X), P^T, W^T, M^T; then every product has
// its left operand in registers layout and the right operands M^T <- M'^T conj(U), P^T <- P^T conj(U) are the
// digits of exp(Y) with a sign flip.  conj(z) / d is folded into W, so that the gradient is a real combination of
// t_e = Im Tr(M B_e); the traces of sixteen slices are one digit GEMM against the basis.
#pragma once

#include <climits>

#include "pm_fx.cuh"
#include "pm_grad.cuh"

namespace pm {
namespace fx {

// ---------------------------------------------------------------- scans

// tile of M^T from a row-major double matrix
template <int D> __device__ __forceinline__ void ld_transposed(const double2 *m, int lane, Tile<D> &t, unsigned &bad) {
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e) {
        const double2 v = __ldg(m + L<D>::col(lane, e) * D + L<D>::row(lane, e));
        bad |= !(fabs(v.x) < 2.0) || !(fabs(v.y) < 2.0);
        t.re[e] = from_double(v.x, 0);
        t.im[e] = from_double(v.y, 0);
    }
}
template <int D> __device__ __forceinline__ void ld_natural(const double2 *m, int lane, Tile<D> &t, unsigned &bad) {
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e) {
        const double2 v = __ldg(m + L<D>::row(lane, e) * D + L<D>::col(lane, e));
        bad |= !(fabs(v.x) < 2.0) || !(fabs(v.y) < 2.0);
        t.re[e] = from_double(v.x, 0);
        t.im[e] = from_double(v.y, 0);
    }
}
// transposed tile -> row-major doubles (NaN when bad)
template <int D> __device__ __forceinline__ void st_doubles(double2 *m, int lane, const Tile<D> &t, unsigned bad) {
    const double n = bad ? nan("") : 0.0;
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e)
        m[L<D>::col(lane, e) * D + L<D>::row(lane, e)] = make_double2(to_double(t.re[e]) + n, to_double(t.im[e]) + n);
}

constexpr int kGroup = 8;      // blocks per group
constexpr int kScanWarps = 8;  // warps per scan block
template <int D> struct ScanSmem {
    // elements of a leaf scan: the leaves of a forward block (FP32 D = 8: 64, else at most 16) and U(T)
    static constexpr int MAXE = D == 8 ? 65 : 17;
    static constexpr int TILE = Cfg<D>::TILE, RHS = Cfg<D>::RHS;
    static constexpr size_t BYTES = (size_t)MAXE * TILE + (size_t)kScanWarps * RHS;
};

// out^T = early^T late^T for transposed tiles in shared memory
template <int D>
__device__ __forceinline__ void combine(const longlong2 *late, const longlong2 *early, uint32_t *rhs, int lane, Tile<D> &out) {
    Digits<D> d;
    Tile<D> t;
    ld_priv<D>(late, lane, t);
    split<D>(t, d);
    put_rhs<D>(rhs, lane, d, kTrans);
    ld_priv<D>(early, lane, t);
    split<D>(t, d);
    mul(d, rhs, lane, out);
}

// product of m matrices (matrix i at ptr(i), later ones on the left) by the warps of the block -> transposed tile 0
template <int D, typename Fn>
__device__ void block_chain(int m, Fn &&ptr, longlong2 *tiles, uint32_t *rhs, int lane, int warp, unsigned &bad) {
    Tile<D> t;
#pragma unroll
    for (int e = 0; e < L<D>::NE; ++e) {
        t.re[e] = L<D>::row(lane, e) == L<D>::col(lane, e) ? (i64)1 << F : 0;
        t.im[e] = 0;
    }
    const int a = m * warp / kScanWarps, b = m * (warp + 1) / kScanWarps;
    for (int i = a; i < b; ++i) {
        if (i == a) {
            ld_transposed<D>(ptr(i), lane, t, bad);
        } else {  // t <- t m^T
            Tile<D> x;
            Digits<D> d;
            ld_natural<D>(ptr(i), lane, x, bad);
            split<D>(x, d);
            put_rhs<D>(rhs, lane, d, kPlain);
            split<D>(t, d);
            mul(d, rhs, lane, t);
        }
    }
    longlong2 *mine = tiles + (size_t)warp * L<D>::NE * 32;
    st_priv<D>(mine, lane, t);
    __syncthreads();
    for (int h = 1; h < kScanWarps && m > 0; h <<= 1) {
        const int left = warp * 2 * h;
        if (left + h < kScanWarps)
            combine<D>(tiles + (size_t)(left + h) * L<D>::NE * 32, tiles + (size_t)left * L<D>::NE * 32, rhs, lane, t);
        __syncthreads();
        if (left + h < kScanWarps) st_priv<D>(tiles + (size_t)left * L<D>::NE * 32, lane, t);
        __syncthreads();
    }
}

// product of each group of kGroup blocks
template <int D>
__global__ void __launch_bounds__(kScanWarps * 32) fx_group_kernel(const double2 *blocks, int n, double2 *groups) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    longlong2 *tiles = (longlong2 *)smem;
    uint32_t *rhs = (uint32_t *)(smem + (size_t)ScanSmem<D>::MAXE * ScanSmem<D>::TILE + (size_t)warp * ScanSmem<D>::RHS);
    const int first = blockIdx.x * kGroup, m = min(kGroup, n - first);
    unsigned bad = 0;
    // a chain of m factors spread over kScanWarps warps leaves empty warps at identity for m < 8
    const int a = warp < m;
    Tile<D> t;
    if (a) ld_transposed<D>(blocks + (size_t)(first + warp) * D * D, lane, t, bad);
    else {
#pragma unroll
        for (int e = 0; e < L<D>::NE; ++e) {
            t.re[e] = L<D>::row(lane, e) == L<D>::col(lane, e) ? (i64)1 << F : 0;
            t.im[e] = 0;
        }
    }
    st_priv<D>(tiles + (size_t)warp * L<D>::NE * 32, lane, t);
    const int any = __syncthreads_or((int)bad);
    for (int h = 1; h < kScanWarps; h <<= 1) {
        const int left = warp * 2 * h;
        if (left + h < kScanWarps)
            combine<D>(tiles + (size_t)(left + h) * L<D>::NE * 32, tiles + (size_t)left * L<D>::NE * 32, rhs, lane, t);
        __syncthreads();
        if (left + h < kScanWarps) st_priv<D>(tiles + (size_t)left * L<D>::NE * 32, lane, t);
        __syncthreads();
    }
    if (warp == 0) {
        ld_priv<D>(tiles, lane, t);
        st_doubles<D>(groups + (size_t)blockIdx.x * D * D, lane, t, any);
    }
}

// Exclusive prefixes (blockIdx.y = 0) or suffixes (1) of the leaves of forward block blockIdx.x; the prefix block of
// the last forward block also writes U(T) (pin[L], U_out), z and the loss.  A bad leaf (NaN, which fixed point has not) makes
// the elements that contain it NaN: the prefixes of later leaves, the suffixes of earlier ones.
template <int D>
__global__ void __launch_bounds__(kScanWarps * 32) fx_scan_kernel(const ScanParams sp, const double2 *groups) {
    constexpr int NT = L<D>::NE * 32, DD = D * D;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x, n = sp.n_blocks, nl = sp.leaves_per_block;
    const bool suf = blockIdx.y != 0;
    __shared__ int s_bad;  // the bad element nearest to the seed
    if (threadIdx.x == 0) s_bad = suf ? -1 : INT_MAX;
    longlong2 *tiles = (longlong2 *)smem;
    uint32_t *rhs = (uint32_t *)(smem + (size_t)ScanSmem<D>::MAXE * ScanSmem<D>::TILE + (size_t)warp * ScanSmem<D>::RHS);
    const int gb = b / kGroup, ng = (n + kGroup - 1) / kGroup;
    unsigned bad = 0;
    if (!suf) {  // groups before b's, then the blocks of b's group before b
        block_chain<D>(gb + b % kGroup, [&](int i) { return i < gb ? groups + (size_t)i * DD : sp.blockpart + (size_t)(gb * kGroup + i - gb) * DD; },
                       tiles, rhs, lane, warp, bad);
    } else {  // the blocks of b's group after b, then the later groups
        const int in = min(kGroup * (gb + 1), n) - 1 - b;
        block_chain<D>(in + ng - 1 - gb, [&](int i) { return i < in ? sp.blockpart + (size_t)(b + 1 + i) * DD : groups + (size_t)(gb + 1 + i - in) * DD; },
                       tiles, rhs, lane, warp, bad);
    }
    const bool seed_bad = __syncthreads_or((int)bad) != 0;
    // elements: prefix x_0 = seed, x_l = leaf_{l-1} (one more for U(T)); suffix x_{nl-1} = seed, x_l = leaf_{l+1}
    const double2 *leaf = sp.leafpart + (size_t)b * nl * DD;
    const bool last = !suf && b == n - 1;
    const int ne = nl + (last ? 1 : 0);
    Tile<D> t;
    if (suf && nl > 1) {
        if (warp == 0) {
            ld_priv<D>(tiles, lane, t);
            st_priv<D>(tiles + (size_t)(nl - 1) * NT, lane, t);
        }
        __syncthreads();
    }
    for (int l = warp; l < ne; l += kScanWarps) {
        if (l == (suf ? nl - 1 : 0)) continue;
        bad = 0;
        ld_transposed<D>(leaf + (size_t)(suf ? l + 1 : l - 1) * DD, lane, t, bad);
        st_priv<D>(tiles + (size_t)l * NT, lane, t);
        if (bad) {
            if (suf) atomicMax(&s_bad, l);
            else atomicMin(&s_bad, l);
        }
    }
    __syncthreads();
    constexpr int PER = (ScanSmem<D>::MAXE + kScanWarps - 1) / kScanWarps;
    for (int off = 1; off < ne; off <<= 1) {
        Tile<D> r[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int l = warp + k * kScanWarps;
            if (!suf && l < ne && l >= off) combine<D>(tiles + (size_t)l * NT, tiles + (size_t)(l - off) * NT, rhs, lane, r[k]);
            if (suf && l + off < ne) combine<D>(tiles + (size_t)(l + off) * NT, tiles + (size_t)l * NT, rhs, lane, r[k]);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int l = warp + k * kScanWarps;
            if (suf ? l + off < ne : (l < ne && l >= off)) st_priv<D>(tiles + (size_t)l * NT, lane, r[k]);
        }
        __syncthreads();
    }
    double2 *out = (suf ? sp.sout : sp.pin) + (size_t)b * nl * DD;
    for (int l = warp; l < ne; l += kScanWarps) {
        ld_priv<D>(tiles + (size_t)l * NT, lane, t);
        st_doubles<D>(out + (size_t)l * DD, lane, t, seed_bad || (suf ? l <= s_bad : l >= s_bad));
    }
    if (!last) return;
    __syncthreads();
    const double2 *U = sp.pin + (size_t)n * nl * DD;
    if (sp.vdag && warp == 0) {
        double zr = 0.0, zi = 0.0;
        for (int e = lane; e < DD; e += 32) {
            const double2 x = sp.vdag[e], y = U[(e % D) * D + e / D];
            zr = fma(x.x, y.x, fma(-x.y, y.y, zr));
            zi = fma(x.x, y.y, fma(x.y, y.x, zi));
        }
        for (int off = 16; off > 0; off >>= 1) {
            zr += __shfl_xor_sync(0xffffffffu, zr, off);
            zi += __shfl_xor_sync(0xffffffffu, zi, off);
        }
        if (lane == 0) {
            const double dd = (double)sp.d_out;
            sp.z[0] = zr;
            sp.z[1] = zi;
            sp.z[2] = 1.0 - (zr * zr + zi * zi) / (dd * dd);
        }
    }
    if (sp.U_out) {
        const int d = sp.d_out;
        for (int e = threadIdx.x; e < d * d; e += blockDim.x) {
            const double2 v = U[(e / d) * D + (e % d)];
            if (sp.out_c128) ((double2 *)sp.U_out)[e] = v;
            else ((float2 *)sp.U_out)[e] = make_float2((float)v.x, (float)v.y);
        }
    }
}

template <int D> cudaError_t scan_run(const ScanParams &sp, double2 *groups, bool suffixes, cudaStream_t st) {
    const int smem = (int)ScanSmem<D>::BYTES;
    cudaError_t e = cudaFuncSetAttribute(fx_group_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fx_scan_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    fx_group_kernel<D><<<(sp.n_blocks + kGroup - 1) / kGroup, kScanWarps * 32, smem, st>>>(sp.blockpart, sp.n_blocks, groups);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    fx_scan_kernel<D><<<dim3(sp.n_blocks, suffixes ? 2 : 1), kScanWarps * 32, smem, st>>>(sp, groups);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- the adjoint sweep

template <int D> struct AdjCfg {
    static constexpr int W = D == 16 ? 8 : 16;                  // warps per block
    static constexpr bool TILES_GLOBAL = D == 16;               // 24 KB of tiles per warp: in L2 for D = 16
    static constexpr int NTILE = 6;                             // Y, Y^2, D1, D2, P^T, W^T
    static constexpr int TILE = Cfg<D>::TILE, RHS = Cfg<D>::RHS;
    // global memory per leaf: packed exponents and M of a tile of slices, and the tiles
    static constexpr size_t LEAF_BYTES = (size_t)kGT * D * D * 8 * 3 + (TILES_GLOBAL ? (size_t)NTILE * TILE : 0);
};
template <int D> __host__ __device__ inline size_t adj_warp_bytes(int nb) {
    // three right operands (their space holds the coefficients, then the traces of a tile), tiles, class tile
    const size_t gam = (size_t)(nb + 8) * kGT * 8, r = (size_t)3 * AdjCfg<D>::RHS;
    return (gam > r ? gam : r) + (AdjCfg<D>::TILES_GLOBAL ? 0 : (size_t)AdjCfg<D>::NTILE * AdjCfg<D>::TILE) + 64;
}
template <int D> __host__ __device__ inline size_t adj_smem_bytes(int nb, int warps) {
    return (size_t)warps * adj_warp_bytes<D>(nb) + (((size_t)nb * 8 + 15) & ~(size_t)15);
}
__host__ __device__ constexpr int ntiles_of(int nb) { return nb > 0 ? (nb + 7) / 8 : 1; }
template <int D> __host__ __device__ constexpr size_t trace_digit_bytes(int nb) {
    return (size_t)(2 * D * D / 16) * ntiles_of(nb) * ND * 32 * sizeof(uint2);
}

// The basis as the right operand of the trace GEMM t_e = Im Tr(M B_e) = sum_pq Re(M^T)_pq Im(B_e)_pq +
// Im(M^T)_pq Re(B_e)_pq: 2 D^2 terms (first the D^2 of Im B), word pair (kstep, tile of eight matrices, digit, lane).
template <int D>
__global__ void __launch_bounds__(32) trace_digits_kernel(const double *packed, const double *bnorm, int nb, uint2 *out) {
    constexpr int DD = D * D;
    const int lane = threadIdx.x, ks = blockIdx.x, nt = blockIdx.y, e = 8 * nt + (lane >> 2);
    uint32_t w[2][ND];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        i64 v[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int k = 16 * ks + 8 * h + 2 * (lane & 3) + c, pos = k % DD, p = pos / D, q = pos % D;
            double x = 0.0;
            if (e < nb) {
                const double *P = packed + (size_t)e * DD;  // upper triangle Re, strict lower Im
                if (k < DD) x = p > q ? P[p * D + q] : (p < q ? -P[q * D + p] : 0.0);
                else x = p <= q ? P[p * D + q] : P[q * D + p];
            }
            v[c] = e < nb ? from_double(x, basis_exp(bnorm[e])) : 0;
        }
        split_pair(v[0], v[1], w[h]);
    }
#pragma unroll
    for (int i = 0; i < ND; ++i) out[(((size_t)ks * gridDim.y + nt) * ND + i) * 32 + lane] = make_uint2(w[0][i], w[1][i]);
}

// t [slice][matrix] of a tile of sixteen slices from M^T (rows of 2 D^2 fixed-point numbers)
template <int D>
__device__ __forceinline__ void traces(const uint2 *bd, int nb, const double *bnorm, const i64 *m, int lane, double *t) {
    constexpr int DD = D * D, KS = 2 * DD / 16;
    const int g = lane >> 2, t4 = lane & 3, ntl = ntiles_of(nb);
    for (int nt = 0; nt < ntl; ++nt) {
        i64 o[4] = {0, 0, 0, 0};
#pragma unroll 1
        for (int k0 = 0; k0 < KS; k0 += 2) {
            float acc[NA][4];
            acc_init(acc);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                const int k = 16 * (k0 + ks) + 2 * t4;
                uint32_t a[4][ND];
                const longlong2 x0 = *reinterpret_cast<const longlong2 *>(m + (size_t)g * 2 * DD + k);
                const longlong2 x1 = *reinterpret_cast<const longlong2 *>(m + (size_t)(g + 8) * 2 * DD + k);
                const longlong2 x2 = *reinterpret_cast<const longlong2 *>(m + (size_t)g * 2 * DD + k + 8);
                const longlong2 x3 = *reinterpret_cast<const longlong2 *>(m + (size_t)(g + 8) * 2 * DD + k + 8);
                split_pair(x0.x, x0.y, a[0]);
                split_pair(x1.x, x1.y, a[1]);
                split_pair(x2.x, x2.y, a[2]);
                split_pair(x3.x, x3.y, a[3]);
                uint2 b[ND];
#pragma unroll
                for (int j = 0; j < ND; ++j) b[j] = __ldg(bd + (((size_t)(k0 + ks) * ntl + nt) * ND + j) * 32 + lane);
#pragma unroll
                for (int i = 0; i < ND; ++i)
#pragma unroll
                    for (int j = 0; j <= last_digit(i); ++j) mma(acc[i + j], a[0][i], a[1][i], a[2][i], a[3][i], b[j].x, b[j].y);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) o[u] += collect(acc, u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = 8 * nt + 2 * t4 + (u & 1);
            if (e < nb) t[(size_t)(g + 8 * (u >> 1)) * nb + e] = ldexp(to_double(o[u]), basis_exp(bnorm[e]));
        }
    }
}

template <int D, int INTEG>
__global__ void __launch_bounds__(AdjCfg<D>::W * 32, 1) fx_adjoint_kernel(const GradParams p) {
    constexpr int NE = L<D>::NE, DD = D * D, PS = Cfg<D>::PS, EPL = DD / 32, NT = NE * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int nb = p.n_basis, K = p.K;
    const size_t wb = adj_warp_bytes<D>(nb);
    unsigned char *wbase = smem + (size_t)warp * wb;
    const int64_t slot = (int64_t)blockIdx.x * W + warp, leaf = p.fx_leaf0 + slot, NL = p.n_leaves, N = p.n_steps;
    double *bnorm = (double *)(smem + (size_t)W * wb);
    for (int i = tid; i < nb; i += blockDim.x) bnorm[i] = p.bnorm1[i];
    __syncthreads();
    if (slot >= p.fx_slots || leaf >= NL) return;  // no block barrier below
    const int64_t j0 = N * leaf / NL;
    const int len = (int)(N * (leaf + 1) / NL - j0);
    if (len <= 0) return;

    i64 *gbuf = (i64 *)((unsigned char *)p.fx_g + (size_t)slot * AdjCfg<D>::LEAF_BYTES);
    i64 *mbuf = gbuf + kGT * DD;
    uint32_t *r1 = (uint32_t *)wbase, *r2 = r1 + rhs_words<D>(), *r3 = r2 + rhs_words<D>();
    longlong2 *tiles = AdjCfg<D>::TILES_GLOBAL ? (longlong2 *)(mbuf + 2 * kGT * DD)
                                               : (longlong2 *)(wbase + wb - 64 - (size_t)AdjCfg<D>::NTILE * AdjCfg<D>::TILE);
    longlong2 *SY = tiles, *SY2 = tiles + NT, *SD1 = tiles + 2 * NT, *SD2 = tiles + 3 * NT, *SP = tiles + 4 * NT,
              *SW = tiles + 5 * NT;
    i64 *xpk = (i64 *)r1;  // packed exponent, before the right operands
    double *gam = (double *)wbase;  // coefficients of a tile (before its slices), traces of a tile (after them)
    int *cls = (int *)(wbase + wb - 64);
    const double *ctrl = (const double *)p.ctrl;

    unsigned flags = 0, bad = 0;
    const double gscale = -2.0 / p.d_true;  // 1 / d is in W
    // W = conj(z) / d V^dagger S enters scaled by a power of two to a norm near one (p.z[3] >= ||V||_2^2)
    const double wn = sqrt(p.z[3] * (p.z[0] * p.z[0] + p.z[1] * p.z[1])) / p.d_true;
    const int ve = (wn > 1e-150 && wn < 1e150) ? ilogb(wn) + 1 : 0;

    auto split_of = [&](const longlong2 *S, Digits<D> &d) {
        Tile<D> t;
        ld_priv<D>(S, lane, t);
        split<D>(t, d);
    };
    // x / k!
    auto over = [&](i64 x, int k) -> i64 { return k <= 1 ? x : (k == 2 ? halve(x) : mulc(x, c_inv[k])); };
    auto axpy = [&](Tile<D> &a, const longlong2 *S, int k) {  // a += S / k!
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const longlong2 x = S[e * 32 + lane];
            a.re[e] += over(x.x, k);
            a.im[e] += over(x.y, k);
        }
    };
    auto scale = [&](Tile<D> &a, int k) {
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            a.re[e] = over(a.re[e], k);
            a.im[e] = over(a.im[e], k);
        }
    };

    // P^T at the leaf's end (the prefix of the next leaf; U(T) after the last), W^T = (conj(z) / d V^dagger S)^T
    {
        Tile<D> t;
        ld_transposed<D>(p.pin + (size_t)(leaf + 1) * DD, lane, t, bad);
        st_priv<D>(SP, lane, t);
        // S V'^T...: W^T = S^T (z* V^dagger / d)^T: left operand S^T, right operand digits of (z* / d) V^dagger, natural
        const double sc = ldexp(1.0 / p.d_true, -ve), zr = p.z[0] * sc, zi = p.z[1] * sc;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const double2 v = __ldg(p.vdag + L<D>::row(lane, e) * D + L<D>::col(lane, e));
            const double re = fma(zr, v.x, zi * v.y), im = fma(zr, v.y, -zi * v.x);
            bad |= !(fabs(re) < 2.0) || !(fabs(im) < 2.0);
            t.re[e] = from_double(re, 0);
            t.im[e] = from_double(im, 0);
        }
        Digits<D> d;
        split<D>(t, d);
        put_rhs<D>(r1, lane, d, kPlain);
        ld_transposed<D>(p.sout + (size_t)leaf * DD, lane, t, bad);
        split<D>(t, d);
        mul(d, r1, lane, t);
        st_priv<D>(SW, lane, t);
    }

    for (int t0 = ((len - 1) / kGT) * kGT; t0 >= 0; t0 -= kGT) {
        const int nr = min(kGT, len - t0);
        __syncwarp();
        if (lane < kGT) {
            double *gcol = gam + lane;
            slice_coefficients<double, INTEG, kGT>(p, j0 + t0 + lane, lane < nr, gcol);
            double nu = 0.0;
            for (int e = 0; e < nb; ++e) nu = fma(fabs(gcol[e * kGT]), bnorm[e], nu);
            int c = p.n_dcls - 1;  // first class (derivative bound) that covers nu
            if (!(nu <= p.dcls_cap[c])) {
                flags |= (isnan(nu) || isinf(nu)) ? kDevNonfinite : kDevCapped;
            } else {
                int lo = 0, hi = c;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (nu <= p.dcls_cap[mid]) hi = mid; else lo = mid + 1;
                }
                c = lo;
            }
            cls[lane] = p.dcls_code[c];
        }
        __syncwarp();
        assemble_tile<D>((const uint2 *)p.fx_basis, nb, gam, cls_s(cls[lane >> 2]), cls_s(cls[(lane >> 2) + 8]), bnorm, lane, gbuf);
        __syncwarp();

        for (int rr = nr - 1; rr >= 0; --rr) {
            const int code = cls[rr], q = cls_q(code), rh = cls_r(code), s = cls_s(code);
            Tile<D> T, M;
            Digits<D> dt, dm;  // digits of the T and M chains: each matrix is split once per use as both operands
            {
                const longlong2 *src = reinterpret_cast<const longlong2 *>(gbuf + (size_t)rr * DD) + lane;
#pragma unroll
                for (int t = 0; t < EPL / 2; ++t) {
                    const longlong2 v = src[32 * t];
                    const int pos = 2 * (lane + 32 * t);
                    i64 *dst = xpk + (pos / D) * PS + (pos % D);
                    dst[0] = v.x;
                    dst[1] = v.y;
                }
            }
            __syncwarp();
            // Y = X^T: Re Y_ij = Im G_ji, Im Y_ij = -Re G_ji
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                const int i = L<D>::row(lane, e), j = L<D>::col(lane, e);
                const i64 a = xpk[i * PS + j], b = xpk[j * PS + i];
                T.re[e] = j > i ? b : (j < i ? -a : 0);
                T.im[e] = -(i <= j ? a : b);
            }
            __syncwarp();
            st_priv<D>(SY, lane, T);

            // (P_j W_j)^T = W^T P^T, scaled by 2^-s like Y
            split_of(SP, dt);
            put_rhs<D>(r3, lane, dt, kTrans);
            split_of(SW, dt);
            mul(dt, r3, lane, M);
            if (s > 0) {
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    M.re[e] = (M.re[e] + (1ll << (s - 1))) >> s;
                    M.im[e] = (M.im[e] + (1ll << (s - 1))) >> s;
                }
            }
            st_priv<D>(SD1, lane, M);  // D1

            // powers Y^k and their derivatives D_k; T = Y^q and M = D_q at the end
            uint32_t *rY = r1, *rD = r2;
            split<D>(T, dt);
            split<D>(M, dm);
            put_rhs<D>(rY, lane, dt, kAntiHerm);
            put_rhs<D>(rD, lane, dm, kTrans);
            for (int k = 2; k <= q; ++k) {
                // D2 = D1 Y + Y D1, D3 = D2 Y + Y^2 D1
                mul_sum(dm, rY, dt, rD, lane, M);
                mul(dt, rY, lane, T);
                if (k < q) {
                    st_priv<D>(SY2, lane, T);
                    st_priv<D>(SD2, lane, M);
                    split<D>(T, dt);
                    split<D>(M, dm);
                }
            }
            if (rh > 1) {  // Y^q and D_q as right operands of the Horner steps
                split<D>(T, dt);
                put_rhs<D>(rY, lane, dt, q == 2 ? kHerm : kAntiHerm);
                split<D>(M, dm);
                put_rhs<D>(rD, lane, dm, kTrans);
            }
            auto add_block = [&](int b) {
                const i64 a0 = c_inv_fx[q * b];
#pragma unroll
                for (int e = 0; e < NE; ++e)
                    if (L<D>::row(lane, e) == L<D>::col(lane, e)) T.re[e] += a0;
                if (q >= 2) {
                    axpy(T, SY, q * b + 1);
                    axpy(M, SD1, q * b + 1);
                }
                if (q >= 3) {
                    axpy(T, SY2, q * b + 2);
                    axpy(M, SD2, q * b + 2);
                }
            };
            scale(T, q * rh);
            scale(M, q * rh);
            add_block(rh - 1);
            // Horner steps T <- T Y^q + B_b, M <- M Y^q + T D_q + its derivative, then squarings M <- M T + T M, T <- T T
            for (int i = rh - 2; i >= -s; --i) {
                split<D>(T, dt);
                split<D>(M, dm);
                if (i < 0) {
                    put_rhs<D>(rY, lane, dt, kTrans);
                    put_rhs<D>(rD, lane, dm, kTrans);
                }
                mul_sum(dm, rY, dt, rD, lane, M);
                mul(dt, rY, lane, T);
                if (i >= 0) add_block(i);
            }
            // V = exp(Y) = U^T: M^T <- M'^T V^dagger, P^T <- P^T V^dagger, W^T <- V W^T
            split<D>(T, dt);
            put_rhs<D>(r1, lane, dt, kHerm);  // the digits of conj(V) = (V^dagger)^T
            split<D>(M, dm);
            mul(dm, r1, lane, M);
            split_of(SP, dm);
            mul(dm, r1, lane, T);
            st_priv<D>(SP, lane, T);
            split_of(SW, dm);
            put_rhs<D>(r3, lane, dm, kTrans);
            mul(dt, r3, lane, T);
            st_priv<D>(SW, lane, T);
            // M^T of the slice for the traces
#pragma unroll
            for (int e = 0; e < NE; e += 2) {
                const int pos = L<D>::row(lane, e) * D + L<D>::col(lane, e);
                *reinterpret_cast<longlong2 *>(mbuf + (size_t)rr * 2 * DD + pos) = make_longlong2(M.re[e], M.re[e + 1]);
                *reinterpret_cast<longlong2 *>(mbuf + (size_t)rr * 2 * DD + DD + pos) = make_longlong2(M.im[e], M.im[e + 1]);
            }
            __syncwarp();
        }

        // t_e of the tile's slices, then dL/dc = -(2 / d) sum_e (d gamma_e / dc) t_e (scaled back by 2^ve)
        double *tr = gam;
        traces<D>((const uint2 *)p.fx_trace, nb, bnorm, mbuf, lane, tr);
        __syncwarp();
        const bool any_bad = __any_sync(0xffffffffu, flags || bad);
        const double h = p.dt, gs = any_bad ? nan("") : ldexp(gscale, ve);
        const int R = (INTEG == kMidpoint) ? 1 : ((INTEG == kGL2) ? 2 : 3);
        for (int w = lane; w < nr * K * R; w += 32) {
            const int rr = w % nr, kr = w / nr, k = kr / R, role = kr % R;
            const int64_t j = j0 + t0 + rr;
            const double *te = tr + (size_t)rr * nb;
            auto T = [&](int raw) -> double {
                const int sl = p.slot_of[raw];
                return sl >= 0 ? te[sl] : 0.0;
            };
            auto emit = [&](int64_t sidx, double v) {
                double *gr = (double *)p.grad + (size_t)k * p.S + sidx;
                if (INTEG == kSimpson) atomicAdd(gr, gs * v);  // end points are shared by two slices
                else *gr = gs * v;
            };
            if (INTEG == kMidpoint) {
                emit(j, h * T(1 + k));
                continue;
            }
            // samples of the slice: GL4 nodes (2j, 2j + 1); Simpson (2j, 2j + 1, 2j + 2)
            const double wc = (INTEG == kGL2) ? (1.7320508075688772 / 12.0) * h * h : h * h / 12.0;
            const double w1 = (INTEG == kGL2) ? h * 0.5 : h / 6.0;
            const int64_t s1 = 2 * j, s2 = (INTEG == kGL2) ? 2 * j + 1 : 2 * j + 2;
            if (INTEG == kSimpson && role == 1) {  // centre sample: Omega_1 only
                emit(2 * j + 1, 4.0 * h / 6.0 * T(1 + k));
                continue;
            }
            const bool first = (role == 0);  // c1 (first node / start) or c2 (second node / end)
            double v = w1 * T(1 + k) + (first ? -wc : wc) * T(1 + K + k);
            // pairs (a, b), a < b: gamma = wc (c1_a c2_b - c2_a c1_b)
            int e = 1 + 2 * K;
            for (int a = 0; a < K; ++a)
                for (int b = a + 1; b < K; ++b, ++e) {
                    if (a != k && b != k) continue;
                    double cf;
                    if (first) cf = (k == a) ? wc * ctrl[(int64_t)b * p.S + s2] : -wc * ctrl[(int64_t)a * p.S + s2];
                    else cf = (k == b) ? wc * ctrl[(int64_t)a * p.S + s1] : -wc * ctrl[(int64_t)b * p.S + s1];
                    v = fma(cf, T(e), v);
                }
            emit(first ? s1 : s2, v);
        }
    }
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (lane == 0 && flags) atomicOr(p.status, flags);
}

// One launch, or with fewer workspace slots than leaves (a cap far below the default) one per fx_slots leaves: a loop over
// the leaves in the kernel cost every call 7 % (registers: d = 8, N = 65536 1.53 -> 1.63 ms).
template <int D, int INTEG> cudaError_t adjoint_launch(GradParams gp, int sm_count, size_t optin, cudaStream_t st) {
    auto k = fx_adjoint_kernel<D, INTEG>;
    int w = AdjCfg<D>::W;
    while (w > 1 && adj_smem_bytes<D>(gp.n_basis, w) > optin) --w;
    // short runs: fewer warps per block, so that the leaves spread over the SMs
    while (w > 1 && (gp.fx_slots + w - 1) / w < sm_count) w = (w + 1) / 2;
    const size_t smem = adj_smem_bytes<D>(gp.n_basis, w);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    for (gp.fx_leaf0 = 0; gp.fx_leaf0 < gp.n_leaves && e == cudaSuccess; gp.fx_leaf0 += gp.fx_slots) {
        k<<<(unsigned)((gp.fx_slots + w - 1) / w), w * 32, smem, st>>>(gp);
        e = cudaGetLastError();
    }
    return e;
}

template <int D>
cudaError_t trace_digits(const double *packed, const double *bnorm, int nb, void *out, cudaStream_t st) {
    trace_digits_kernel<D><<<dim3(2 * D * D / 16, ntiles_of(nb)), 32, 0, st>>>(packed, bnorm, nb, (uint2 *)out);
    return cudaGetLastError();
}

}  // namespace fx
}  // namespace pm
