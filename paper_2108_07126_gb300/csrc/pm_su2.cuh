// U(T) of two-level systems (d = 1, 2), one thread per leaf.
//
// A Hermitian 2 x 2 exponent is G = m I + x sx + y sy + z sz, so
//   exp(-i G) = e^{-i m} (cos r I - i (sin r / r) (x sx + y sy + z sz)),  r^2 = x^2 + y^2 + z^2:
// cos r and sin r / r are two short real Taylor polynomials in r^2 (after s halvings, undone by s doublings), a
// product of two slice propagators is a product of unit quaternions (16 multiply-adds instead of 32), and the phases
// m add up.  A slice takes about 50 operations in registers; the matrix scheme of pm_fused.cuh takes 6 products of 32
// multiply-adds and their traffic through shared memory.
//
// The phases are added as 128-bit integers in units of 2^-60, exact in any order, and the trace and the difference of the diagonal
// are taken slice by slice: as sums of doubles the phases rounded at the size of the total, and half the sum of a basis matrix's
// diagonal was rounded once for all slices (d = 2 with a trace, N = 16384: error 9e-14 against 80-bit floats, now 4e-14, as the
// matrix products).  Integer instructions, beside the FP64 pipe: times unchanged (Rabi 22.4 us).
//
// A short run is bound by latency: one slice per thread while the chip has room (each step of the tree costs less
// than a slice), the warp and block trees in registers and shuffles, and the block that arrives last multiplies
// all block partials at once instead of climbing a tree of arrivals.
#pragma once

#include "pm_fused.cuh"

namespace pm {
namespace su2 {

typedef unsigned long long u64;
typedef unsigned __int128 u128;

// a I - i (x sx + y sy + z sz), times e^{-i ph 2^-60} (ph in two's complement)
template <typename Real> struct Q {
    Real a, x, y, z;
    u128 ph;
};

constexpr double kTwoPiHi = 6.283185307179586, kTwoPiLo = 2.4492935982947064e-16, kInvTwoPi = 0.15915494309189535;

// m 2^60 mod 2 pi, two roundings (m - k 2 pi to 53 bits of 2 pi is exact); not a finite number: ok becomes false
__device__ __forceinline__ long long reduced_phase(double m, bool &ok) {
    ok = ok && isfinite(m);
    const double k = rint(m * kInvTwoPi);
    return __double2ll_rn(fma(-k, kTwoPiHi, m) * 0x1p60) + __double2ll_rn(-k * kTwoPiLo * 0x1p60);
}
__device__ __forceinline__ long long phase(double m, bool &ok) {
    return fabs(m) <= 4.0 ? fx::from_double(m, fx::F - 60) : reduced_phase(m, ok);  // integer instructions
}
__device__ __forceinline__ long long phase(float m, bool &ok) {
    return fabsf(m) <= 4.f ? __float2ll_rn(m * 0x1p60f) : reduced_phase((double)m, ok);
}
// ph 2^-60 mod 2 pi: its multiple of 2^-20 (53 bits) less k 2 pi is exact in one fma
__device__ __forceinline__ double angle(u128 ph) {
    const __int128 t = (__int128)ph;
    const double a = (double)(long long)(t >> 40) * 0x1p-20, b = (double)(long long)(ph & (((u64)1 << 40) - 1)) * 0x1p-60;
    const double k = rint(a * kInvTwoPi);
    return fma(-k, kTwoPiHi, a) + fma(-k, kTwoPiLo, b);
}
// Newton-Schulz step to norm one
template <typename Real> __device__ __forceinline__ void normalise(Q<Real> &q) {
    const Real f = Real(0.5) * (Real(3) - fma(q.a, q.a, fma(q.x, q.x, fma(q.y, q.y, q.z * q.z))));
    q.a *= f;
    q.x *= f;
    q.y *= f;
    q.z *= f;
}

// later * earlier
template <typename Real> __device__ __forceinline__ Q<Real> mul(const Q<Real> &l, const Q<Real> &e) {
    Q<Real> r;
    r.a = fma(l.a, e.a, -fma(l.x, e.x, fma(l.y, e.y, l.z * e.z)));
    r.x = fma(l.a, e.x, fma(l.x, e.a, fma(l.y, e.z, -l.z * e.y)));
    r.y = fma(l.a, e.y, fma(l.y, e.a, fma(l.z, e.x, -l.x * e.z)));
    r.z = fma(l.a, e.z, fma(l.z, e.a, fma(l.x, e.y, -l.y * e.x)));
    r.ph = l.ph + e.ph;
    return r;
}

template <typename Real> __device__ __forceinline__ Q<Real> shfl_down(const Q<Real> &q, int off) {
    Q<Real> r;
    r.a = __shfl_down_sync(0xffffffffu, q.a, off);
    r.x = __shfl_down_sync(0xffffffffu, q.x, off);
    r.y = __shfl_down_sync(0xffffffffu, q.y, off);
    r.z = __shfl_down_sync(0xffffffffu, q.z, off);
    const u64 lo = __shfl_down_sync(0xffffffffu, (u64)q.ph, off), hi = __shfl_down_sync(0xffffffffu, (u64)(q.ph >> 64), off);
    r.ph = (u128)hi << 64 | lo;
    return r;
}

template <typename Real> __device__ __forceinline__ Q<Real> identity() { return Q<Real>{Real(1), Real(0), Real(0), Real(0), (u128)0}; }

// ordered product over the threads of the block (thread 0 earliest) -> thread 0
template <typename Real> __device__ Q<Real> block_product(Q<Real> q, Q<Real> *sm, int W) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) q = mul(shfl_down(q, off), q);  // lanes beyond the last multiple are not used
    if (W == 1) return q;
    if (lane == 0) sm[warp] = q;
    __syncthreads();
    if (warp == 0) {
        q = lane < W ? sm[lane] : identity<Real>();
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) q = mul(shfl_down(q, off), q);
    }
    return q;
}

// cos r and sin r / r for r^2 = r2 <= 1/4: Taylor polynomials, remainder below the unit roundoff
__device__ __forceinline__ void cos_sinc(double r2, double &c, double &s) {
    c = fma(r2, -1.0 / 87178291200.0, 1.0 / 479001600.0);
    s = fma(r2, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
    c = fma(r2, -c, 1.0 / 3628800.0);
    s = fma(r2, -s, 1.0 / 39916800.0);
    c = fma(r2, -c, 1.0 / 40320.0);
    s = fma(r2, -s, 1.0 / 362880.0);
    c = fma(r2, -c, 1.0 / 720.0);
    s = fma(r2, -s, 1.0 / 5040.0);
    c = fma(r2, -c, 1.0 / 24.0);
    s = fma(r2, -s, 1.0 / 120.0);
    c = fma(r2, -c, 0.5);
    s = fma(r2, -s, 1.0 / 6.0);
    c = fma(r2, -c, 1.0);
    s = fma(r2, -s, 1.0);
}
__device__ __forceinline__ void cos_sinc(float r2, float &c, float &s) {
    c = fma(r2, -1.f / 3628800.f, 1.f / 40320.f);
    s = fma(r2, -1.f / 39916800.f, 1.f / 362880.f);
    c = fma(r2, -c, 1.f / 720.f);
    s = fma(r2, -s, 1.f / 5040.f);
    c = fma(r2, -c, 1.f / 24.f);
    s = fma(r2, -s, 1.f / 120.f);
    c = fma(r2, -c, 0.5f);
    s = fma(r2, -s, 1.f / 6.f);
    c = fma(r2, -c, 1.f);
    s = fma(r2, -s, 1.f);
}

constexpr int kMaxWarps = 8;
// largest power of r in cos r and sin r as polynomials
template <typename Real> __host__ __device__ constexpr int degree() { return sizeof(Real) == 8 ? 15 : 11; }

template <typename Real, int INTEG>
__global__ void __launch_bounds__(kMaxWarps * 32) su2_kernel(const FusedParams p) {
    __shared__ Q<Real> sm[kMaxWarps];
    __shared__ Q<double> smd[kMaxWarps];
    __shared__ double2 basis[kMaxBasis][2];  // (x, y) and half the diagonal (z + m, m - z) of every basis matrix
    __shared__ unsigned long long cnt[4];
    __shared__ unsigned s_flags;
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, W = blockDim.x >> 5, nb = p.n_basis;
    const Real *packed = (const Real *)p.packed;
    for (int e = tid; e < nb; e += blockDim.x) {
        const double p0 = packed[4 * e], p1 = packed[4 * e + 1], p2 = packed[4 * e + 2], p3 = packed[4 * e + 3];
        basis[e][0] = make_double2(p1, p2);
        basis[e][1] = make_double2(0.5 * p0, 0.5 * p3);
    }
    if (tid < 4) cnt[tid] = 0ull;
    if (tid == 0) s_flags = 0u;
    __syncthreads();

    const int64_t n_leaves = (int64_t)gridDim.x * blockDim.x, leaf = (int64_t)blockIdx.x * blockDim.x + tid;
    const int64_t j0 = p.n_steps * leaf / n_leaves;
    const int len = (int)(p.n_steps * (leaf + 1) / n_leaves - j0);
    Q<Real> R = identity<Real>();
    unsigned flags = 0;
    int s_max = 0;
    Real gam[kMaxBasis];
    for (int t = 0; t < len; ++t) {
        slice_coefficients<Real, INTEG, 1>(p, j0 + t, true, gam);
        Real x = 0, y = 0, g0 = 0, g1 = 0;
        double nu = 0.0;
        for (int e = 0; e < nb; ++e) {
            const double2 b0 = basis[e][0], b1 = basis[e][1];
            x = fma(gam[e], (Real)b0.x, x);
            y = fma(gam[e], (Real)b0.y, y);
            g0 = fma(gam[e], (Real)b1.x, g0);
            g1 = fma(gam[e], (Real)b1.y, g1);
            nu = fma(fabs((double)gam[e]), p.bnorm1[e], nu);
        }
        find_class(p, nu, &flags);  // NaN, infinite and capped norms (the halvings follow r itself)
        // the trace and the difference of the diagonal slice by slice: of the basis they would be rounded once for all slices
        Real z = g0 - g1;
        // halve until r <= 1/2, double back
        Real r2 = fma(x, x, fma(y, y, z * z));
        int s = 0;
        for (; r2 > Real(0.25) && s < 64; ++s) {
            x *= Real(0.5);
            y *= Real(0.5);
            z *= Real(0.5);
            r2 *= Real(0.25);
        }
        Real c, sc;
        cos_sinc(r2, c, sc);
        for (int i = 0; i < s; ++i) {  // cos 2r = cos^2 - sin^2, sin 2r = 2 sin cos (sin r = sc r)
            const Real c2 = fma(c, c, -(sc * sc) * r2);
            sc = Real(2) * c * sc;
            c = c2;
        }
        s_max = max(s_max, s);
        bool ok = true;
        const __int128 ph = (__int128)phase(g0, ok) + phase(g1, ok);
        if (!ok) c = (Real)nan("");
        R = mul(Q<Real>{c, sc * x, sc * y, sc * z, (u128)ph}, R);
    }
    // FP32: the Newton-Schulz step on a unit quaternion, on the block's product in double (below) and on leaves of more than 16
    // slices.  The norm of a slice is exact to a rounding; it drifts in the products (Rabi qubit, N = 16384 in leaves of one
    // slice: 2.7e-5 with the step on every leaf alone)
    if (p.unitary_step && p.n_steps > 16 * n_leaves) normalise(R);
    // statistics (no matrix products in the exponentials)
    const unsigned wl = __reduce_add_sync(0xffffffffu, (unsigned)len);
    const int ws = __reduce_max_sync(0xffffffffu, s_max);
    const unsigned wf = __reduce_or_sync(0xffffffffu, flags);
    if (lane == 0) {
        atomicAdd(&cnt[1], (unsigned long long)wl);
        if (wl) atomicMax(&cnt[2], (unsigned long long)degree<Real>());
        atomicMax(&cnt[3], (unsigned long long)ws);
        if (wf) atomicOr(&s_flags, wf);
    }
    R = block_product(R, sm, W);
    __syncthreads();
    Q<double> U{(double)R.a, (double)R.x, (double)R.y, (double)R.z, R.ph};
    if (p.unitary_step) normalise(U);

    if (gridDim.x > 1) {
        double *part = (double *)p.partials;
        if (tid == 0) {
            double *o = part + (size_t)blockIdx.x * 8;
            __stcg(o, U.a);
            __stcg(o + 1, U.x);
            __stcg(o + 2, U.y);
            __stcg(o + 3, U.z);
            __stcg((u64 *)o + 4, (u64)U.ph);
            __stcg((u64 *)o + 5, (u64)(U.ph >> 64));
            atomicAdd(&p.counters[0], cnt[0]);
            atomicAdd(&p.counters[1], cnt[1]);
            atomicMax(&p.counters[2], cnt[2]);
            atomicMax(&p.counters[3], cnt[3]);
            if (s_flags) atomicOr(&p.status[0], s_flags);
            __threadfence();
            s_last = atomicAdd(&p.tickets[0], 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        // the last block: the partials in order, a contiguous range per thread
        const int n = gridDim.x, a = (int)((int64_t)n * tid / blockDim.x), b = (int)((int64_t)n * (tid + 1) / blockDim.x);
        Q<double> q = identity<double>();
        for (int i = a; i < b; ++i) {
            const double *o = part + (size_t)i * 8;
            const u64 lo = __ldcg((const u64 *)o + 4), hi = __ldcg((const u64 *)o + 5);
            q = mul(Q<double>{__ldcg(o), __ldcg(o + 1), __ldcg(o + 2), __ldcg(o + 3), (u128)hi << 64 | lo}, q);
        }
        U = block_product(q, smd, W);
        if (tid == 0) p.tickets[0] = 0u;  // ready for the next launch
    }
    if (tid != 0) return;
    double sn, cs;
    sincos(angle(U.ph), &sn, &cs);
    // (re + i im) e^{-i ph}
    auto out = [&](int i, double re, double im) {
        const double2 v = make_double2(fma(re, cs, im * sn), fma(im, cs, -re * sn));
        if (p.out_c128) ((double2 *)p.U_out)[i] = v;
        else ((float2 *)p.U_out)[i] = make_float2((float)v.x, (float)v.y);
    };
    out(0, U.a, -U.z);
    if (p.d_out == 2) {
        out(1, -U.y, -U.x);
        out(2, U.y, -U.x);
        out(3, U.a, U.z);
    }
    if (gridDim.x > 1) {
        for (int i = 0; i < 4; ++i) p.counters[4 + i] = atomicExch(&p.counters[i], 0ull);
        p.status[1] = atomicExch(&p.status[0], 0u);
    } else {
        for (int i = 0; i < 4; ++i) p.counters[4 + i] = cnt[i];
        p.status[1] = s_flags;
    }
}

template <typename Real, int INTEG>
cudaError_t launch(const FusedParams &p, int grid, int warps, cudaStream_t st) {
    su2_kernel<Real, INTEG><<<grid, warps * 32, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace su2
}  // namespace pm
