// moments.cuh -- the per-edge coefficient system of the quadratically consistent shape
// functions (App. B, eqs. A0, A1, condquad; App. A: minimum-norm solution).
//
// For a Delaunay edge e = (nu, sigma) with stencil S_e, the coefficients A_mu (mu in S_e)
// must satisfy sum A = 0, sum r A = 0 and sum r r^T A = -(1/2)(r_nu - r_sigma)(r_nu - r_sigma)^T
// (eq. condquad rewritten with eqs. A0-A1, eq. A2_2).  In coordinates centred at the edge
// midpoint and scaled by the edge length (the solution does not depend on the frame), with
// p_mu = [1, x, y, x^2, xy, y^2], that is P A = b, P = [p_mu] (6 x k), and the minimum-norm
// solution is A_mu = p_mu . y with M y = b, M = sum_mu p_mu p_mu^T (6 x 6, SPD for a stencil
// not on one conic).  M is factorised by an unrolled Cholesky held in registers.
#pragma once

#include "common.cuh"

namespace pfem {

// packed lower triangle of a symmetric 6x6 matrix: (r, c), r >= c
__host__ __device__ constexpr int tri_ix(int r, int c) { return r * (r + 1) / 2 + c; }

template <typename S> struct Moment {
    S m[21];

    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 21; ++i) m[i] = S(0);
    }

    // M += p p^T for p = [1, x, y, x^2, xy, y^2]
    __device__ __forceinline__ void add(S x, S y)
    {
        const S p[6] = {S(1), x, y, x * x, x * y, y * y};
        m[0] += S(1);
#pragma unroll
        for (int r = 1; r < 6; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) m[tri_ix(r, c)] = fma(p[r], p[c], m[tri_ix(r, c)]);
    }

    // In-place Cholesky M = L L^T; returns false when a pivot is not clearly positive
    // (stencil numerically on one conic: the moment system is rank deficient).
    __device__ __forceinline__ bool factor(S rel_tol)
    {
        S tr = S(0);
#pragma unroll
        for (int r = 0; r < 6; ++r) tr += m[tri_ix(r, r)];
        const S tol = rel_tol * tr;
        const S tols[6] = {tol, tol, tol, tol, tol, tol};
        return factor_tol(tols);
    }

    // The same with a tolerance for each pivot.
    __device__ __forceinline__ bool factor_tol(const S tols[6])
    {
        bool ok = true;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            S s = m[tri_ix(j, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) s = fma(-m[tri_ix(j, k)], m[tri_ix(j, k)], s);
            const S tol = tols[j];
            ok &= s > tol;
            const S d = sqrt(s > tol ? s : tol);
            const S inv = S(1) / d;
            m[tri_ix(j, j)] = inv;               // store the reciprocal of the pivot
#pragma unroll
            for (int i = j + 1; i < 6; ++i) {
                S t = m[tri_ix(i, j)];
#pragma unroll
                for (int k = 0; k < j; ++k) t = fma(-m[tri_ix(i, k)], m[tri_ix(j, k)], t);
                m[tri_ix(i, j)] = t * inv;
            }
        }
        return ok;
    }

    // Solve L L^T y = b with the factor from factor().
    __device__ __forceinline__ void solve(const S b[6], S y[6]) const
    {
        S z[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            S t = b[r];
#pragma unroll
            for (int k = 0; k < r; ++k) t = fma(-m[tri_ix(r, k)], z[k], t);
            z[r] = t * m[tri_ix(r, r)];
        }
#pragma unroll
        for (int r = 5; r >= 0; --r) {
            S t = z[r];
#pragma unroll
            for (int k = r + 1; k < 6; ++k) t = fma(-m[tri_ix(k, r)], y[k], t);
            y[r] = t * m[tri_ix(r, r)];
        }
    }
};

// Exact FP32 -> FP64 widening by integer operations on the bit patterns (sign; exponent
// rebiased by 1023 - 127 = 896; the 23 mantissa bits at the top of the 52).  FP32 subnormals
// (below 1.2e-38) become zero.  On sm_103a the format conversion instructions share the
// narrow FP64 pipe, while these run on the integer pipes.
__device__ __forceinline__ double f64_of(float x)
{
    const unsigned u = __float_as_uint(x);
    const unsigned e = (u >> 23) & 0xffu;
    const unsigned sign = u & 0x80000000u;
    const unsigned hi = e ? sign | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu) : sign;
    const unsigned lo = e ? u << 29 : 0u;
    return __hiloint2double((int)hi, (int)lo);
}

// FP64 -> FP32 by truncating the mantissa (relative error below 2^-23), for finite values
// below FP32's largest; magnitudes below FP32's normal range become zero.
__device__ __forceinline__ float f32_trunc(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    const unsigned u = (hi & 0x80000000u) | ((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    return e > 0 ? __uint_as_float(u) : 0.0f;
}

// Refinement of the FP32 moment solve: none, one step with the residual r = b - M y in 64-bit
// fixed point (FixRes), steps until the solution has FP64's accuracy (fix64.cuh), or for an FP64 solve
// one step with the residual in FP64.
enum { REFINE_NONE = 0, REFINE_FIX = 1, REFINE_FIX64 = 2, REFINE_STEP = 3 };

// ----------------------------------------------------------------- fixed-point residual
// The residual r = b - sum_mu p_mu (p_mu . y) of one edge system on the integer pipes.
//
// An SM of GB300 issues two FP64 instructions a clock: one FP64 instruction of a warp holds its
// scheduler's FP64 pipe for 64 cycles, and in FP64 this residual takes 13 of them a stencil point
// and edge (832 cycles).  Here it takes about 45 integer instructions.  Everything is scaled by
// powers of two, so the scaling is exact:
//  - coordinates X = x / g in Q32, |X| < 1/2, g = 2^k from the largest |x|, |y| of the stencil.
//    A coordinate down to 2^-8 of the largest keeps all 24 bits of its FP32 value; smaller ones
//    are rounded at 2^-33 g, far below the rounding of the FP32 offsets themselves;
//  - the solution in the scaled monomials, y'_k = y_k g^deg(k), as 30-bit integers relative to
//    the largest of |y'| and |b'|.  y is an approximate solution: the refinement corrects the
//    one it is given, and rounding it to this grid leaves values that FP32 represents;
//  - t = p . y, X t, Y t and the six sums as 64-bit integers with unit 2^-61 of that largest
//    value.  |t| <= 1 + 2/2 + 3/4 = 2.75 of it, so products do not overflow; the sums may wrap, which
//    two's complement undoes since the residual itself is small (the FP32 Cholesky solve is
//    backward stable).
// A product drops bits below 2^-61, where FP64 rounds t, X t, Y t and every partial sum to 53
// bits, and the sums are exact: measured against 64-bit arithmetic the projection's error is the
// FP64 residual's (see k_p2m_tab).
struct FixRes {
    float sx, gi;               // 2^32 / g and 1 / g
    int bm;                     // biased exponent: |y'|, |b'| < 2^(bm - 126)
    int Y[6];
    long long r[6];

    // 2^e for -126 <= e <= 127
    static __device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }

    // ext: the stencil's largest |x|, |y|; y is rounded to the grid.  False when the system is
    // beyond the scaling's range (extent 2^40 edge lengths and more).
    __device__ __forceinline__ bool init(float ext, const float b[6], float y[6])
    {
        const int be = (int)(__float_as_uint(ext) >> 23);       // ext < 2^(be - 126)
        if (be < 96 || be > 166) return false;
        gi = pow2(125 - be);
        sx = pow2(157 - be);
        const float g = pow2(be - 125), g2 = g * g, gi2 = gi * gi;
        const float s[6] = {1.f, g, g, g2, g2, g2}, si[6] = {1.f, gi, gi, gi2, gi2, gi2};
        float ym = 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) ym = fmaxf(ym, fmaxf(fabsf(y[k] * s[k]), fabsf(b[k] * si[k])));
        bm = (int)(__float_as_uint(ym) >> 23);
        if (bm < 30 || bm > 250) return false;
        const float sy = pow2(155 - bm), us = pow2(bm - 155);
        const float sb = pow2(61), ub = pow2(126 - bm);         // b' 2^(187 - bm)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            Y[k] = __float2int_rn(y[k] * s[k] * sy);            // |Y| <= 2^29
            y[k] = (float)Y[k] * us * si[k];
            r[k] = k < 3 ? 0 : __float2ll_rn(b[k] * si[k] * ub * sb);
        }
        return true;
    }

    // (a * u) >> 32 with u = uh 2^32 + ul, ul signed
    struct Split {
        int h, l;
    };
    static __device__ __forceinline__ Split split(long long u)
    {
        const int l = (int)u;
        return {(int)(u >> 32) + (int)((unsigned)l >> 31), l};
    }
    static __device__ __forceinline__ long long mul(int a, Split u)
    {
        return (long long)a * u.h + __mulhi(a, u.l);
    }

    // r -= p (p . y) for the point at (x, y)
    __device__ __forceinline__ void point(float x, float y)
    {
        const int X = __float2int_rn(x * sx), Z = __float2int_rn(y * sx);
        const Split u = split(((long long)Y[1] << 32) + (long long)X * Y[3] + (long long)Z * Y[4]);
        const Split v = split(((long long)Y[2] << 32) + (long long)Z * Y[5]);
        const long long t = ((long long)Y[0] << 32) + mul(X, u) + mul(Z, v);
        const Split ts = split(t);
        const long long xt = mul(X, ts), zt = mul(Z, ts);
        const Split xs = split(xt), zs = split(zt);
        r[0] -= t;
        r[1] -= xt;
        r[2] -= zt;
        r[3] -= mul(X, xs);
        r[4] -= mul(Z, xs);
        r[5] -= mul(Z, zs);
    }

    // the residual in the edge frame's units
    __device__ __forceinline__ void result(float out[6]) const
    {
        const float g = 1.f / gi, g2 = g * g, u = pow2(bm - 126), w = pow2(-61);
        const float s[6] = {1.f, g, g, g2, g2, g2};
#pragma unroll
        for (int k = 0; k < 6; ++k) out[k] = __ll2float_rn(r[k]) * w * u * s[k];
    }
};

// Pivot tolerance (relative to the trace) of the fused P2M's Cholesky solve, which hands a
// system below it to the FP64 SVD pass: the normal equations square the stencil's condition,
// so a system is solved fast only while that keeps the precision's accuracy.  Jittered lattices
// stay far above both (smallest pivot 3e-3 of the trace at jitter 0.3); on uniform random
// particles about 0.6 % of the nodes fall below the FP32 value.
#ifndef PFEM_FAST_TOL32
#define PFEM_FAST_TOL32 3e-4f
#endif
#ifndef PFEM_FAST_TOL64
#define PFEM_FAST_TOL64 1e-6
#endif
template <typename S> struct FastTol;
template <> struct FastTol<double> { static constexpr double v = PFEM_FAST_TOL64; };
template <> struct FastTol<float> { static constexpr float v = PFEM_FAST_TOL32; };

}  // namespace pfem
