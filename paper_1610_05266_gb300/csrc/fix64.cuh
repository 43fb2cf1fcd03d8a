// fix64.cuh -- the FP64 moment solve of the table path without the FP64 pipe.
//
// An SM of GB300 issues two FP64 instructions a clock, so a warp's FP64 instruction takes its
// scheduler 64 cycles; assembling, factoring and solving the three 6 x 6 systems of a node in FP64
// took about 2600 of them.  Here each edge system is factored in FP32 and its solution y
// refined in 64-bit fixed point: residuals r = b - M y on the integer pipes, corrections through the
// FP32 factor, each step gaining the bits that FP32 has over the system's condition (on jittered
// lattices two steps, at about 100 integer instructions a stencil point).  Positions enter as 64-bit
// fixed point too: an offset between two of them is exact where FP64 rounds it.
//
// Scaling, all by powers of two: coordinates X in Q64, |X| < 1/2, from the largest of the
// stencil; y'_k = y_k g^deg(k) and b' likewise, as integers with unit 2^-s, |y'|, |b'| <= 2^(60 - s); t
// = p . y in the same unit, |t| <= 2.75 of the largest |y'|.  A product is rounded within 1.5 units.
// t itself is the coefficient A, which on irregular stencils is far below |y'| (an edge short beside
// its stencil, particles close together): it is shifted up by its headroom of 2^h before X t, Y t
// and the sums are formed, so that their rounding, which the inverse of M enlarges, is in units of
// 2^-(s + h) (the rounding of t is not enlarged: P^T M^-1 P is a projection).  The sums may wrap:
// the residual itself is small.
//
// Error of the coefficients against 128-bit arithmetic, the largest of an edge over its largest
// coefficient; the FP64 Cholesky of the same edges in brackets:
//   lattice, jitter 0.3, 504,000 edges   median 4e-17 (8e-16), 99.9 % 7e-16 (4e-15), worst 8e-15 (1e-14)
//   uniform random, 504,000 edges        median 2e-16 (1e-15), 99.9 % 1e-14 (2e-14), worst 2e-13 (8e-13)
// Before the shift by h, with a stalled refinement accepted at 2^-36 of the largest |y'|, the uniform
// random set's were 7e-16, 6e-14 and 2e-11.
//
// Measured (round trip, FP64 values; FP64 systems before): 513^2 nodes / 1024^2 particles 1798 -> 624 us,
// 33^2 / 64^2 200 -> 89 us with four lanes a node; the mesh's error against 64-bit arithmetic 2.6e-16 ->
// 1.6e-16 of its 2-norm.
#pragma once

#include "moments.cuh"

namespace pfem {

// x mod 1 in Q64 (rounded to nearest below 2^-12, exact above), by integer operations.
__device__ __forceinline__ long long fx64(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff, s = e - 1011;
    const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
    unsigned long long q = 0;
    if (s >= 0) q = s < 64 ? m << s : 0ull;
    else if (s > -54) q = (m + (1ull << (-s - 1))) >> -s;
    return (long long)((b >> 63) ? 0ull - q : q);
}
__device__ __forceinline__ long long fx64(float x)
{
    const unsigned b = __float_as_uint(x);
    const int e = (int)(b >> 23) & 0xff, s = e - 86;
    const unsigned long long m = (b & 0x7fffffu) | (e ? 1u << 23 : 0u);
    unsigned long long q = 0;
    if (s >= 0) q = s < 64 ? m << s : 0ull;
    else if (s > -25) q = (m + (1ull << (-s - 1))) >> -s;
    return (long long)((b >> 31) ? 0ull - q : q);
}

__device__ __forceinline__ bool is_finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool is_finite_bits(float x) { return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u; }

// I / nc in Q64, rounded to nearest (0 <= I < nc < 2^31).
__device__ __forceinline__ long long node_fx64(int I, int nc)
{
    const unsigned long long d = (unsigned long long)nc, a = (unsigned long long)I << 32;
    const unsigned long long h = a / d, r = (a - h * d) << 32, l = r / d, r2 = r - l * d;
    return (long long)((h << 32) + l + (2 * r2 >= d ? 1 : 0));
}

// A 64-bit integer as h 2^32 + l with both parts signed.
struct Split64 {
    int h, l;
};
__device__ __forceinline__ Split64 split64(long long u)
{
    const int l = (int)u;
    return {(int)(u >> 32) + (int)((unsigned)l >> 31), l};
}
// a b / 2^64 within 1.5 (|a| < 2^63 - 2^31, |b| < 2^62)
__device__ __forceinline__ long long mul64(Split64 a, Split64 b)
{
    return (long long)a.h * b.h + (long long)(__mulhi(a.h, b.l) + __mulhi(a.l, b.h) + 1);
}

struct EdgeFix64 {
    Split64 Y[6];
    long long Y0, Y1, Y2;

    __device__ __forceinline__ void set(const long long y[6])
    {
        Y0 = y[0];
        Y1 = y[1];
        Y2 = y[2];
#pragma unroll
        for (int k = 3; k < 6; ++k) Y[k] = split64(y[k]);
    }
    // t = p . y at (X, Z)
    __device__ __forceinline__ long long value(Split64 X, Split64 Z) const
    {
        const Split64 u = split64(Y1 + mul64(X, Y[3]) + mul64(Z, Y[4]));
        const Split64 v = split64(Y2 + mul64(Z, Y[5]));
        return Y0 + mul64(X, u) + mul64(Z, v);
    }
    // r -= p (p . y) 2^h; tm: the largest upper half of |p . y|
    __device__ __forceinline__ void residual(Split64 X, Split64 Z, int h, long long r[6], int &tm) const
    {
        long long t = value(X, Z);
        const int top = (int)(t >> 32);
        tm = max(tm, top ^ (top >> 31));
        t <<= h;
        const Split64 ts = split64(t);
        const long long xt = mul64(X, ts), zt = mul64(Z, ts);
        const Split64 xs = split64(xt), zs = split64(zt);
        r[0] -= t;
        r[1] -= xt;
        r[2] -= zt;
        r[3] -= mul64(X, xs);
        r[4] -= mul64(Z, xs);
        r[5] -= mul64(Z, zs);
    }
};

// Offsets of a node's particles from it in fixed point, scaled up by a common power of two 2^L so
// that every |offset| < 2^60: o[0..nu) in Q64.  Returns L, or NOT_FINITE when a position is not.
constexpr int NOT_FINITE = -1000;
template <typename P, int UM, typename Slots>
__device__ __forceinline__ int node_offsets64(const void *pos, int Iu, int Ju, int nc, Slots &&us,
                                               int nu, longlong2 (&o)[UM])
{
    const long long nx = node_fx64(Iu, nc), ny = node_fx64(Ju, nc);
    unsigned long long m = 0;
    bool bad = false;
    for (int i = 0; i < nu; ++i) {
        P px, py;
        load_pos((const P *)pos, us[i], px, py);
        bad |= !is_finite_bits(px) || !is_finite_bits(py);     // no second way out of the loop: the warp
                                                              // would not come together after it
        const long long x = fx64(px) - nx, y = fx64(py) - ny;
        m |= (unsigned long long)(x ^ (x >> 63)) | (unsigned long long)(y ^ (y >> 63));
        o[i] = make_longlong2(x, y);
    }
    const int L = __clzll((long long)m) - 4;
    for (int i = 0; i < nu; ++i) {
        if (L >= 0) o[i] = make_longlong2(o[i].x << L, o[i].y << L);
        else o[i] = make_longlong2(o[i].x >> -L, o[i].y >> -L);
    }
    return bad ? NOT_FINITE : L;
}

// One edge's system over the particles of `mask`: its FP32 factor, the units of the fixed point and the
// refinement of a solution.  Coordinates are about the edge's midpoint, doubled: x = X 2^-63 in FP32, X'
// = X 2^(k - 64) in fixed point, so X' = x 2^(k - 1).
template <int UM> struct EdgeSystem {
    const longlong2 (&o)[UM];
    unsigned mask;
    long long mx, my, dx, dy;           // midpoint doubled; half the edge = X of its first end
    int k;
    float ex, ey;                       // the edge in FP32 units
    float c1;                           // 2^(1 - k)
    Moment<float> M;

    static __device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }

    __device__ __forceinline__ EdgeSystem(const longlong2 (&off)[UM], unsigned m, longlong2 on, longlong2 os)
        : o(off), mask(m), mx(on.x + os.x), my(on.y + os.y), dx(on.x - os.x), dy(on.y - os.y)
    {
    }

    // Assemble and factor; false when a pivot is below `least` of the trace.
    __device__ __forceinline__ bool factor(float least)
    {
        M.zero();
        int hm = 0;
        for (unsigned m = mask; m; m &= m - 1) {
            const longlong2 p = o[__ffs(m) - 1];
            const int hx = (int)((2 * p.x - mx) >> 32), hy = (int)((2 * p.y - my) >> 32);
            hm = max(hm, max(hx ^ (hx >> 31), hy ^ (hy >> 31)));
            M.add((float)hx * 4.656612873077393e-10f, (float)hy * 4.656612873077393e-10f);
        }
        ex = (float)dx * 2.168404344971009e-19f;
        ey = (float)dy * 2.168404344971009e-19f;
        const float l2 = fmaf(ex, ex, ey * ey);
        // the tolerance of the system scaled by the edge length: pivots of degree d carry l^2d
        const float i2 = 1.f / l2, i4 = i2 * i2;
        const float tol = least *
                          (M.m[tri_ix(0, 0)] + (M.m[tri_ix(1, 1)] + M.m[tri_ix(2, 2)]) * i2 +
                           (M.m[tri_ix(3, 3)] + M.m[tri_ix(4, 4)] + M.m[tri_ix(5, 5)]) * i4);
        const float t1 = tol * l2, t2 = t1 * l2;
        const float tols[6] = {tol, t1, t1, t2, t2, t2};
        // k: the left shift that brings the largest coordinate up to a half in Q64
        k = __clz(hm + 1) - 1;
        c1 = pow2(1 - k);
        return M.factor_tol(tols) && k <= 20;
    }

    // factor of degree deg(q) from FP32 to fixed-point units of a solution
    __device__ __forceinline__ float unit(int q) const { return q == 0 ? 1.f : q < 3 ? c1 : c1 * c1; }

    __device__ __forceinline__ void coords(int i, Split64 &X, Split64 &Z) const
    {
        const longlong2 p = o[i];
        X = split64((2 * p.x - mx) << k);
        Z = split64((2 * p.y - my) << k);
    }

    // The unit 2^-s of a solution y (FP32 units) with right-hand side b (fixed-point units): |y'|, |b'| <=
    // 2^(60 - s), at least 2^-most; false when it would be above 2^-20.  ym: the largest of them.
    __device__ __forceinline__ bool range(const float y[6], const float b[6], int most, int &s, float &ym) const
    {
        ym = 0.f;
#pragma unroll
        for (int q = 0; q < 6; ++q) ym = fmaxf(ym, fmaxf(fabsf(y[q] * unit(q)), fabsf(b[q])));
        s = min(186 - (int)(__float_as_uint(ym) >> 23), most);
        return s >= 20;
    }

    // Y = y in units 2^-s, refined until M' Y = B.  ym: the largest of |y|; ref: a value that the
    // largest |p . y| is not to be taken below.  False when that is not reached.
    //
    // A step's correction d shrinks by about its ratio to the one before, so the next one is expected at
    // d^2 / last.  It is left out when it is below 2^-51 (top / ym), top the largest |p . y|: where y
    // is large beside its values the ratios are uneven.  A correction that shrinks no more is the floor
    // that the residual's rounding sets.  It is accepted where the values it changes, whose 2-norm is
    // the root of d . r (r = M d), stay below 2^-50 of top; else the system is left to FP64, which takes 0.1 % of the
    // edges of a uniform random set and none of a jittered lattice's.
    __device__ __forceinline__ bool refine(const float y[6], int s, float ym, float ref, const long long B[6],
                                           long long Y[6]) const
    {
        const float us = pow2(-s), sc = pow2(s - 60);
#pragma unroll
        for (int q = 0; q < 6; ++q) Y[q] = __float2ll_rn(y[q] * unit(q) * sc * 1152921504606846976.0f);
        EdgeFix64 E;
        float last = ym;                 // the correction before
        int h = 0;                       // headroom of t in the pass before, less a bit for its change
        for (int it = 0; it < 12; ++it) {
            E.set(Y);
            long long r[6];
            int tm = 0;
#pragma unroll
            for (int q = 0; q < 6; ++q) r[q] = B[q] << h;
            for (unsigned m = mask; m; m &= m - 1) {
                Split64 X, Z;
                coords(__ffs(m) - 1, X, Z);
                E.residual(X, Z, h, r, tm);
            }
            const float uh = us * pow2(-h), top = fmaxf(((float)tm + 1.f) * pow2(32 - s), ref);
            float rf[6], d[6], dm = 0.f, v2 = 0.f;
#pragma unroll
            for (int q = 0; q < 6; ++q) rf[q] = __ll2float_rn(r[q]) * uh * unit(q);
            M.solve(rf, d);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                v2 = fmaf(d[q], rf[q], v2);
                d[q] *= unit(q);
                dm = fmaxf(dm, fabsf(d[q]));
                Y[q] += __float2ll_rn(d[q] * sc * 1152921504606846976.0f);
            }
            // (the first pass has no headroom yet; a t that has outgrown it has spoilt the sums)
            if (it > 0 && tm < 1 << (29 - h)) {
                if (dm <= 1.1102230246251565e-16f * top ||
                    dm * dm * ym <= 4.440892098500626e-16f * last * top * top)
                    return true;
                if (dm > 0.25f * last) return fabsf(v2) <= 7.888609052210118e-31f * top * top;
            }
            h = min(max(__clz((int)((unsigned)tm + 1u)) - 4, 0), 16);
            last = dm;
        }
        return false;
    }

    // y of the coefficients: b = -(1/2) (ex^2, ex ey, ey^2) in the quadratic rows.
    __device__ __forceinline__ bool solve_coefficients(long long Y[6], int &s) const
    {
        const float b[6] = {0.f, 0.f, 0.f, -0.5f * ex * ex, -0.5f * ex * ey, -0.5f * ey * ey};
        float y[6];
        M.solve(b, y);
        const float ic2 = 1.f / (c1 * c1);
        const float bf[6] = {0.f, 0.f, 0.f, b[3] * ic2, b[4] * ic2, b[5] * ic2};
        float ym;
        if (!range(y, bf, 62, s, ym)) return false;
        const long long xn = dx << k, yn = dy << k;              // X' of the first end; b' = -2 (X'^2, X'Y', Y'^2)
        const long long half = 1ll << (62 - s);
        const long long B[6] = {0, 0, 0, -((__mul64hi(xn, xn) + half) >> (63 - s)),
                                -((__mul64hi(xn, yn) + half) >> (63 - s)),
                                -((__mul64hi(yn, yn) + half) >> (63 - s))};
        return refine(y, s, ym, 0.f, B, Y);
    }

    // z with M z = u, u' in units 2^-56 (|u'| < 2^7): the adjoint's right-hand side, formed of values whose
    // largest is 1/2 to 1.
    __device__ __forceinline__ bool solve_adjoint(const long long u[6], long long Z[6], int &s) const
    {
        float uf[6], ux[6], z[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            uf[q] = __ll2float_rn(u[q]) * 1.3877787807814457e-17f;
            ux[q] = uf[q] * unit(q);
        }
        M.solve(ux, z);
        float zm;
        if (!range(z, uf, 110, s, zm)) return false;
        long long B[6];
#pragma unroll
        for (int q = 0; q < 6; ++q)
            B[q] = s >= 56 ? u[q] << (s - 56) : (u[q] + (1ll << (55 - s))) >> (56 - s);
        return refine(z, s, zm, 0.5f, B, Z);
    }
};

// Pivot tolerance of a system whose solution is refined.  The refinement finds out for itself where
// the FP32 factor cannot carry it, so the line lies a decade below the FP32 solve's: at 3e-5 470 of
// 504,000 edges of a uniform random set are left to FP64, at 3e-4 1161, at 3e-6 371, and the largest
// error of those solved here is 1.8e-13 each time.  The adjoint keeps the FP32 solve's line: its
// nodes beyond that take FP64's Cholesky form (k_bwd_fix).
constexpr float TOL_FIX64 = 3e-5f;

// Weights of the quadratic part in fixed point: w[i] += 2 lambda_nu lambda_sg A_{i e} / unit over the
// edges e0 <= e < e1.  The unit is 2^-56 of the node's largest coefficient 2 lambda lambda' or less: a
// node close to a particle, or to an edge, has small ones, and its weights keep FP64's relative
// accuracy.  Returns 0, or -PFEM_DEFER for a system below the tolerance, whose refinement stalls, or
// beyond the fixed-point range, a coefficient of 2 or more (a node outside its triangle by the rounding
// of a sliver) among them.
constexpr int W64_SHIFT = 56;            // weights up to 2^7 of the largest coefficient
constexpr double W64_UNIT = 1.3877787807814457e-17;
template <int UM>
__device__ __forceinline__ int node_solve64(const longlong2 (&o)[UM], const unsigned vm[3],
                                            const int vi[3], const double lam[3], int e0, int e1,
                                            long long *w, double &unit, int defer)
{
    const double coef[3] = {2.0 * lam[0] * lam[1], 2.0 * lam[1] * lam[2], 2.0 * lam[2] * lam[0]};
    // 2^up: the largest of |coef| lies in [1/2, 1) 2^-up (zero: any)
    const int up = min(1022 - max(max((__double2hiint(coef[0]) >> 20) & 0x7ff, (__double2hiint(coef[1]) >> 20) & 0x7ff),
                                  (__double2hiint(coef[2]) >> 20) & 0x7ff), 100);
    if (up < -1) return defer;
    unit = __hiloint2double((1023 - W64_SHIFT - up) << 20, 0);
    const double to61 = __hiloint2double((1023 + 61 + up) << 20, 0);
#pragma unroll 1
    for (int e = e0; e < e1; ++e) {
        const int f = e == 2 ? 0 : e + 1;
        EdgeSystem<UM> sys(o, vm[e] | vm[f], o[vi[e]], o[vi[f]]);
        long long Y[6];
        int s;
        if (!sys.factor(TOL_FIX64) || !sys.solve_coefficients(Y, s)) return defer;
        EdgeFix64 E;
        E.set(Y);
        const Split64 cf = split64(__double2ll_rn((e == 0 ? coef[0] : e == 1 ? coef[1] : coef[2]) * to61));
        const int sh = W64_SHIFT + 3 - s;                        // product: coef A 2^(s - 3)
        int tm = 0;
        for (unsigned m = sys.mask; m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            Split64 X, Z;
            sys.coords(i, X, Z);
            const long long t = E.value(X, Z);
            const int h = (int)(t >> 32);
            tm = max(tm, h ^ (h >> 31));
            const long long ct = mul64(split64(t), cf);
            w[i] += sh >= 0 ? ct << sh : ct >> -sh;
        }
        // |A| <= (tm + 1) 2^(32 - s), the coefficient 2^-29 of cf.h + 1: keep the weights well inside their
        // range
        if (((float)tm + 1.f) * EdgeSystem<UM>::pow2(32 - s) * (fabsf((float)cf.h) + 1.f) > 30.f * 536870912.f) return defer;
    }
    return 0;
}

}  // namespace pfem
