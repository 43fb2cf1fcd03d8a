// m2p.cuh -- the mesh cell and linear FE weights of a particle (eq. m2p), shared by the single-problem
// and batched M2P and its adjoint.
#pragma once

#include "common.cuh"
#include "fix64.cuh"

namespace pfem {

// A particle's cell (i, j), the offset of the node between (i,j) and (i+1,j+1) on its triangle (1 below
// the diagonal, n above) and the weights on (i,j), that node and (i+1,j+1).
template <typename R> struct MeshCell {
    int i, j, mid;
    long long n00;
    R w0, w1, w2;
};

// Half of nc is taken in R: an FP32 particle with the three FP64-pipe instructions of (R)(0.5 * nc)
// held M2P at 41 us for 2048^2 particles of four components (23 without).
template <typename R> __device__ __forceinline__ R local_coord(R x, int i, int nc)
{
    const R xw = x - floor(x);                          // exact
    R s = fma(xw, (R)nc, (R)(-i));
    if (s > (R)0.5 * (R)nc) s -= (R)nc;                  // fixed point rounded up to 2^32 -> cell 0
    return s;
}

// FP64 positions in fixed point (fix64.cuh: their arithmetic would hold the FP64 pipe): the cell, and the
// local coordinate in units of 2^-62 (absolute, where FP64 rounds it to 2^-53 of itself: a weight near
// zero is a multiple of 2^-62).  The cell comes from the coordinate rounded to 2^-32, so the
// local coordinate may lie a rounding outside [0, 1].  Below 2^-12 a position has bits beyond 2^-64, whose
// rounding nc enlarges: with more than 2048 cells a side, where that passes FP64's own rounding, those
// positions, 2^-12 of all, take the FP64 product.
__device__ __forceinline__ bool needs_f64(double x, int nc) { return nc > 2048 && (unsigned)__double2hiint(x) < 1011u << 20; }
static __device__ __noinline__ long long local_f64(double x, int nc, int i)
{
    return __double2ll_rn(fma(x, (double)nc, (double)-i) * 4611686018427387904.0);
}
template <bool FINE = true>
__device__ __forceinline__ long long local_fix(double x, int nc, int &i)
{
    const unsigned long long q = (unsigned long long)fx64(x);
    const unsigned f = (unsigned)q;
    unsigned t = (unsigned)(q >> 32);
    t += f > 0x80000000u || (f == 0x80000000u && (t & 1u)) ? 1u : 0u;
    i = bin_of(t, nc);
    if (FINE && needs_f64(x, nc)) return local_f64(x, nc, i);
    int d = (int)__umul64hi(q, (unsigned long long)nc) - i;
    d -= d > 1 ? nc : 0;
    d += d < -1 ? nc : 0;
    return (long long)((q * (unsigned long long)nc) >> 2) + ((long long)d << 62);
}

// x 2^-62 as a double
__device__ __forceinline__ double unit62(long long x)
{
    const double d = __ll2double_rn(x);
    return x == 0 ? 0.0 : __hiloint2double(__double2hiint(d) - (62 << 20), __double2loint(d));
}

// FINE: with the product of needs_f64 positions in place (out of line, as are all its uses: predicated, its FP64
// instructions cost M2P of other positions up to a quarter).
template <typename P, typename R, bool FINE = true>
__device__ __forceinline__ MeshCell<R> mesh_cell(P px, P py, int n)
{
    const int nc = n - 1;
    MeshCell<R> c;
    if constexpr (sizeof(P) == 8) {
        const long long s = local_fix<FINE>(px, nc, c.i), t = local_fix<FINE>(py, nc, c.j);
        const long long hi = max(s, t), lo = min(s, t);
        c.mid = s >= t ? 1 : n;
        c.w0 = (R)unit62((1ll << 62) - hi);
        c.w1 = (R)unit62(hi - lo);
        c.w2 = (R)unit62(lo);
        if (!is_finite_bits(px) || !is_finite_bits(py)) c.w0 = c.w1 = c.w2 = (R)__longlong_as_double(0x7ff8000000000000LL);
    } else {
        c.i = bin_of(fx_of(px), nc);
        c.j = bin_of(fx_of(py), nc);
        const P s = local_coord<P>(px, c.i, nc), t = local_coord<P>(py, c.j, nc);
        const P hi = s >= t ? s : t, lo = s >= t ? t : s;
        c.mid = s >= t ? 1 : n;
        c.w0 = R(P(1) - hi);
        c.w1 = R(hi - lo);
        c.w2 = R(lo);
    }
    c.n00 = (long long)c.j * n + c.i;
    return c;
}

// The cell alone; returns whether the particle lies on or below its diagonal (s >= t).
template <typename P>
__device__ __forceinline__ bool cell_index(P px, P py, int nc, int &i, int &j)
{
    if constexpr (sizeof(P) == 8) {
        const long long s = local_fix(px, nc, i), t = local_fix(py, nc, j);
        return s >= t;
    } else {
        i = bin_of(fx_of(px), nc);
        j = bin_of(fx_of(py), nc);
        return local_coord<P>(px, i, nc) >= local_coord<P>(py, j, nc);
    }
}

// M2P of the particles m0 + 256 u < end, u < U, on a mesh of n nodes per side; CT components, or C with
// CT = 0; FINE: n may be above 2049.
template <typename P, typename V, typename R, int CT, int U, bool FINE = true>
__device__ __forceinline__ void m2p_particles(int n, long long m0, long long end, const P *__restrict__ pos,
                                              int Crt, const V *__restrict__ mesh, V *__restrict__ vals)
{
    const int C = CT > 0 ? CT : Crt;
    MeshCell<R> cell[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const long long m = min(m0 + 256 * u, end - 1);
        P px, py;
        load_pos(pos, m, px, py);
        cell[u] = mesh_cell<P, R, false>(px, py, n);
    }
    if constexpr (sizeof(P) == 8 && FINE)
        if (n > 2049)                            // again, where a coordinate needs the product
#pragma unroll
            for (int u = 0; u < U; ++u) {
                P px, py;
                load_pos(pos, min(m0 + 256 * u, end - 1), px, py);
                if (needs_f64(px, n - 1) || needs_f64(py, n - 1)) cell[u] = mesh_cell<P, R>(px, py, n);
            }
    if constexpr (CT == 4 && sizeof(V) == 4 && sizeof(R) == 4) {
        float4 a[U], b[U], c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4 *p = reinterpret_cast<const float4 *>(mesh) + cell[u].n00;
            a[u] = __ldg(p);
            b[u] = __ldg(p + cell[u].mid);
            c[u] = __ldg(p + n + 1);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const R w0 = cell[u].w0, w1 = cell[u].w1, w2 = cell[u].w2;
            float4 o;
            o.x = fmaf(w0, a[u].x, fmaf(w1, b[u].x, w2 * c[u].x));
            o.y = fmaf(w0, a[u].y, fmaf(w1, b[u].y, w2 * c[u].y));
            o.z = fmaf(w0, a[u].z, fmaf(w1, b[u].z, w2 * c[u].z));
            o.w = fmaf(w0, a[u].w, fmaf(w1, b[u].w, w2 * c[u].w));
            if (m0 + 256 * u < end) __stcs(reinterpret_cast<float4 *>(vals) + m0 + 256 * u, o);
        }
    } else if constexpr (CT > 0) {
        R a[U][CT], b[U][CT], c[U][CT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const V *p = mesh + cell[u].n00 * CT;
#pragma unroll
            for (int k = 0; k < CT; ++k) {
                a[u][k] = load_val<V, R>(p + k);
                b[u][k] = load_val<V, R>(p + cell[u].mid * CT + k);
                c[u][k] = load_val<V, R>(p + (n + 1) * CT + k);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < CT; ++k) {
                const R v = cell[u].w0 * a[u][k] + cell[u].w1 * b[u][k] + cell[u].w2 * c[u][k];
                if (m0 + 256 * u < end) store_val<V, R>(vals + (m0 + 256 * u) * CT + k, v);
            }
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const V *p = mesh + cell[u].n00 * C;
            if (m0 + 256 * u < end)
                for (int k = 0; k < C; ++k)
                    store_val<V, R>(vals + (m0 + 256 * u) * C + k,
                                    cell[u].w0 * load_val<V, R>(p + k) +
                                        cell[u].w1 * load_val<V, R>(p + (long long)cell[u].mid * C + k) +
                                        cell[u].w2 * load_val<V, R>(p + (long long)(n + 1) * C + k));
        }
    }
}

}  // namespace pfem
