// p2m.cuh -- per-node particle-to-mesh projection (Sec. 2.2 eq. p2m) with linear FE or
// quadratically consistent shape functions (App. B eq. phiquad), one thread per mesh node.
//
// For node r_i in the particle Delaunay triangle T = (a, b, c) with barycentrics lambda, the
// only nonzero linear shape functions are lambda_a, lambda_b, lambda_c, and eq. (phiquad)
// sums A_{mu nu sigma} phi_nu phi_sigma over ordered pairs of distinct, adjacent nu, sigma --
// the three edges of T, each twice.  So
//     w_{i mu} = lambda_mu [mu in T] + sum_{e=(nu,sigma) in T} 2 lambda_nu lambda_sigma A_{mu e},
// and alpha_i = sum_mu w_{i mu} alpha_mu for every field component in one pass.
#pragma once

#include <type_traits>

#include "fix64.cuh"
#include "geom.cuh"
#include "moments.cuh"
#include "startab.cuh"

namespace pfem {

struct P2MArgs {
    int n;                      // mesh nodes per side (image row/column included)
    Bins B;
    int R0;                     // first search radius in bins
    const void *pos;            // [N,2] positions in slot order
    const int *perm;            // slot -> original index, or nullptr (values in slot order)
    const void *vals;           // [N,C]
    int C;
    void *out;                  // [n,n,C] mesh values (apply mode)
    int *w_idx;                 // [n*n, K] (weights mode)
    void *w;                    // [n*n, K]
    int K;
    DevStatus *status;
    // Queue of nodes whose moment system the fast solve could not factor (rank deficient, or
    // too ill-conditioned for its precision), recomputed by k_p2m_fix; capacity 0 = no queue.
    int *defer_count = nullptr;
    long long *defer_list = nullptr;
    int defer_cap = 0;
    // Index of this problem's first node in a batch (0 for one problem): queue entries and
    // error details are node indices of the whole batch.
    long long noff = 0;
    int ucap = PFEM_UMAX;       // distinct particles of one node in the fast pass
};

// node_quadratic's code for "queue this node for the FP64 SVD pass" (not a public status), and
// the marker of a node that was queued.
constexpr int PFEM_DEFER = 64;
constexpr int PFEM_DEFERRED = 1;

// A node whose moment system the fast solve could not factor, or whose search ran out of its
// region (-PFEM_FAR), is queued for the fix pass (FP64, SVD solve, widest search radius) and
// returns PFEM_DEFERRED; with no queue (the fix pass itself, or a workspace without room) it
// becomes PFEM_ERR_DEGENERATE or PFEM_ERR_CAPACITY.
__device__ __forceinline__ int defer_or_error(const P2MArgs &a, int st, long long node)
{
    if (st != -PFEM_DEFER && st != -PFEM_FAR) return st;
    if (a.defer_cap <= 0) return st == -PFEM_FAR ? -PFEM_ERR_CAPACITY : -PFEM_ERR_DEGENERATE;
    const int i = atomicAdd(a.defer_count, 1);
    if (i >= a.defer_cap) return -PFEM_ERR_CAPACITY;
    a.defer_list[i] = node;
    return PFEM_DEFERRED;
}

// A queue that does not hold every node of the mesh (a small workspace, or none) is left to the nodes
// that FP64's own pivot tolerance sends to the SVD: the more that the FP32 factor of the refined
// solve cannot carry (fix64.cuh; 0.3 % of a uniform random set's) would fill it.  Those are solved
// in place by the FP64 Cholesky.
__device__ __forceinline__ bool short_queue(const P2MArgs &a) { return a.defer_cap < (long long)a.n * a.n; }

// Minimum-norm least-squares solution of P A = b (App. A: the SVD with rank detection), for the
// 6 x k matrix P whose columns are the stencil's monomial vectors; pt holds P^T (k rows of 6,
// k <= SVD_ROWS) and is overwritten.  jacobi_svd gives P^T V = W with orthogonal columns
// w_j = sigma_j u_j (left in pt), V orthogonal and sig2[j] = sigma_j^2; then P = V W^T and
// A = sum_j (v_j . b / sigma_j^2) w_j over the singular values above max(k, 6) eps sigma_max
// (smaller ones are rank deficiency).
//
// Steps: a Householder QR P^T = Q [R; 0] (Golub & Van Loan, 5.2), which keeps the singular
// values; one-sided (Hestenes) Jacobi on the 6 x 6 factor R -- plane rotations of pairs of its
// columns until all are mutually orthogonal, accumulated in V, so that R V = W6 -- with R, V and
// the rotations in registers; then W = Q [W6; 0].  The sweeps, the long part, so run on 6 rows
// instead of k.
constexpr int SVD_ROWS = 32;

// Householder QR of pt (k x 6): R (6 x 6; rows past min(k, 6) zero) and the reflections, v_j
// kept in pt[j..k-1][j] with vv[j] = v_j . v_j (0: no reflection).
static __device__ __forceinline__ void householder_qr(int k, double (*pt)[6], double R[6][6],
                                                      double vv[6])
{
    const int m = k < 6 ? k : 6;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < 6; ++j) R[i][j] = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        vv[j] = 0.0;
        if (j >= m) continue;
        double nx = 0.0;
        for (int i = j; i < k; ++i) nx = fma(pt[i][j], pt[i][j], nx);
        const double x0 = pt[j][j];
        const double alpha = x0 >= 0.0 ? -sqrt(nx) : sqrt(nx);
        if (nx > 0.0) {
            pt[j][j] = x0 - alpha;
            vv[j] = 2.0 * (nx + fabs(x0) * sqrt(nx));     // v.v = 2 (|x|^2 - alpha x0)
#pragma unroll
            for (int c = j + 1; c < 6; ++c) {
                double d = 0.0;
                for (int i = j; i < k; ++i) d = fma(pt[i][j], pt[i][c], d);
                const double f = 2.0 * d / vv[j];
                for (int i = j; i < k; ++i) pt[i][c] = fma(-f, pt[i][j], pt[i][c]);
            }
        }
        R[j][j] = nx > 0.0 ? alpha : x0;
#pragma unroll
        for (int c = j + 1; c < 6; ++c) R[j][c] = pt[j][c];
    }
}

// out[0..k) = Q [y; 0] = H_0 H_1 ... H_5 [y; 0] with the reflections of householder_qr.
static __device__ __forceinline__ void apply_q(int k, const double (*pt)[6], const double vv[6],
                                               const double y[6], double *out)
{
    for (int i = 0; i < k; ++i) out[i] = i < 6 ? y[i] : 0.0;
#pragma unroll
    for (int j = 5; j >= 0; --j) {
        if (vv[j] == 0.0) continue;
        double d = 0.0;
        for (int i = j; i < k; ++i) d = fma(pt[i][j], out[i], d);
        const double f = 2.0 * d / vv[j];
        for (int i = j; i < k; ++i) out[i] = fma(-f, pt[i][j], out[i]);
    }
}

// One-sided (Hestenes) Jacobi on R (6 x 6): plane rotations of pairs of its columns until all
// are mutually orthogonal, accumulated in V, so that R V = W6 (left in R), sig2[j] = |w6_j|^2.
//  - Each sweep takes the 15 column pairs in the round-robin order of 5 rounds of 3 disjoint
//    pairs, so that three rotations are independent.
//  - A rotation's tangent comes from FP32 arithmetic: any exact rotation keeps the singular
//    values, and its angle only sets how fast the off-diagonal products fall.  c = 1/sqrt(1+t^2)
//    and s = c t are formed in FP64 from that t, so the rotation is orthogonal to FP64
//    precision.  (FP64 divides and square roots are long instruction sequences on the narrow
//    FP64 pipe.)
//  - Columns whose squared norm is below 1e-31 of ||R||_F^2 are left alone: the rank detection
//    drops them (its threshold is above (6 eps)^2 sigma_max^2 >= 1.7e-30 ||R||_F^2 / 6), and their
//    rounding noise would otherwise keep a sweep from converging.
static __device__ __forceinline__ void jacobi6(double R[6][6], double V[6][6], double sig2[6])
{
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < 6; ++j) V[i][j] = i == j ? 1.0 : 0.0;
    double f2 = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < 6; ++j) f2 = fma(R[i][j], R[i][j], f2);
    const double tiny2 = 1e-31 * f2;
    constexpr int RR[5][3][2] = {{{0, 1}, {2, 3}, {4, 5}}, {{0, 2}, {1, 4}, {3, 5}},
                                 {{0, 3}, {1, 5}, {2, 4}}, {{0, 4}, {1, 3}, {2, 5}},
                                 {{0, 5}, {1, 2}, {3, 4}}};
    for (int sweep = 0; sweep < 40; ++sweep) {
        bool rotated = false;
#pragma unroll
        for (int r = 0; r < 5; ++r) {
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                const int p = RR[r][h][0], q = RR[r][h][1];
                double al = 0.0, be = 0.0, ga = 0.0;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    al = fma(R[i][p], R[i][p], al);
                    be = fma(R[i][q], R[i][q], be);
                    ga = fma(R[i][p], R[i][q], ga);
                }
                if (!(ga * ga > 1e-30 * al * be) || al < tiny2 || be < tiny2) continue;
                // tangent of the rotation angle: zeta = (be - al) / (2 ga), in FP32 while the
                // operands are well inside its range (near-coincident particles can make the
                // scaled monomials huge), else in FP64
                double t;
                const double dba = be - al;
                // binary exponents from the bit patterns (integer pipes): |dba| < 2^96 and
                // 2^-95 <= |ga| < 2^96
                const int ed = (__double2hiint(dba) >> 20) & 0x7ff, eg = (__double2hiint(ga) >> 20) & 0x7ff;
                if (ed < 1023 + 96 && eg > 1023 - 96 && eg < 1023 + 96) {
                    const float gf = f32_trunc(ga), df = f32_trunc(dba);
                    const float zf = df / (2.f * gf);
                    const float tf = copysignf(1.f, zf) / (fabsf(zf) + sqrtf(fmaf(zf, zf, 1.f)));
                    if (!(tf != 0.f)) continue; // |zeta| beyond 1e19: the angle is below FP64's
                    t = f64_of(tf);
                } else {
                    const double zeta = dba / (2.0 * ga);
                    t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
                    if (!(t != 0.0)) continue;
                }
                rotated = true;
                const double c = rsqrt(fma(t, t, 1.0)), s = c * t;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const double x = R[i][p], y = R[i][q];
                    R[i][p] = fma(c, x, -s * y);
                    R[i][q] = fma(s, x, c * y);
                    const double u = V[i][p], w = V[i][q];
                    V[i][p] = fma(c, u, -s * w);
                    V[i][q] = fma(s, u, c * w);
                }
            }
        }
        if (!rotated) break;
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double s2 = 0.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) s2 = fma(R[i][j], R[i][j], s2);
        sig2[j] = s2;
    }
}

// The SVD P^T V = W of the k x 6 matrix in pt (overwritten with W): householder_qr, jacobi6 on
// R, then W = Q [W6; 0].
static __device__ __forceinline__ void jacobi_svd(int k, double (*pt)[6], double V[6][6],
                                                  double sig2[6])
{
    double R[6][6], vv[6];
    householder_qr(k, pt, R, vv);
    jacobi6(R, V, sig2);
    double W[SVD_ROWS][6];
    for (int i = 0; i < k; ++i)
#pragma unroll
        for (int c = 0; c < 6; ++c) W[i][c] = i < 6 ? R[i][c] : 0.0;
#pragma unroll
    for (int j = 5; j >= 0; --j) {
        if (vv[j] == 0.0) continue;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            double d = 0.0;
            for (int i = j; i < k; ++i) d = fma(pt[i][j], W[i][c], d);
            const double f = 2.0 * d / vv[j];
            for (int i = j; i < k; ++i) W[i][c] = fma(-f, pt[i][j], W[i][c]);
        }
    }
    for (int i = 0; i < k; ++i)
#pragma unroll
        for (int c = 0; c < 6; ++c) pt[i][c] = W[i][c];
}

// Squared singular values kept by the rank detection: above (max(k, 6) eps)^2 sigma_max^2.
__device__ __forceinline__ double svd_threshold2(int k, const double sig2[6])
{
    double smax2 = 0.0;
    for (int j = 0; j < 6; ++j) smax2 = fmax(smax2, sig2[j]);
    const double tol = (double)(k > 6 ? k : 6) * 2.220446049250313e-16;
    return tol * tol * smax2;
}

static __device__ __noinline__ void minnorm_lsq(int k, double (*pt)[6], const double b[6],
                                                double *A)
{
    // A = sum_j (v_j . b / sigma_j^2) w_j = Q [sum_j (v_j . b / sigma_j^2) w6_j; 0]
    double R[6][6], vv[6], V[6][6], sig2[6];
    householder_qr(k, pt, R, vv);
    jacobi6(R, V, sig2);
    const double thr2 = svd_threshold2(k, sig2);
    double z[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        if (!(sig2[j] > thr2)) continue;
        double d = 0.0;
#pragma unroll
        for (int r = 0; r < 6; ++r) d = fma(V[r][j], b[r], d);
        const double cj = d / sig2[j];
#pragma unroll
        for (int i = 0; i < 6; ++i) z[i] = fma(cj, R[i][j], z[i]);
    }
    apply_q(k, pt, vv, z, A);
}

// Node position and minimal-image offsets in the compute precision R.
template <typename P, typename R> struct NodePos;

template <> struct NodePos<double, double> {
    double x, y;
    __device__ __forceinline__ void init(int Iu, int Ju, int nc)
    {
        x = (double)Iu / (double)nc;
        y = (double)Ju / (double)nc;
    }
    __device__ __forceinline__ void off(const void *pos, int s, double &dx, double &dy) const
    {
        double px, py;
        load_pos((const double *)pos, s, px, py);
        dx = wrap1(px - x);
        dy = wrap1(py - y);
    }
};

// FP32 offsets: the node coordinate I/nc is carried as hi + lo, so that an offset is accurate
// to FP32 relative precision (px - hi is exact for nearby values, and wraps exactly).
template <> struct NodePos<float, float> {
    float xh, xl, yh, yl;
    __device__ __forceinline__ void init(int Iu, int Ju, int nc)
    {
        const float f = (float)nc;
        xh = (float)Iu / f;
        xl = fmaf(-xh, f, (float)Iu) / f;
        yh = (float)Ju / f;
        yl = fmaf(-yh, f, (float)Ju) / f;
    }
    __device__ __forceinline__ void off(const void *pos, int s, float &dx, float &dy) const
    {
        float px, py;
        load_pos((const float *)pos, s, px, py);
        dx = wrap1(px - xh) - xl;
        dy = wrap1(py - yh) - yl;
    }
};

template <typename V, typename R>
__device__ __forceinline__ void load_vals(const V *vals, const int *perm, int s, int C, R out[8])
{
    const long long idx = perm ? (long long)__ldg(perm + s) : (long long)s;
    const V *p = vals + idx * C;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c < C) out[c] = load_val<V, R>(p + c);
}

template <>
__device__ __forceinline__ void load_vals<float, float>(const float *vals, const int *perm, int s,
                                                        int C, float out[8])
{
    const long long idx = perm ? (long long)__ldg(perm + s) : (long long)s;
    if (C == 4 && (reinterpret_cast<uintptr_t>(vals) & 15) == 0) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(vals) + idx);
        out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
        return;
    }
    const float *p = vals + idx * C;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c < C) out[c] = __ldg(p + c);
}

template <typename V, typename R>
__device__ __forceinline__ void store_vals(V *out, long long node, int C, const R acc[8])
{
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c < C) store_val<V, R>(out + node * C + c, acc[c]);
}

template <>
__device__ __forceinline__ void store_vals<float, float>(float *out, long long node, int C,
                                                        const float acc[8])
{
    if (C == 4 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
        reinterpret_cast<float4 *>(out)[node] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        return;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c < C) out[node * C + c] = acc[c];
}

// Quadratic weights of one node over its distinct particles U = T + stars of T's vertices:
// offsets are loaded once per particle, each edge's stencil is a bit mask over U, and
// w_u = lambda_u [u in T] + sum_e 2 lambda_nu lambda_sg A_{u e} accumulates per particle.
// Calls emit(slot, w) once per particle of U.  Returns 0, -PFEM_DEFER (a moment matrix the
// Cholesky solve cannot factor, or more than UMAX distinct particles: queue the node for the
// SVD pass) or, in the SVD pass, -PFEM_ERR_CAPACITY (more than UMAX_SVD distinct particles).
constexpr int UMAX = PFEM_UMAX; // fast pass: jittered lattices have at most about 20
constexpr int UMAX_SVD = 32;   // SVD pass (the stencil masks are 32-bit)
static_assert(UMAX_SVD <= SVD_ROWS, "stencils of the SVD pass fit jacobi_svd's rows");

// SVD = true: the FP64 pass over queued nodes (node_u_fix).
// The node's distinct particles U = T + stars of T's vertices (slots us[0..nu)), the stencil
// of the edge (tri[e], tri[e+1]) as the bit mask vm[e] | vm[e+1] over U, vi[e] the index of
// tri[e] in U, and uw initialised to the linear weights lambda.  Returns 0, or -1 when U has
// more than UM particles.
template <int UM, typename R, typename SA>
__device__ __forceinline__ int node_u_build(const int tri[3], const SA *st, const R lam[3],
                                            int *us, R *uw, int &nu, unsigned vm[3], int vi[3],
                                            int cap = UM)
{
    nu = 0;
    bool over = false;
    auto add = [&](int s) -> int {
        for (int i = 0; i < nu; ++i)
            if (us[i] == s) return i;
        if (nu == cap) { over = true; return 0; }
        us[nu] = s;
        uw[nu] = R(0);
        return nu++;
    };
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        vi[e] = add(tri[e]);
        uw[vi[e]] += lam[e];
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        unsigned m = 1u << vi[e];
        for (int i = 0; i < st[e].n; ++i) m |= 1u << add(st[e][i]);
        vm[e] = m;
    }
    return over ? -1 : 0;
}

// node_u_build without the weights: the particle set and the stencil masks only.
template <int UM, typename SA>
__device__ __forceinline__ int node_u_sets(const int tri[3], const SA *st, int *us, int &nu,
                                           unsigned vm[3], int vi[3], int cap = UM)
{
    nu = 0;
    bool over = false;
    auto add = [&](int s) -> int {
        for (int i = 0; i < nu; ++i)
            if (us[i] == s) return i;
        if (nu == cap) { over = true; return 0; }
        us[nu] = s;
        return nu++;
    };
#pragma unroll
    for (int e = 0; e < 3; ++e) vi[e] = add(tri[e]);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        unsigned m = 1u << vi[e];
        for (int i = 0; i < st[e].n; ++i) m |= 1u << add(st[e][i]);
        vm[e] = m;
    }
    return over ? -1 : 0;
}

// The edge systems e0 <= e < e1 of a node over its particle set: uw[u] += 2 lambda_nu lambda_sg
// A_{u e}, or with RAW (one edge) uw[u] = A_{u e}.
// Returns 0, or -PFEM_DEFER when a moment matrix is below the fast-solve tolerance.
// offset(i, x, y): the offset of particle i from the node.
template <typename R, typename S, int REFINE, bool SVD, int UM, bool RAW, typename W, typename Offset>
__device__ __forceinline__ int node_edges(W &&uw, const unsigned vm[3], const int vi[3], const R lam[3],
                                          int e0, int e1, Offset &&offset)
{
    // The three edges in a loop that is not unrolled: one copy of the edge code keeps the
    // kernels' instruction footprint and register spills down (fused kernel with the refined
    // solve: 1.047 -> 1.010 ms at 1025^2 nodes / 2048^2 particles; spills 164 -> 40 bytes).
#ifndef PFEM_EDGE_UNROLL
#define PFEM_EDGE_UNROLL 1
#endif
    constexpr int edge_unroll = PFEM_EDGE_UNROLL;
#pragma unroll edge_unroll
    for (int e = e0; e < e1; ++e) {
        const int f = e == 2 ? 0 : e + 1;
        const unsigned mask = vm[e] | vm[f];
        S rnx, rny, rsx, rsy;
        offset(vi[e], rnx, rny);
        offset(vi[f], rsx, rsy);
        const S mx = (rnx + rsx) * S(0.5), my = (rny + rsy) * S(0.5);
        const S ex = rnx - rsx, ey = rny - rsy;
        const S inv = S(1) / sqrt(fma(ex, ex, ey * ey));
        if constexpr (SVD) {
            double pt[UM][6];
            int ids[UM];
            int k = 0;
            for (unsigned m = mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                S ox, oy;
                offset(i, ox, oy);
                const double x = (double)((ox - mx) * inv), y = (double)((oy - my) * inv);
                pt[k][0] = 1.0; pt[k][1] = x; pt[k][2] = y;
                pt[k][3] = x * x; pt[k][4] = x * y; pt[k][5] = y * y;
                ids[k++] = i;
            }
            const double tx = (double)(ex * inv), ty = (double)(ey * inv);
            const double b[6] = {0.0, 0.0, 0.0, -0.5 * tx * tx, -0.5 * tx * ty, -0.5 * ty * ty};
            double A[UM];
            minnorm_lsq(k, pt, b, A);
            const double coef = 2.0 * (double)lam[e] * (double)lam[f];
            for (int j = 0; j < k; ++j) uw(ids[j]) += (R)(coef * A[j]);
            continue;
        }
        Moment<S> M;
        M.zero();
        S ext = S(0);                   // largest coordinate, for the residual's scale
        for (unsigned m = mask; m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            S ox, oy;
            offset(i, ox, oy);
            const S x = (ox - mx) * inv, yv = (oy - my) * inv;
            M.add(x, yv);
            if (REFINE == REFINE_FIX) ext = fmax(ext, fmax(fabs(x), fabs(yv)));
        }
        if (!M.factor(FastTol<S>::v)) return -PFEM_DEFER;
        const S tx = ex * inv, ty = ey * inv;
        const S b[6] = {S(0), S(0), S(0), S(-0.5) * tx * tx, S(-0.5) * tx * ty, S(-0.5) * ty * ty};
        S y[6];
        M.solve(b, y);
        if constexpr (REFINE == REFINE_FIX) {
            FixRes fr;
            if (!fr.init(ext, b, y)) return -PFEM_DEFER;
            for (unsigned m = mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                S ox, oy;
                offset(i, ox, oy);
                fr.point((ox - mx) * inv, (oy - my) * inv);
            }
            S rs[6], dy[6];
            fr.result(rs);
            M.solve(rs, dy);
#pragma unroll
            for (int k = 0; k < 6; ++k) y[k] = __fadd_rn(y[k], dy[k]);
        }
        if constexpr (REFINE == REFINE_STEP) {
            // corrected semi-normal equations (Bjorck 1987): with the residual formed from the points
            // the error grows with the condition of P instead of that of M, its square.  504,000
            // edges of a uniform random set: worst 3e-10 of an edge's largest coefficient -> 1e-13.
            S r[6], dy[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) r[k] = b[k];
            for (unsigned m = mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                S ox, oy;
                offset(i, ox, oy);
                const S x = (ox - mx) * inv, z = (oy - my) * inv;
                const S t = fma(z * z, y[5], fma(x * z, y[4], fma(x * x, y[3], fma(z, y[2], fma(x, y[1], y[0])))));
                const S xt = x * t, zt = z * t;
                r[0] -= t;
                r[1] = fma(-x, t, r[1]);
                r[2] = fma(-z, t, r[2]);
                r[3] = fma(-x, xt, r[3]);
                r[4] = fma(-z, xt, r[4]);
                r[5] = fma(-z, zt, r[5]);
            }
            M.solve(r, dy);
#pragma unroll
            for (int k = 0; k < 6; ++k) y[k] += dy[k];
        }
        const R coef = R(2) * lam[e] * lam[f];
        for (unsigned m = mask; m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            S ox, oy;
            offset(i, ox, oy);
            const S x = (ox - mx) * inv, yv = (oy - my) * inv;
            const S A = fma(yv * yv, y[5], fma(x * yv, y[4], fma(x * x, y[3], fma(yv, y[2], fma(x, y[1], y[0])))));
            uw(i) = RAW ? R(A) : fma(coef, R(A), uw(i));
        }
    }
    return 0;
}

// node_edges with offsets re-read from the positions, which neighbouring nodes share in L1.
template <typename P, typename R, typename S, int REFINE, bool SVD, int UM>
__device__ __forceinline__ int node_u_solve(const P2MArgs &a, const NodePos<P, R> &np,
                                            const int *us, R *uw, const unsigned vm[3],
                                            const int vi[3], const R lam[3], int e0 = 0, int e1 = 3)
{
    return node_edges<R, S, REFINE, SVD, UM, false>([&](int i) -> R & { return uw[i]; }, vm, vi, lam, e0, e1, [&](int i, S &x, S &y) {
        R dx, dy;
        np.off(a.pos, us[i], dx, dy);
        x = S(dx);
        y = S(dy);
    });
}

// The edges e0 <= e < e1 of a node of the fix pass in FP64: each by Cholesky down to the FP64 pivot
// tolerance -- a system too ill-conditioned for the FP32 factor is usually well within FP64's -- refined
// where the weights are FP64, and below it (rank deficient, or conditioned beyond it) by the SVD.  A
// system that Cholesky cannot factor adds nothing to uw.
template <typename P, typename R, int UM>
__device__ __forceinline__ void node_u_fix(const P2MArgs &a, const NodePos<P, R> &np, const int *us, R *uw,
                                           const unsigned vm[3], const int vi[3], const R lam[3], int e0, int e1)
{
    constexpr int REFINE = sizeof(R) == 8 ? REFINE_STEP : REFINE_NONE;
#pragma unroll 1
    for (int e = e0; e < e1; ++e)
        if (node_u_solve<P, R, double, REFINE, false, UM>(a, np, us, uw, vm, vi, lam, e, e + 1) != 0)
            node_u_solve<P, R, double, REFINE_NONE, true, UM>(a, np, us, uw, vm, vi, lam, e, e + 1);
}

template <typename P, typename R, typename S, int REFINE, bool SVD = false, typename SA,
          typename Emit>
__device__ __forceinline__ int node_quadratic(const P2MArgs &a, const NodePos<P, R> &np,
                                              const int tri[3], const SA *st, const R lam[3],
                                              Emit &&emit)
{
    constexpr int UM = SVD ? UMAX_SVD : UMAX;
    int us[UM];
    R uw[UM];
    int nu;
    unsigned vm[3];
    int vi[3];
    if (node_u_build<UM>(tri, st, lam, us, uw, nu, vm, vi, SVD ? UM : min(a.ucap, UM)) != 0)
        return SVD ? -PFEM_ERR_CAPACITY : -PFEM_DEFER;
    if constexpr (SVD) {
        node_u_fix<P, R, UM>(a, np, us, uw, vm, vi, lam, 0, 3);
    } else {
        const int r = node_u_solve<P, R, S, REFINE, false, UM>(a, np, us, uw, vm, vi, lam);
        if (r != 0) return r;
    }
    for (int i = 0; i < nu; ++i) emit(us[i], uw[i]);
    return 0;
}

// node_quadratic with the solution refined in 64-bit fixed point (fix64.cuh): calls emit(slot, w) for
// the quadratic part of every particle of U, then for the linear part of the vertices.
template <typename P, typename R, typename SA, typename Emit>
__device__ __forceinline__ int node_quadratic64(const P2MArgs &a, int Iu, int Ju, const int tri[3],
                                                const SA *st, const R lam[3], Emit &&emit)
{
    int us[UMAX];
    int nu;
    unsigned vm[3];
    int vi[3];
    if (node_u_sets<UMAX>(tri, st, us, nu, vm, vi, min(a.ucap, UMAX)) != 0) return -PFEM_DEFER;
    longlong2 o[UMAX];
    long long w[UMAX];
    if (node_offsets64<P>(a.pos, Iu, Ju, a.n - 1, us, nu, o) == NOT_FINITE) return -PFEM_DEFER;
    for (int i = 0; i < nu; ++i) w[i] = 0;
    const double l64[3] = {(double)lam[0], (double)lam[1], (double)lam[2]};
    double unit;
    const int r = node_solve64(o, vm, vi, l64, 0, 3, w, unit, -PFEM_DEFER);
    if (r != 0) return r;
    for (int i = 0; i < nu; ++i) emit(us[i], (R)(__ll2double_rn(w[i]) * unit));
#pragma unroll
    for (int e = 0; e < 3; ++e) emit(tri[e], lam[e]);
    return 0;
}

// Barycentric coordinates of the node (the origin of np's offsets) in triangle tri.  Here and in the
// edge systems every fused multiply-add is written out: the compiler would choose them differently
// in the kernels that share this arithmetic, whose results agree bit for bit.
template <typename P, typename R>
__device__ __forceinline__ void barycentric(const P2MArgs &a, const NodePos<P, R> &np,
                                            const int tri[3], R lam[3])
{
    R d[3][2];
#pragma unroll
    for (int e = 0; e < 3; ++e) np.off(a.pos, tri[e], d[e][0], d[e][1]);
    const R area2 = fma(d[1][0] - d[0][0], d[2][1] - d[0][1], -((d[1][1] - d[0][1]) * (d[2][0] - d[0][0])));
    lam[0] = fma(d[1][0], d[2][1], -(d[1][1] * d[2][0])) / area2;
    lam[1] = fma(d[2][0], d[0][1], -(d[2][1] * d[0][0])) / area2;
    lam[2] = fma(d[0][0], d[1][1], -(d[0][1] * d[1][0])) / area2;
}

template <typename V> __device__ __forceinline__ V nan_of();
template <> __device__ __forceinline__ float nan_of<float>() { return __int_as_float(0x7fc00000); }
template <> __device__ __forceinline__ double nan_of<double>() { return __longlong_as_double(0x7ff8000000000000LL); }

// One mesh node.  WEIGHTS = false: write alpha_i for all C components; true: write the
// node's distinct (slot, weight) pairs.
template <typename P, typename V, typename R, typename S, int REFINE, int SHAPE, bool WEIGHTS,
          bool SVD = false>
__device__ __forceinline__ void p2m_node(const P2MArgs &a, int I, int J)
{
    const int nc = a.n - 1;
    const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
    const long long node = (long long)J * a.n + I;
    const uint2 qn = make_uint2(node_fx(Iu, nc), node_fx(Ju, nc));
    int tri[3];
    int stars[3][KMAX];
    int ns[3] = {0, 0, 0};
    int st = locate(a.B, qn, a.R0, tri, stars[0], ns[0]);
    if (SHAPE == PFEM_SHAPE_QUADRATIC && st == 0) {
        for (int e = 0; e < 3 && st == 0; ++e)
            if (ns[e] == 0) {
                const int c = star_of(a.B, tri[e], a.R0, stars[e]);
                if (c < 0) st = c;
                else ns[e] = c;
            }
    }
    NodePos<P, R> np;
    np.init(Iu, Ju, nc);
    R lam[3] = {R(0), R(0), R(0)};
    if (st == 0) barycentric(a, np, tri, lam);

    if (!WEIGHTS) {
        R acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = R(0);
        auto emit = [&](int s, R wgt) {
            R v[8];
            load_vals<V, R>((const V *)a.vals, a.perm, s, a.C, v);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < a.C) acc[c] = fma(wgt, v[c], acc[c]);
        };
        if (st == 0) {
            if (SHAPE == PFEM_SHAPE_QUADRATIC) {
                const ArrStar sa[3] = {{stars[0], ns[0]}, {stars[1], ns[1]}, {stars[2], ns[2]}};
                if constexpr (REFINE == REFINE_FIX64) {
                    st = node_quadratic64<P, R>(a, Iu, Ju, tri, sa, lam, emit);
                    if (st == -PFEM_DEFER && short_queue(a))          // (nothing was emitted)
                        st = node_quadratic<P, R, double, sizeof(R) == 8 ? REFINE_STEP : REFINE_NONE, false>(a, np, tri, sa, lam, emit);
                } else {
                    st = node_quadratic<P, R, S, REFINE, SVD>(a, np, tri, sa, lam, emit);
                }
            } else {
                for (int e = 0; e < 3; ++e) emit(tri[e], lam[e]);
            }
        }
        st = defer_or_error(a, st, a.noff + node);
        if (st != 0) {
            if (st < 0) record_error(a.status, -st, a.noff + node);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = (R)nan_of<R>();
        }
        store_vals<V, R>((V *)a.out, node, a.C, acc);
    } else {
        int idx[PFEM_KW_MAX];
        R wl[PFEM_KW_MAX];
        int cnt = 0;
        bool over = false;
        auto emit = [&](int s, R wgt) {
            for (int i = 0; i < cnt; ++i)
                if (idx[i] == s) { wl[i] += wgt; return; }
            if (cnt < a.K) { idx[cnt] = s; wl[cnt] = wgt; ++cnt; }
            else over = true;
        };
        if (st == 0) {
            if (SHAPE == PFEM_SHAPE_QUADRATIC) {
                const ArrStar sa[3] = {{stars[0], ns[0]}, {stars[1], ns[1]}, {stars[2], ns[2]}};
                if constexpr (REFINE == REFINE_FIX64) {
                    st = node_quadratic64<P, R>(a, Iu, Ju, tri, sa, lam, emit);
                    if (st == -PFEM_DEFER && short_queue(a))          // (nothing was emitted)
                        st = node_quadratic<P, R, double, sizeof(R) == 8 ? REFINE_STEP : REFINE_NONE, false>(a, np, tri, sa, lam, emit);
                } else {
                    st = node_quadratic<P, R, S, REFINE, SVD>(a, np, tri, sa, lam, emit);
                }
            } else {
                for (int e = 0; e < 3; ++e) emit(tri[e], lam[e]);
            }
            if (over && st == 0) st = -PFEM_ERR_CAPACITY;
        }
        st = defer_or_error(a, st, a.noff + node);
        if (st != 0) {
            if (st < 0) record_error(a.status, -st, a.noff + node);
            cnt = 0;
        }
        int *oi = a.w_idx + node * a.K;
        R *ow = (R *)a.w + node * a.K;
        for (int k = 0; k < a.K; ++k) {
            oi[k] = k < cnt ? idx[k] : -1;
            ow[k] = k < cnt ? wl[k] : R(0);
        }
    }
}

// Resident blocks per SM the compiler must allow (it caps registers at 65536 / (128 x 12) = 42):
// the per-node work is latency-bound, and measured on GB300 (sweep 1..16) twelve 128-thread
// blocks per SM were fastest despite the extra register spills.
#ifndef PFEM_P2M_MIN_BLOCKS
#define PFEM_P2M_MIN_BLOCKS 12
#endif

template <typename P, typename V, typename R, typename S, int REFINE, int SHAPE, bool WEIGHTS>
__global__ void __launch_bounds__(128, PFEM_P2M_MIN_BLOCKS) k_p2m(P2MArgs a)
{
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    if (I >= a.n || J >= a.n) return;
    p2m_node<P, V, R, S, REFINE, SHAPE, WEIGHTS>(a, I, J);
}

// Linear shape functions: one thread a node.  The node's triangle comes from the star of its nearest
// particle, by the hull over the thread's list in shared memory as in the star table (gift wrapping
// over lists in local memory took 169 us for 513^2 nodes over 1254^2 particles, this 92); the table itself
// would hold the stars of every particle, six a node there.  Every lane of the warp calls (locate_hull).
template <typename P, typename V, typename R, bool WEIGHTS>
__device__ __forceinline__ void linear_node(const P2MArgs &a, const HullList &L, int I, int J)
{
    const int nc = a.n - 1;
    const bool mine = I <= nc && J <= nc;
    const int Iu = I >= nc ? 0 : I, Ju = J >= nc ? 0 : J;
    const long long node = (long long)J * a.n + I;
    int tri[3];
    int st = locate_hull(a.B, mine, make_uint2(node_fx(Iu, nc), node_fx(Ju, nc)), a.R0, L, tri);
    if (!mine) return;
    R lam[3] = {R(0), R(0), R(0)}, acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = R(0);
    if (st == 0) {
        NodePos<P, R> np;
        np.init(Iu, Ju, nc);
        barycentric(a, np, tri, lam);
        if (!WEIGHTS)
            for (int e = 0; e < 3; ++e) {
                R v[8];
                load_vals<V, R>((const V *)a.vals, a.perm, tri[e], a.C, v);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < a.C) acc[c] = fma(lam[e], v[c], acc[c]);
            }
        else if (a.K < 3) st = -PFEM_ERR_CAPACITY;
    }
    st = defer_or_error(a, st, a.noff + node);
    if (st < 0) record_error(a.status, -st, a.noff + node);
    if (!WEIGHTS) {
        if (st != 0)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = (R)nan_of<R>();
        store_vals<V, R>((V *)a.out, node, a.C, acc);
    } else {
        int *oi = a.w_idx + node * a.K;
        R *ow = (R *)a.w + node * a.K;
        for (int k = 0; k < a.K; ++k) {
            const bool v = st == 0 && k < 3;
            oi[k] = v ? tri[k] : -1;
            ow[k] = v ? lam[k] : R(0);
        }
    }
}

// Resident 128-thread blocks per SM: the warp search wants registers (at 64 it spills). 8, 6, 5, 4 blocks:
// 257^2 nodes over 1024^2 uniform random particles 597, 341, 300, 277 us, 1025^2 over 1025^2 4565, 2715,
// 2666, 2856, 513^2 over 1254^2 lattice particles 135, 115, 107, 107.
#ifndef PFEM_LINEAR_MIN_BLOCKS
#define PFEM_LINEAR_MIN_BLOCKS 5
#endif
template <typename P, typename V, typename R, bool WEIGHTS>
__global__ void __launch_bounds__(STAR_TPB, PFEM_LINEAR_MIN_BLOCKS) k_p2m_linear(P2MArgs a)
{
    __shared__ __align__(16) unsigned char lists[HullList::BYTES];
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    linear_node<P, V, R, WEIGHTS>(a, HullList::at(lists, threadIdx.x), I, J);
}

// The queued nodes again, overwriting the fast pass's placeholder output: the geometry searched
// per thread with the widest search radius (the launcher passes it in a.B.rmax), and with
// quadratic shape functions every edge solved in FP64 (node_u_fix).  A node that fails here
// reports its error.
template <typename P, typename V, typename R, int SHAPE, bool WEIGHTS>
__global__ void __launch_bounds__(128) k_p2m_fix(P2MArgs a)
{
    const int cnt = min(*a.defer_count, a.defer_cap);
    P2MArgs f = a;
    f.defer_cap = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
        const long long node = a.defer_list[i];
        p2m_node<P, V, R, double, REFINE_NONE, SHAPE, WEIGHTS, true>(
            f, (int)(node % a.n), (int)(node / a.n));
    }
}

// ---------------------------------------------------------------- star table path
// The node's particle set and stencil masks as node_u_sets gives them (same order), from stars of up
// to 8 particles held in registers: n the stars' sizes, su the thread's column of shared memory
// (stride between entries) that receives the slots.  Returns the set's size; the slots are complete
// up to SET_MAX.  Jittered lattices fit everywhere.
//
// The node kernel is bound by latency: what a thread kept in local memory (the growing set, which
// node_u_sets searches entry by entry, and the weights) came to half a megabyte a resident SM's
// threads, and its loads waited on L2.  node_u_sets took 178 us of the kernel's 660 us at 1025^2
// nodes / 2048^2 particles; here every step is the same in every lane, the stars' rows come in two
// loads each, and slots and weights lie in shared memory: 560 us.  (The offsets in shared memory as
// well, or everything in registers with the loops over all 16 entries unrolled, cost blocks per SM:
// 600 and 770 us.)
constexpr int SET_MAX = 16;
// Rows of a thread's column: the slots (two spare) and the weights.
constexpr int SET_W = SET_MAX + 2, SET_ROWS = SET_W + SET_MAX;

// An array whose entries lie `stride` apart.
template <typename T> struct Strided {
    T *p;
    int stride;
    __device__ __forceinline__ T &operator[](int i) const { return p[i * stride]; }
};

__device__ __forceinline__ int node_sets8(const StarTab &t, const int tri[3], const int n[3], int *su,
                                          int stride, unsigned vm[3])
{
    int s[3][8];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int4 *row = reinterpret_cast<const int4 *>(t.nbr + (long long)tri[e] * KMAX);
        const int4 lo = __ldg(row), hi = __ldg(row + 1);
        s[e][0] = lo.x; s[e][1] = lo.y; s[e][2] = lo.z; s[e][3] = lo.w;
        s[e][4] = hi.x; s[e][5] = hi.y; s[e][6] = hi.z; s[e][7] = hi.w;
        su[e * stride] = tri[e];
    }
    int nu = 3;
    unsigned bit[2][8];                  // set bit of each entry of the first two stars (0: none)
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        unsigned m = 1u << e;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int x = s[e][j];
            unsigned b = 0u;
#pragma unroll
            for (int f = 0; f < 3; ++f)
                if (f != e) b |= x == tri[f] ? 1u << f : 0u;
#pragma unroll
            for (int f = 0; f < e; ++f)
#pragma unroll
                for (int i = 0; i < 8; ++i) b |= s[f][i] == x ? bit[f][i] : 0u;
            const bool valid = j < n[e], fresh = valid && b == 0u;
            su[min(nu, SET_MAX) * stride] = x;
            b = fresh ? 1u << nu : b;
            nu += fresh ? 1 : 0;
            b = valid ? b : 0u;
            if (e < 2) bit[e < 2 ? e : 0][j] = b;
            m |= b;
        }
        vm[e] = m;
    }
    return nu;
}

// The lanes of a node (a group of Q consecutive ones that run the same control flow), and the sum
// and the least of their values.
template <int Q> __device__ __forceinline__ unsigned group_mask()
{
    return ((1u << Q) - 1u) << (threadIdx.x & 31 & ~(Q - 1));
}
template <int Q, typename T> __device__ __forceinline__ T group_sum(T v)
{
#pragma unroll
    for (int o = 1; o < Q; o <<= 1) v += __shfl_xor_sync(group_mask<Q>(), v, o);
    return v;
}
template <int Q> __device__ __forceinline__ int group_min(int v)
{
#pragma unroll
    for (int o = 1; o < Q; o <<= 1) v = min(v, __shfl_xor_sync(group_mask<Q>(), v, o));
    return v;
}

// node_sets8 where it applies: true when the sets of all nodes of the warp fit (one path a warp: a
// few nodes with larger sets would otherwise cost it both).  st != 0: no node here.  The lanes that vote
// are those that happen to arrive together, which need not be the whole warp; the Q lanes of a node,
// which exchange values on the path that is chosen, agree on the answer over their own mask.
template <int Q>
__device__ __forceinline__ bool warp_sets8(const StarTab &t, int st, const int tri[3], const TabStar sa[3],
                                           int cap, int *su, int stride, int &nu, unsigned vm[3])
{
    bool fits = true;
    if (st == 0) {
        const int n[3] = {sa[0].n, sa[1].n, sa[2].n};
        fits = max(n[0], max(n[1], n[2])) <= 8;
        if (fits) {
            nu = node_sets8(t, tri, n, su, stride, vm);
            fits = nu <= min(cap, SET_MAX);
        }
    }
    return group_min<Q>(__all_sync(__activemask(), fits) ? 1 : 0) != 0;
}

// The fix pass of the table path: the queued nodes located with the star table (complete after
// the retry kernels; the launcher passes the widest search radius for the nearest particle),
// four lanes a node as in tab_node, the edges as in node_u_fix.  A queued node's time is one thread's chain of FP64 instructions, so the edges of a node run side by side: about
// 1500 queued nodes of 513^2 over 1024^2 uniform random particles 1150 -> 434 us.
template <typename P, typename V, typename R>
__global__ void __launch_bounds__(128) k_p2m_fix_tab(P2MArgs a, StarTab t)
{
    constexpr int Q = 4, UM = UMAX_SVD;
    const int cnt = min(*a.defer_count, a.defer_cap);
    const int q = threadIdx.x & (Q - 1), e0 = q, e1 = min(q + 1, 3);
    P2MArgs f = a;
    f.defer_cap = 0;
    const int nc = a.n - 1;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / Q; i < cnt; i += gridDim.x * blockDim.x / Q) {
        const long long node = a.defer_list[i];
        const int I = (int)(node % a.n), J = (int)(node / a.n);
        const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
        const uint2 qn = make_uint2(node_fx(Iu, nc), node_fx(Ju, nc));
        int tri[3];
        int st = locate_tab(f.B, t, qn, f.R0, tri);
        if (st == -PFEM_FAR) st = -PFEM_ERR_CAPACITY;
        TabStar sa[3];
#pragma unroll
        for (int e = 0; e < 3; ++e)
            if (st == 0) {
                sa[e] = tab_star(t, tri[e]);
                if (sa[e].n < 0) st = sa[e].n == -1 ? -PFEM_ERR_CAPACITY : sa[e].n;
            }
        R acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = R(0);
        if (st == 0) {
            NodePos<P, R> np;
            np.init(Iu, Ju, nc);
            R lam[3];
            barycentric(f, np, tri, lam);
            int us[UM];
            R uw[UM];
            int nu;
            unsigned vm[3];
            int vi[3];
            if (node_u_sets<UM>(tri, sa, us, nu, vm, vi) != 0) {
                st = -PFEM_ERR_CAPACITY;
            } else {
                for (int k = 0; k < nu; ++k) uw[k] = R(0);
                if (q == 0)
#pragma unroll
                    for (int e = 0; e < 3; ++e) uw[vi[e]] += lam[e];
                node_u_fix<P, R, UM>(f, np, us, uw, vm, vi, lam, e0, e1);
                __syncwarp(0xfu << (threadIdx.x & 28));
                for (int k = 0; k < nu; ++k) {
                    const R wk = group_sum<Q>(uw[k]);
                    if ((k & (Q - 1)) != q) continue;
                    R v[8];
                    load_vals<V, R>((const V *)f.vals, f.perm, us[k], f.C, v);
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (c < f.C) acc[c] = fma(wk, v[c], acc[c]);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < f.C) acc[c] = group_sum<Q>(acc[c]);
            }
        }
        if (q != 0) continue;
        if (st != 0) {
            record_error(f.status, -st, node);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = (R)nan_of<R>();
        }
        store_vals<V, R>((V *)f.out, node, f.C, acc);
    }
}

// The table path's fast pass in one kernel: each thread locates its node with the star table,
// builds its particle set and solves its three edge systems, without a node record in between.
// The refined solve's residual runs on the integer pipes (FixRes); in FP64 it held the FP64 pipe
// for 0.47 ms of this kernel's 0.99 ms at 1025^2 nodes / 2048^2 particles, C = 4, FP32 (now 0.56
// ms with the sets in shared memory; 4097^2 / 8192^2: 14.6 -> 8.2 ms).  What bounds it now are the
// waits for star rows and positions in L2 (24 of 32 lanes active).  Errors against 64-bit arithmetic are unchanged (1.1e-7
// of the mesh's 2-norm; the two results differ by 2e-8 of it, and edge by edge the errors agree at every
// quantile, on stretched, clustered and uniform random sets too).  The float-float refinement that
// PFEM_SOLVE_F32_REFINED_FF names (48 bits, about 200 FP32 instructions a point and edge) took
// 0.84 ms in two kernels; it takes this path too, whose residual is the more exact.
// Resident 128-thread blocks per SM: 7 with one lane a node (1025^2 / 2048^2 round trip: 6, 7, 8, 9
// blocks 1124, 1096, 1107, 1123 us), and for the solution refined to FP64, with its longer live
// ranges, 6 (513^2 / 1024^2: 4, 5, 6 blocks 739, 713, 700 us); 8 and 4 with four lanes a node, where
// there are not enough nodes to fill the SMs.
template <int REFINE, int Q = 1> constexpr int tab_min_blocks()
{
    return REFINE == REFINE_FIX64 ? (Q > 1 ? 4 : 6) : (Q > 1 ? 8 : 7);
}

// The edge systems of a node's set (slots us, weights weight) and the apply of the result; tab_node
// says what Q and q are.  Returns 0 or -PFEM_DEFER.
template <int UM, typename P, typename V, typename R, typename S, int REFINE, int Q, typename Slots,
          typename Weights, typename Apply>
__device__ __forceinline__ int set_solve(const P2MArgs &a, const NodePos<P, R> &np, int Iu, int Ju, int q,
                                         const int tri[3], int nu, const unsigned vm[3], const int vi[3],
                                         const R lam[3], Slots us, Weights weight, Apply &&apply)
{
    const int e0 = Q > 1 ? q : 0, e1 = Q > 1 ? min(q + 1, 3) : 3;
    int st;
    if constexpr (REFINE == REFINE_FIX64) {
        longlong2 o[UM];
        long long w[UM];
        const bool finite = node_offsets64<P>(a.pos, Iu, Ju, a.n - 1, us, nu, o) != NOT_FINITE;
        for (int i = 0; i < nu; ++i) w[i] = 0;
        const double l64[3] = {(double)lam[0], (double)lam[1], (double)lam[2]};
        double unit = 0.0;
        st = group_min<Q>(finite ? node_solve64(o, vm, vi, l64, e0, e1, w, unit, -PFEM_DEFER) : -PFEM_DEFER);
        if (st == 0) {
            for (int i = 0; i < nu; ++i) apply(us[i], (R)(__ll2double_rn(group_sum<Q>(w[i])) * unit));
#pragma unroll
            for (int e = 0; e < 3; ++e) apply(tri[e], lam[e]);
        }
    } else {
        for (int i = 0; i < nu; ++i) weight[i] = R(0);
        auto ref = [&](int i) -> R & { return weight[i]; };
        auto offset = [&](int i, S &x, S &y) {
            R dx, dy;
            np.off(a.pos, us[i], dx, dy);
            x = S(dx);
            y = S(dy);
        };
        if constexpr (Q == 1) {
#pragma unroll
            for (int e = 0; e < 3; ++e) weight[vi[e]] += lam[e];
            st = node_edges<R, S, REFINE, false, UM, false>(ref, vm, vi, lam, 0, 3, offset);
            if (st == 0)
                for (int i = 0; i < nu; ++i) apply(us[i], weight[i]);
        } else {
            st = group_min<Q>(node_edges<R, S, REFINE, false, UM, true>(ref, vm, vi, lam, e0, e1, offset));
            const R coef[3] = {R(2) * lam[0] * lam[1], R(2) * lam[1] * lam[2], R(2) * lam[2] * lam[0]};
            if (st == 0)
                for (int i = 0; i < nu; ++i) {
                    R w = i == vi[0] ? lam[0] : i == vi[1] ? lam[1] : i == vi[2] ? lam[2] : R(0);
#pragma unroll
                    for (int e = 0; e < 3; ++e)
                        w = fma(coef[e], __shfl_sync(group_mask<Q>(), weight[i], e, Q), w);
                    apply(us[i], w);
                }
        }
    }
    return st;
}

// Node (I, J) of the problem of a (mesh output a.out; queue entries and error details at node
// a.noff + J * a.n + I of the batch), by Q = 1 lane, or by Q = 4 lanes that all locate it, solve an
// edge each (the fourth none) and take the components c = q, q + 4 of the apply.  Both give the same
// result bit for bit: the edges' contributions and the particles are added up in the same order.
// su: the calling thread's column of SET_ROWS words in shared memory, entry i at i * stride.
template <typename P, typename V, typename R, typename S, int REFINE, int Q = 1>
__device__ __forceinline__ void tab_node(const P2MArgs &a, const StarTab &t, int I, int J, int *su, int stride)
{
    const int q = Q > 1 ? (int)threadIdx.x & (Q - 1) : 0;
    const int nc = a.n - 1;
    const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
    const long long node = (long long)J * a.n + I;
    const uint2 qn = make_uint2(node_fx(Iu, nc), node_fx(Ju, nc));
    int tri[3];
    int st = locate_tab(a.B, t, qn, a.R0, tri);
    TabStar sa[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
        if (st == 0) {
            sa[e] = tab_star(t, tri[e]);
            if (sa[e].n < 0) st = sa[e].n == -1 ? -PFEM_FAR : sa[e].n;
        }
    R acc[8];                   // all components (Q = 1), or q, q + 4
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = R(0);
    auto apply = [&](int s, R w) {
        if constexpr (Q == 1) {
            R v[8];
            load_vals<V, R>((const V *)a.vals, a.perm, s, a.C, v);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < a.C) acc[c] = fma(w, v[c], acc[c]);
        } else {
            const V *p = (const V *)a.vals + (a.perm ? (long long)__ldg(a.perm + s) : (long long)s) * a.C;
#pragma unroll
            for (int k = 0; k < 8 / Q; ++k)
                if (q + Q * k < a.C) acc[k] = fma(w, load_val<V, R>(p + q + Q * k), acc[k]);
        }
    };
    int nu = 0;
    unsigned vm[3] = {0u, 0u, 0u};
    const bool small = warp_sets8<Q>(t, st, tri, sa, a.ucap, su, stride, nu, vm);
    if (st == 0) {
        NodePos<P, R> np;
        np.init(Iu, Ju, nc);
        R lam[3];
        barycentric(a, np, tri, lam);
        int vi[3] = {0, 1, 2};
        if (small) {
            st = set_solve<SET_MAX, P, V, R, S, REFINE, Q>(a, np, Iu, Ju, q, tri, nu, vm, vi, lam, Strided<int>{su, stride},
                                                           Strided<R>{reinterpret_cast<R *>(su) + SET_W * stride, stride},
                                                           apply);
        } else {
            int us[UMAX];
            R uw[REFINE == REFINE_FIX64 ? 1 : UMAX];
            if (node_u_sets<UMAX>(tri, sa, us, nu, vm, vi, min(a.ucap, UMAX)) != 0)
                st = a.defer_cap > 0 ? -PFEM_DEFER : -PFEM_ERR_CAPACITY;
            else
                st = set_solve<UMAX, P, V, R, S, REFINE, Q>(a, np, Iu, Ju, q, tri, nu, vm, vi, lam, Strided<int>{us, 1},
                                                            Strided<R>{uw, 1}, apply);
        }
    }
    if (st != 0) {
        if (q == 0) {
            st = defer_or_error(a, st, a.noff + node);
            if (st < 0) record_error(a.status, -st, a.noff + node);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = (R)nan_of<R>();
    }
    if constexpr (Q == 1) {
        store_vals<V, R>((V *)a.out, node, a.C, acc);
    } else {
#pragma unroll
        for (int k = 0; k < 8 / Q; ++k)
            if (q + Q * k < a.C) store_val<V, R>((V *)a.out + node * a.C + q + Q * k, acc[k]);
    }
}

// Shared words a thread: slots, and weights where they are FP32 ones.
template <int REFINE> constexpr int tab_rows() { return REFINE == REFINE_FIX64 ? SET_W : SET_ROWS; }

template <typename P, typename V, typename R, typename S, int REFINE, int Q>
__global__ void __launch_bounds__(128, tab_min_blocks<REFINE, Q>()) k_p2m_tab(P2MArgs a, StarTab t)
{
    __shared__ int su[tab_rows<REFINE>() * 128];
    // 16 x 8 nodes a block, or 8 x 4 with four lanes a node
    const int x = threadIdx.x / Q;
    const int I = blockIdx.x * (Q > 1 ? 8 : 16) + (Q > 1 ? x & 7 : x & 15);
    const int J = blockIdx.y * (Q > 1 ? 4 : 8) + (Q > 1 ? x >> 3 : x >> 4);
    if (I >= a.n || J >= a.n) return;
    tab_node<P, V, R, S, REFINE, Q>(a, t, I, J, su + threadIdx.x, 128);
}

// Explicit weights of every node with the star table: as k_p2m_tab, writing the node's row of (slot,
// weight) pairs, -1 and 0 past them.  vec: rows that 16-byte stores can write.
template <typename P, typename R, int REFINE>
__global__ void __launch_bounds__(128, tab_min_blocks<REFINE>()) k_shape_tab(P2MArgs a, StarTab t, bool vec)
{
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    if (I >= a.n || J >= a.n) return;
    const int nc = a.n - 1;
    const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
    const long long node = (long long)J * a.n + I;
    int tri[3];
    int st = locate_tab(a.B, t, make_uint2(node_fx(Iu, nc), node_fx(Ju, nc)), a.R0, tri);
    TabStar sa[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
        if (st == 0) {
            sa[e] = tab_star(t, tri[e]);
            if (sa[e].n < 0) st = sa[e].n == -1 ? -PFEM_FAR : sa[e].n;
        }
    int us[UMAX];
    R uw[UMAX];
    int nu = 0;
    if (st == 0) {
        NodePos<P, R> np;
        np.init(Iu, Ju, nc);
        R lam[3];
        barycentric(a, np, tri, lam);
        unsigned vm[3];
        int vi[3];
        if (node_u_sets<UMAX>(tri, sa, us, nu, vm, vi, min(a.ucap, UMAX)) != 0) {
            st = -PFEM_DEFER;
        } else if constexpr (REFINE == REFINE_FIX64) {
            longlong2 o[UMAX];
            long long w[UMAX];
            const bool finite = node_offsets64<P>(a.pos, Iu, Ju, nc, us, nu, o) != NOT_FINITE;
            for (int i = 0; i < nu; ++i) w[i] = 0;
            const double l64[3] = {(double)lam[0], (double)lam[1], (double)lam[2]};
            double unit = 0.0;
            st = finite ? node_solve64(o, vm, vi, l64, 0, 3, w, unit, -PFEM_DEFER) : -PFEM_DEFER;
            for (int i = 0; i < nu; ++i) uw[i] = (R)(__ll2double_rn(w[i]) * unit);
#pragma unroll
            for (int e = 0; e < 3; ++e) uw[vi[e]] += lam[e];
        } else {
            for (int i = 0; i < nu; ++i) uw[i] = R(0);
#pragma unroll
            for (int e = 0; e < 3; ++e) uw[vi[e]] += lam[e];
            st = node_u_solve<P, R, float, REFINE, false, UMAX>(a, np, us, uw, vm, vi, lam);
        }
        if (st == 0 && nu > a.K) st = -PFEM_ERR_CAPACITY;
    }
    if (st != 0) {
        st = defer_or_error(a, st, node);
        if (st < 0) record_error(a.status, -st, node);
        nu = 0;
    }
    int *oi = a.w_idx + node * a.K;
    R *ow = (R *)a.w + node * a.K;
    if (vec) {
        using V4 = std::conditional_t<sizeof(R) == 4, float4, double4>;
        for (int k = 0; k < a.K; k += 4) {
            int s[4];
            R w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[i] = k + i < nu ? us[k + i] : -1;
                w[i] = k + i < nu ? uw[k + i] : R(0);
            }
            *reinterpret_cast<int4 *>(oi + k) = make_int4(s[0], s[1], s[2], s[3]);
            V4 v;
            v.x = w[0]; v.y = w[1]; v.z = w[2]; v.w = w[3];
            *reinterpret_cast<V4 *>(ow + k) = v;
        }
    } else {
        for (int k = 0; k < a.K; ++k) {
            oi[k] = k < nu ? us[k] : -1;
            ow[k] = k < nu ? uw[k] : R(0);
        }
    }
}

}  // namespace pfem
