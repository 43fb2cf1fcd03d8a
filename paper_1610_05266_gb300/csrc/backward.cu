// backward.cu -- adjoint of P2M with respect to particle values and positions (no paper
// counterpart; the paper only runs the forward projection).
//
// Forward, per node i:  alpha_i = sum_mu w_{i mu}(r) alpha_mu  with
//   w_{i mu} = lambda_mu [mu in T] + sum_{e=(nu,sg) in T} c_e A_{mu e},   c_e = 2 lambda_nu lambda_sg,
//   A_{mu e} = p_mu . y_e,  M_e y_e = b_e,  M_e = sum_{mu in S_e} p_mu p_mu^T.
// With beta_mu = gbar_i . alpha_mu, the node contributes
//   dL/dalpha_mu += w_{i mu} gbar_i,
//   dL/dr via lambda (barycentric cofactors) and via every edge: u = sum beta_mu p_mu,
//   B_e = u . y_e, z = M_e^{-1} u (one extra solve), and for each stencil member
//   pbar_mu = c_e [(beta_mu - z.p_mu) y_e - (y_e.p_mu) z],  tbar from b_e, lambdabar from c_e B_e.
// The frame (edge midpoint, edge length) is held fixed: A does not depend on it (eq. A2_2), so
// the derivative at a fixed frame is the derivative of A.
//
// Determinism without atomics on values: phase 1 writes each node's entries (slot, w, dpos)
// into arrays of K entries a node; phase 2 builds a transposed index by a stable counting sort
// keyed by particle slot (entries per particle ordered by entry id) and gathers per particle.
//
// The entries of phase 1 are laid out entry by entry (entry k of node i at k * nodes + i), only as
// many as the node has, so that a warp's nodes write whole lines; weight and position adjoint of
// an entry lie together, since the gather reads them together.  Phase 1 also counts the entries
// of each particle as it writes them.  (Node by node, padded to K = 32 entries and counted by a
// pass of its own, the solve kernel's scattered 4-byte stores bound it: 1040 us at 1025^2 nodes /
// 2048^2 particles, C = 1, FP32, and 376 us for the transposed gather.)
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "p2m.cuh"

namespace pfem {

struct BwdArgs {
    P2MArgs f;                  // forward geometry/values (f.out unused)
    const void *grad_mesh;      // [n*n, C]
    int K;                      // entries per node
    long long nodes;            // n*n
    int *e_cnt;                 // [nodes] entries of the node
    int *e_slot;                // [K][nodes]
    int *e_rank;                // [K][nodes] arrival rank of the entry at its particle
    void *e_val;                // [K][nodes] Entry<R>, or the weights alone (R) without positions
    int *count;                 // [N] entries of the particle
};

// Weight and position adjoint of an entry: one 16-byte access in FP32.
template <typename R> struct Entry;
template <> struct __align__(16) Entry<float> {
    float w, dx, dy, pad;
};
template <> struct Entry<double> {
    double w, dx, dy;
};
// An entry's id in the transposed index: its node and its number.
constexpr int ENTRY_BITS = 5;

// Write the entries of a node (nu <= K).
template <typename R, typename T, bool POS>
__device__ __forceinline__ void write_entries(const BwdArgs &b, long long node, int nu, const int *us,
                                              const T *uw, const T *udx, const T *udy)
{
    b.e_cnt[node] = nu;
    for (int k = 0; k < nu; ++k) {
        const long long e = k * b.nodes + node;
        b.e_slot[e] = us[k];
        b.e_rank[e] = atomicAdd(b.count + us[k], 1);
        if constexpr (POS) {
            Entry<R> v;
            v.w = (R)uw[k];
            v.dx = (R)udx[k];
            v.dy = (R)udy[k];
            ((Entry<R> *)b.e_val)[e] = v;
        } else {
            ((R *)b.e_val)[e] = (R)uw[k];
        }
    }
}

constexpr int KBWD = 32;   // distinct particles per node kept by the recompute kernel

// The adjoint of one node over its particle set (us[0..nu), stencil masks vm, tri[e] = us[vi[e]]):
// uw the weights, ub = gbar . alpha per particle, udx/udy the position adjoints (all zero on
// entry).  Returns 0, or -PFEM_DEFER when a moment matrix is below the forward's fast-solve
// tolerance: the node goes to the adjoint's fix pass, as the forward sends it to its own.
template <typename P, typename V, typename R, typename S, int SHAPE, bool POS>
__device__ __forceinline__ int bwd_u_solve(const BwdArgs &b, const NodePos<P, R> &np, const R g[8],
                                           const int tri[3], const int *us, int nu,
                                           const unsigned vm[3], const int vi[3], R *uw, R *ub,
                                           R *udx, R *udy)
{
    const P2MArgs &a = b.f;
    int st = 0;
    for (int i = 0; i < nu; ++i) {
        R v[8];
        load_vals<V, R>((const V *)a.vals, a.perm, us[i], a.C, v);
        R t = R(0);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < a.C) t = fma(g[c], v[c], t);
        ub[i] = t;
    }
    R d[3][2];
#pragma unroll
    for (int e = 0; e < 3; ++e) np.off(a.pos, tri[e], d[e][0], d[e][1]);
    const R Na = d[1][0] * d[2][1] - d[1][1] * d[2][0];
    const R Nb = d[2][0] * d[0][1] - d[2][1] * d[0][0];
    const R Nc = d[0][0] * d[1][1] - d[0][1] * d[1][0];
    const R A2 = Na + Nb + Nc;
    const R lam[3] = {Na / A2, Nb / A2, Nc / A2};
    R lbar[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        uw[vi[e]] += lam[e];
        lbar[e] = ub[vi[e]];
    }
    auto offset = [&](int i, S &x, S &y) {
        R dx, dy;
        np.off(a.pos, us[i], dx, dy);
        x = S(dx);
        y = S(dy);
    };
    if (SHAPE == PFEM_SHAPE_QUADRATIC)
        for (int e = 0; e < 3 && st == 0; ++e) {
            const int f = e == 2 ? 0 : e + 1;
            const unsigned mask = vm[e] | vm[f];
            const S rnx = S(d[e][0]), rny = S(d[e][1]), rsx = S(d[f][0]), rsy = S(d[f][1]);
            const S mx = (rnx + rsx) * S(0.5), my = (rny + rsy) * S(0.5);
            const S ex = rnx - rsx, ey = rny - rsy;
            const S inv = S(1) / sqrt(ex * ex + ey * ey);
            Moment<S> M;
            M.zero();
            S u[6] = {S(0), S(0), S(0), S(0), S(0), S(0)};
            for (unsigned m = mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                S ox, oy;
                offset(i, ox, oy);
                const S x = (ox - mx) * inv, y = (oy - my) * inv;
                M.add(x, y);
                const S bt = S(ub[i]);
                const S p[6] = {S(1), x, y, x * x, x * y, y * y};
#pragma unroll
                for (int r = 0; r < 6; ++r) u[r] = fma(bt, p[r], u[r]);
            }
            if (!M.factor(FastTol<S>::v)) { st = -PFEM_DEFER; break; }
            const S tx = ex * inv, ty = ey * inv;
            const S bb[6] = {S(0), S(0), S(0), S(-0.5) * tx * tx, S(-0.5) * tx * ty,
                             S(-0.5) * ty * ty};
            S y[6], z[6];
            M.solve(bb, y);
            M.solve(u, z);
            const S ce = S(2) * S(lam[e]) * S(lam[f]);
            S Be = S(0);
#pragma unroll
            for (int r = 0; r < 6; ++r) Be = fma(u[r], y[r], Be);
            lbar[e] += R(S(2) * S(lam[f]) * Be);
            lbar[f] += R(S(2) * S(lam[e]) * Be);
            for (unsigned m = mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                S ox, oy;
                offset(i, ox, oy);
                const S x = (ox - mx) * inv, yy = (oy - my) * inv;
                const S p[6] = {S(1), x, yy, x * x, x * yy, yy * yy};
                S Am = S(0), Zm = S(0);
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    Am = fma(p[r], y[r], Am);
                    Zm = fma(p[r], z[r], Zm);
                }
                uw[i] += R(ce * Am);
                if (POS) {
                    const S bt = S(ub[i]);
                    S pb[6];
#pragma unroll
                    for (int r = 0; r < 6; ++r) pb[r] = ce * ((bt - Zm) * y[r] - Am * z[r]);
                    const S xb = pb[1] + S(2) * x * pb[3] + yy * pb[4];
                    const S yb = pb[2] + x * pb[4] + S(2) * yy * pb[5];
                    udx[i] += R(xb * inv);
                    udy[i] += R(yb * inv);
                }
            }
            if (POS) {
                // b = [0,0,0,-tx^2/2,-tx ty/2,-ty^2/2], t = (r_nu - r_sg)/s
                const S txb = ce * (-tx * z[3] - S(0.5) * ty * z[4]);
                const S tyb = ce * (-S(0.5) * tx * z[4] - ty * z[5]);
                udx[vi[e]] += R(txb * inv);
                udy[vi[e]] += R(tyb * inv);
                udx[vi[f]] -= R(txb * inv);
                udy[vi[f]] -= R(tyb * inv);
            }
        }
    if (POS && st == 0) {
        // lambda_k = N_k / A2 with N_a = d_b x d_c, N_b = d_c x d_a, N_c = d_a x d_b
        const R Lam = lbar[0] * lam[0] + lbar[1] * lam[1] + lbar[2] * lam[2];
        const R nb0 = (lbar[0] - Lam) / A2, nb1 = (lbar[1] - Lam) / A2, nb2 = (lbar[2] - Lam) / A2;
        // cross(u, v): d/du = (v.y, -v.x), d/dv = (-u.y, u.x)
        R gx[3] = {R(0), R(0), R(0)}, gy[3] = {R(0), R(0), R(0)};
        gx[1] += nb0 * d[2][1];  gy[1] -= nb0 * d[2][0];
        gx[2] -= nb0 * d[1][1];  gy[2] += nb0 * d[1][0];
        gx[2] += nb1 * d[0][1];  gy[2] -= nb1 * d[0][0];
        gx[0] -= nb1 * d[2][1];  gy[0] += nb1 * d[2][0];
        gx[0] += nb2 * d[1][1];  gy[0] -= nb2 * d[1][0];
        gx[1] -= nb2 * d[0][1];  gy[1] += nb2 * d[0][0];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            udx[vi[e]] += gx[e];
            udy[vi[e]] += gy[e];
        }
    }
    return st;
}

// bwd_u_solve for quadratic shape functions in FP64 without FP64 systems: y and z of each edge from the
// FP32 factor, refined in 64-bit fixed point (fix64.cuh); what is left in FP64 is about 20
// instructions a stencil point.  beta enters as 57-bit integers relative to the node's largest.
template <typename P, typename V, typename R, bool POS>
__device__ __forceinline__ int bwd_u_solve64(const BwdArgs &b, int Iu, int Ju, const R g[8], const int tri[3],
                                             const int *us, int nu, const unsigned vm[3], const int vi[3],
                                             R *uw, R *udx, R *udy)
{
    const P2MArgs &a = b.f;
    const int nc = a.n - 1;
    longlong2 o[UMAX];
    const int L = node_offsets64<P>(a.pos, Iu, Ju, nc, us, nu, o);
    if (L == NOT_FINITE) return -PFEM_DEFER;
    long long bi[POS ? UMAX : 1];
    double lbar[3] = {0.0, 0.0, 0.0}, bunit = 0.0;
    if (POS) {
        double bm = 0.0;
        bool bad = false;
        auto beta = [&](int i) {
            R v[8];
            load_vals<V, R>((const V *)a.vals, a.perm, us[i], a.C, v);
            R t = R(0);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < a.C) t = fma(g[c], v[c], t);
            return (double)t;
        };
        for (int i = 0; i < nu; ++i) {
            const double t = beta(i);
            bad |= !(fabs(t) < 1e290);           // infinities and NaN: left to the fix pass in FP64
            bm = fmax(bm, fabs(t));
            bi[i] = __double_as_longlong(t);
#pragma unroll
            for (int e = 0; e < 3; ++e)
                if (i == vi[e]) lbar[e] = t;
        }
        if (bad) return -PFEM_DEFER;
        // 2^(be - 1022) > bm: beta = bi 2^(be - 1078); without an upstream field beta = 0
        const int be = max((__double2hiint(bm) >> 20) & 0x7ff, 200);
        const double bs = __hiloint2double((1022 + 56 - be + 1023) << 20, 0);
        bunit = __hiloint2double((be - 1022 + 1023) << 20, 0);       // of the scaled beta, 2^56
        for (int i = 0; i < nu; ++i) bi[i] = __double2ll_rn(__longlong_as_double(bi[i]) * bs);
    }
    NodePos<P, R> np;
    np.init(Iu, Ju, nc);
    double d[3][2];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        R x, y;
        np.off(a.pos, tri[e], x, y);
        d[e][0] = (double)x;
        d[e][1] = (double)y;
    }
    const double Na = d[1][0] * d[2][1] - d[1][1] * d[2][0];
    const double Nb = d[2][0] * d[0][1] - d[2][1] * d[0][0];
    const double Nc = d[0][0] * d[1][1] - d[0][1] * d[1][0];
    const double A2 = Na + Nb + Nc;
    const double lam[3] = {Na / A2, Nb / A2, Nc / A2};
    // quadratic part first: it queues nodes
#pragma unroll 1
    for (int e = 0; e < 3; ++e) {
        const int f = e == 2 ? 0 : e + 1;
        EdgeSystem<UMAX> sys(o, vm[e] | vm[f], o[vi[e]], o[vi[f]]);
        long long Y[6], Z[6], u[6] = {0, 0, 0, 0, 0, 0};
        int sy, sz = 0;
        if (!sys.factor(FastTol<float>::v) || !sys.solve_coefficients(Y, sy)) return -PFEM_DEFER;
        const double yu = __hiloint2double((1023 - sy) << 20, 0), ce = 2.0 * lam[e] * lam[f];
        EdgeFix64 Ey, Ez;
        Ey.set(Y);
        if constexpr (!POS) {
            for (unsigned m = sys.mask; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                Split64 X, T;
                sys.coords(i, X, T);
                uw[i] += R(ce * (__ll2double_rn(Ey.value(X, T)) * yu));
            }
        } else {
        for (unsigned m = sys.mask; m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            Split64 X, T;
            sys.coords(i, X, T);
            const Split64 bt = split64(bi[i]);
            const long long bx = mul64(X, bt), by = mul64(T, bt);
            const Split64 xs = split64(bx), ys = split64(by);
            u[0] += bi[i];
            u[1] += bx;
            u[2] += by;
            u[3] += mul64(X, xs);
            u[4] += mul64(T, xs);
            u[5] += mul64(T, ys);
        }
        if (!sys.solve_adjoint(u, Z, sz)) return -PFEM_DEFER;
        Ez.set(Z);
        const double zu = __hiloint2double((1023 - sz) << 20, 0);
        double y[6], z[6], Be = 0.0;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            y[q] = __ll2double_rn(Y[q]) * yu;
            z[q] = __ll2double_rn(Z[q]) * zu;
            Be = fma(__ll2double_rn(u[q]) * W64_UNIT, y[q], Be);
        }
        lbar[e] += 2.0 * lam[f] * Be * bunit;
        lbar[f] += 2.0 * lam[e] * Be * bunit;
        // X' = position * 2^(L + k + 1)
        const double cp = ce * bunit * __hiloint2double((1023 + L + sys.k + 1) << 20, 0);
        for (unsigned m = sys.mask; m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            Split64 X, T;
            sys.coords(i, X, T);
            const double A = __ll2double_rn(Ey.value(X, T)) * yu, Zi = __ll2double_rn(Ez.value(X, T)) * zu;
            uw[i] += R(ce * A);
            const longlong2 p = o[i];
            const double x = __ll2double_rn((2 * p.x - sys.mx) << sys.k) * 5.421010862427522e-20;   // 2^-64
            const double t = __ll2double_rn((2 * p.y - sys.my) << sys.k) * 5.421010862427522e-20;
            const double q = cp * (__ll2double_rn(bi[i]) * W64_UNIT - Zi), Aq = cp * A;
            const double x2 = 2.0 * x, t2 = 2.0 * t;
            udx[i] += R(q * fma(x2, y[3], fma(t, y[4], y[1])) - Aq * fma(x2, z[3], fma(t, z[4], z[1])));
            udy[i] += R(q * fma(t2, y[5], fma(x, y[4], y[2])) - Aq * fma(t2, z[5], fma(x, z[4], z[2])));
        }
        // b' = -(1/2) (E'x^2, E'x E'y, E'y^2), E' = X' of the first end less that of the second
        const double Ex = __ll2double_rn(sys.dx << sys.k) * 1.0842021724855044e-19;    // 2^-63: 2 X' of the first
        const double Et = __ll2double_rn(sys.dy << sys.k) * 1.0842021724855044e-19;
        const double exb = -cp * (Ex * z[3] + 0.5 * Et * z[4]);
        const double eyb = -cp * (0.5 * Ex * z[4] + Et * z[5]);
        udx[vi[e]] += R(exb);
        udy[vi[e]] += R(eyb);
        udx[vi[f]] -= R(exb);
        udy[vi[f]] -= R(eyb);
        }
    }
    for (int e = 0; e < 3; ++e) uw[vi[e]] += R(lam[e]);
    if (POS) {
        // lambda_k = N_k / A2 with N_a = d_b x d_c, N_b = d_c x d_a, N_c = d_a x d_b
        const double Lam = lbar[0] * lam[0] + lbar[1] * lam[1] + lbar[2] * lam[2];
        const double n0 = (lbar[0] - Lam) / A2, n1 = (lbar[1] - Lam) / A2, n2 = (lbar[2] - Lam) / A2;
        udx[vi[0]] += R(n2 * d[1][1] - n1 * d[2][1]);
        udy[vi[0]] += R(n1 * d[2][0] - n2 * d[1][0]);
        udx[vi[1]] += R(n0 * d[2][1] - n2 * d[0][1]);
        udy[vi[1]] += R(n2 * d[0][0] - n0 * d[2][0]);
        udx[vi[2]] += R(n1 * d[0][1] - n0 * d[1][1]);
        udy[vi[2]] += R(n0 * d[1][0] - n1 * d[0][0]);
    }
    return 0;
}

// Linear shape functions: the triangle's vertices are the entries.
template <typename P, typename V, typename R, bool POS>
__global__ void __launch_bounds__(STAR_TPB, PFEM_LINEAR_MIN_BLOCKS) k_bwd_linear(BwdArgs b)
{
    __shared__ __align__(16) unsigned char lists[HullList::BYTES];
    const P2MArgs &a = b.f;
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    const int nc = a.n - 1;
    const bool mesh = I <= nc && J <= nc;
    const int Iu = I >= nc ? 0 : I, Ju = J >= nc ? 0 : J;
    const long long node = (long long)J * a.n + I;
    R g[8];
    bool any = false;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        g[c] = mesh && c < a.C ? load_val<V, R>((const V *)b.grad_mesh + node * a.C + c) : R(0);
        any |= g[c] != R(0);
    }
    int us[3];
    R uw[3] = {R(0), R(0), R(0)}, ub[3], udx[3] = {R(0), R(0), R(0)}, udy[3] = {R(0), R(0), R(0)};
    int nu = 0;
    int st = locate_hull(a.B, any, make_uint2(node_fx(Iu, nc), node_fx(Ju, nc)), a.R0,
                         HullList::at(lists, threadIdx.x), us);       // every lane of the warp
    if (any) {
        if (st == 0) {
            NodePos<P, R> np;
            np.init(Iu, Ju, nc);
            const int vi[3] = {0, 1, 2};
            const unsigned vm[3] = {0u, 0u, 0u};
            bwd_u_solve<P, V, R, R, PFEM_SHAPE_LINEAR, POS>(b, np, g, us, us, 3, vm, vi, uw, ub, udx, udy);
            nu = 3;
        } else {
            st = defer_or_error(a, st, node);
            if (st < 0) record_error(a.status, -st, node);
        }
    }
    if (mesh) write_entries<R, R, POS>(b, node, nu, us, uw, udx, udy);
}

// ---------------------------------------------------------------- node records
// The adjoint runs the table path as two kernels, each with its own register budget: k_p2m_geom
// locates the node and builds its particle set from the star table (memory latency bound), and
// the adjoint's solve kernel reads what it found from a per-node record, one array per field so
// that both kernels access it coalesced.  The forward solves run both halves in k_p2m_tab.
struct NodeRecs {
    int *meta;          // [nodes] nu | vi0 << 5 | vi1 << 10 | vi2 << 15, or -1: no record
    unsigned *mask;     // [3][nodes] vm[e]
    int *us;            // [UMAX][nodes] slots of the particle set
    long long nodes;
};

// Lays the record arrays for `nodes` nodes out from `base` (256-byte aligned arrays; base may be
// null to size them); returns the bytes they take.
inline size_t node_recs_layout(char *base, long long nodes, NodeRecs *r)
{
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_meta = 0;
    const size_t o_mask = al(o_meta + sizeof(int) * (size_t)nodes);
    const size_t o_us = al(o_mask + 3 * sizeof(unsigned) * (size_t)nodes);
    const size_t total = al(o_us + UMAX * sizeof(int) * (size_t)nodes);
    if (base) {
        r->meta = (int *)(base + o_meta);
        r->mask = (unsigned *)(base + o_mask);
        r->us = (int *)(base + o_us);
    }
    r->nodes = nodes;
    return total;
}

// Resident 128-thread blocks per SM of the geometry kernel: its node search waits on memory, and
// its particle sets in shared memory and registers want room (the whole gradient step at 1025^2
// nodes / 2048^2 particles, C = 1, FP32, with 6, 8, 10, 12 blocks: 2395, 2369, 2372, 2391 us).
#ifndef PFEM_GEOM_MIN_BLOCKS
#define PFEM_GEOM_MIN_BLOCKS 8
#endif
// Node (I, J) of the mesh of a.n nodes per side: locate it and build its particle set from the
// star table, and write its record at index J * a.n + I.
__device__ __forceinline__ void geom_node(const P2MArgs &a, const StarTab &t, const NodeRecs &r, int I, int J,
                                          int *su, int stride)
{
    const int nc = a.n - 1;
    const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
    const long long rec = (long long)J * a.n + I;
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
    int meta = -1, nu = 0;
    unsigned vm[3] = {0u, 0u, 0u};
    const bool small = warp_sets8<1>(t, st, tri, sa, a.ucap, su, stride, nu, vm);
    if (st == 0) {
        int vi[3] = {0, 1, 2};
        auto write = [&](auto us) {
            // entries up to the warp's largest set, -1 past this node's, so that the warp's
            // stores to each entry array cover contiguous runs of it
            const int nw = __reduce_max_sync(__activemask(), nu);
            for (int i = 0; i < nw; ++i) r.us[i * r.nodes + rec] = i < nu ? us[i] : -1;
#pragma unroll
            for (int e = 0; e < 3; ++e) r.mask[e * r.nodes + rec] = vm[e];
            meta = nu | vi[0] << 5 | vi[1] << 10 | vi[2] << 15;
        };
        if (small) {
            write(Strided<int>{su, stride});
        } else {
            int us[UMAX];
            if (node_u_sets<UMAX>(tri, sa, us, nu, vm, vi, min(a.ucap, UMAX)) != 0)
                st = a.defer_cap > 0 ? -PFEM_DEFER : -PFEM_ERR_CAPACITY;
            else
                write(Strided<int>{us, 1});
        }
    }
    r.meta[rec] = meta;
    if (st != 0) {
        st = defer_or_error(a, st, rec);
        if (st < 0) record_error(a.status, -st, rec);
    }
}

__global__ void __launch_bounds__(128, PFEM_GEOM_MIN_BLOCKS) k_p2m_geom(P2MArgs a, StarTab t, NodeRecs r)
{
    __shared__ int su[SET_W * 128];
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    if (I >= a.n || J >= a.n) return;
    geom_node(a, t, r, I, J, su + threadIdx.x, 128);
}

// The quadratic adjoint as two kernels: k_p2m_geom writes each node's record (particle set, stencil
// masks), this kernel solves the adjoint of the three edge systems with its own register budget
// and writes the node's entries.
template <typename P, typename V, typename R, typename S, bool POS>
__global__ void __launch_bounds__(128, 4) k_bwd_solve(BwdArgs b, NodeRecs r)
{
    const P2MArgs &a = b.f;
    const long long node = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (node >= r.nodes) return;
    R g[8];
    bool any = false;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        g[c] = c < a.C ? load_val<V, R>((const V *)b.grad_mesh + node * a.C + c) : R(0);
        any |= g[c] != R(0);
    }
    int us[UMAX];
    R uw[UMAX], udx[UMAX], udy[UMAX];
    int nu = 0;
    const int meta = r.meta[node];
    if (any && meta >= 0) {
        nu = meta & 31;
        const int vi[3] = {(meta >> 5) & 31, (meta >> 10) & 31, (meta >> 15) & 31};
        if (nu > b.K) {
            record_error(a.status, PFEM_ERR_CAPACITY, node);
            nu = 0;
        } else {
            for (int i = 0; i < nu; ++i) {
                us[i] = r.us[i * r.nodes + node];
                uw[i] = udx[i] = udy[i] = R(0);
            }
            unsigned vm[3];
            int tri[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                vm[e] = r.mask[e * r.nodes + node];
                tri[e] = us[vi[e]];
            }
            const int nc = a.n - 1;
            const int I = (int)(node % a.n), J = (int)(node / a.n);
            int st;
            if constexpr (sizeof(S) == 8) {
                st = bwd_u_solve64<P, V, R, POS>(b, I == nc ? 0 : I, J == nc ? 0 : J, g, tri, us, nu, vm, vi,
                                                 uw, udx, udy);
            } else {
                NodePos<P, R> np;
                np.init(I == nc ? 0 : I, J == nc ? 0 : J, nc);
                R ub[UMAX];
                st = bwd_u_solve<P, V, R, S, PFEM_SHAPE_QUADRATIC, POS>(b, np, g, tri, us, nu, vm, vi, uw, ub,
                                                                       udx, udy);
            }
            if (st != 0) {
                st = defer_or_error(a, st, node);
                if (st < 0) record_error(a.status, -st, node);
                nu = 0;
            }
        }
    }
    write_entries<R, R, POS>(b, node, nu, us, uw, udx, udy);
}

// ---------------------------------------------------------------- fix pass
// The nodes the fast adjoint queued (an edge system below the forward's fast-solve tolerance,
// more particles than the fast pass holds, or a search that ran out of its region), recomputed
// in FP64 with the forward fix pass's geometry (widest search radius) and SVD solve.  For each
// edge, with P the 6 x k monomial matrix (the stencil in the edge frame), A = P^+ b its
// pseudo-inverse solution and Abar = c_e beta, the reverse-mode derivative of the pseudo-inverse
// at constant rank (Golub & Pereyra 1973) gives
//   Pbar = -u A^T + r (P^+ u)^T + z ((I - P^+ P) Abar)^T,   bbar = u,
// with u = P^+T Abar, z = P^+T A and r = b - P A (zero unless the system is inconsistent, as
// for a stencil of five particles).  A least-squares solution depends on the edge frame, so the
// frame's dependence on the edge endpoints (midpoint m, length s) is differentiated too.

// One edge.  pt: the k members' monomial rows (overwritten), x/y their frame coordinates,
// beta their gbar . alpha, b, ce = 2 lambda_nu lambda_sg.  Out: A (coefficients), xb/yb the
// adjoints of the members' frame coordinates, bb the adjoint of b, and Be = sum beta A.
static __device__ __noinline__ void edge_adjoint_svd(int k, double (*pt)[6], const double *x,
                                                     const double *y, const double *beta,
                                                     const double b[6], double ce, double *A,
                                                     double *xb, double *yb, double bb[6],
                                                     double &Be)
{
    double V[6][6], sig2[6];
    jacobi_svd(k, pt, V, sig2);
    const double thr2 = svd_threshold2(k, sig2);
    double vb[6], wA[6], wAA[6];
    for (int j = 0; j < 6; ++j) {
        double d = 0.0;
        for (int r = 0; r < 6; ++r) d = fma(V[r][j], b[r], d);
        vb[j] = sig2[j] > thr2 ? d : 0.0;
    }
    Be = 0.0;
    for (int i = 0; i < k; ++i) {
        double a = 0.0;
        for (int j = 0; j < 6; ++j)
            if (sig2[j] > thr2) a = fma(vb[j] / sig2[j], pt[i][j], a);
        A[i] = a;
        Be = fma(beta[i], a, Be);
    }
    for (int j = 0; j < 6; ++j) {
        double s1 = 0.0, s2 = 0.0;
        for (int i = 0; i < k; ++i) {
            s1 = fma(pt[i][j], ce * beta[i], s1);
            s2 = fma(pt[i][j], A[i], s2);
        }
        wA[j] = sig2[j] > thr2 ? s1 / sig2[j] : 0.0;    // (w_j . Abar) / sigma_j^2
        wAA[j] = sig2[j] > thr2 ? s2 / sig2[j] : 0.0;   // (w_j . A) / sigma_j^2
    }
    double u[6], z[6], r[6];
    for (int q = 0; q < 6; ++q) {
        double su = 0.0, sz = 0.0, sr = b[q];
        for (int j = 0; j < 6; ++j) {
            su = fma(V[q][j], wA[j], su);
            sz = fma(V[q][j], wAA[j], sz);
            sr = fma(-V[q][j], vb[j], sr);
        }
        u[q] = su;
        z[q] = sz;
        r[q] = sr;
        bb[q] = su;
    }
    for (int i = 0; i < k; ++i) {
        double pu = 0.0, pp = 0.0;
        for (int j = 0; j < 6; ++j)
            if (sig2[j] > thr2) {
                pu = fma(pt[i][j], wA[j] / sig2[j], pu);
                pp = fma(pt[i][j], wA[j], pp);
            }
        const double qi = ce * beta[i] - pp;              // ((I - P^+ P) Abar)_i
        double pb[6];
        for (int q = 0; q < 6; ++q) pb[q] = -u[q] * A[i] + r[q] * pu + z[q] * qi;
        xb[i] = pb[1] + 2.0 * x[i] * pb[3] + y[i] * pb[4];
        yb[i] = pb[2] + x[i] * pb[4] + 2.0 * y[i] * pb[5];
    }
}

// With CHOL (FP64 systems) a node first takes the FP64 Cholesky form of the adjoint, down to FP64's
// pivot tolerance: it is queued where the FP32 factor cannot carry the fixed-point refinement.
template <typename P, typename V, typename R, int SHAPE, bool POS, bool CHOL>
__global__ void __launch_bounds__(64) k_bwd_fix(BwdArgs b)
{
    const P2MArgs &a = b.f;
    const int cnt = min(*a.defer_count, a.defer_cap);
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < cnt; it += gridDim.x * blockDim.x) {
        const long long node = a.defer_list[it];
        const int I = (int)(node % a.n), J = (int)(node / a.n);
        const int nc = a.n - 1;
        const int Iu = I == nc ? 0 : I, Ju = J == nc ? 0 : J;
        double g[8];
        for (int c = 0; c < 8; ++c)
            g[c] = c < a.C ? (double)load_val<V, R>((const V *)b.grad_mesh + node * a.C + c) : 0.0;
        constexpr int UM = UMAX_SVD;
        int us[UM];
        double uw[UM], ub[UM], udx[UM], udy[UM];
        int nu = 0, vi[3], tri[3];
        unsigned vm[3] = {0u, 0u, 0u};
        const uint2 qn = make_uint2(node_fx(Iu, nc), node_fx(Ju, nc));
        int stars[3][KMAX];
        int ns[3] = {0, 0, 0};
        int st = locate(a.B, qn, a.R0, tri, stars[0], ns[0]);
        if (SHAPE == PFEM_SHAPE_QUADRATIC)
            for (int e = 0; e < 3 && st == 0; ++e)
                if (ns[e] == 0) {
                    const int c = star_of(a.B, tri[e], a.R0, stars[e]);
                    if (c < 0) st = c;
                    else ns[e] = c;
                }
        if (st == 0) {
            bool over = false;
            auto add = [&](int s) -> int {
                for (int i = 0; i < nu; ++i)
                    if (us[i] == s) return i;
                if (nu == UM || nu == b.K) { over = true; return 0; }
                us[nu] = s;
                uw[nu] = udx[nu] = udy[nu] = 0.0;
                return nu++;
            };
            for (int e = 0; e < 3; ++e) vi[e] = add(tri[e]);
            if (SHAPE == PFEM_SHAPE_QUADRATIC)
                for (int e = 0; e < 3; ++e) {
                    unsigned m = 1u << vi[e];
                    for (int i = 0; i < ns[e]; ++i) m |= 1u << add(stars[e][i]);
                    vm[e] = m;
                }
            if (over) st = -PFEM_ERR_CAPACITY;
        }
        if constexpr (CHOL) {
            if (st == 0 && nu <= UMAX) {
                NodePos<P, R> np;
                np.init(Iu, Ju, nc);
                R g1[8], w1[UMAX], b1[UMAX], x1[UMAX], y1[UMAX];
                for (int c = 0; c < 8; ++c) g1[c] = (R)g[c];
                for (int k = 0; k < nu; ++k) w1[k] = x1[k] = y1[k] = R(0);
                if (bwd_u_solve<P, V, R, double, SHAPE, POS>(b, np, g1, tri, us, nu, vm, vi, w1, b1, x1, y1) == 0) {
                    write_entries<R, R, POS>(b, node, nu, us, w1, x1, y1);
                    continue;
                }
            }
        }
        if (st == 0) {
            // offsets from the node in FP64 (FP32 positions promoted, as the forward fix pass does)
            NodePos<P, R> np;
            np.init(Iu, Ju, nc);
            double ox[UM], oy[UM];
            for (int i = 0; i < nu; ++i) {
                R dx, dy;
                np.off(a.pos, us[i], dx, dy);
                ox[i] = (double)dx;
                oy[i] = (double)dy;
                R v[8];
                load_vals<V, R>((const V *)a.vals, a.perm, us[i], a.C, v);
                double t = 0.0;
                for (int c = 0; c < 8; ++c)
                    if (c < a.C) t = fma(g[c], (double)v[c], t);
                ub[i] = t;
            }
            double d[3][2];
            for (int e = 0; e < 3; ++e) { d[e][0] = ox[vi[e]]; d[e][1] = oy[vi[e]]; }
            const double Na = d[1][0] * d[2][1] - d[1][1] * d[2][0];
            const double Nb = d[2][0] * d[0][1] - d[2][1] * d[0][0];
            const double Nc = d[0][0] * d[1][1] - d[0][1] * d[1][0];
            const double A2 = Na + Nb + Nc;
            const double lam[3] = {Na / A2, Nb / A2, Nc / A2};
            double lbar[3];
            for (int e = 0; e < 3; ++e) {
                uw[vi[e]] += lam[e];
                lbar[e] = ub[vi[e]];
            }
            if (SHAPE == PFEM_SHAPE_QUADRATIC)
                for (int e = 0; e < 3; ++e) {
                    const int f = e == 2 ? 0 : e + 1;
                    const unsigned mask = vm[e] | vm[f];
                    const double mx = 0.5 * (d[e][0] + d[f][0]), my = 0.5 * (d[e][1] + d[f][1]);
                    const double ex = d[e][0] - d[f][0], ey = d[e][1] - d[f][1];
                    const double sl = sqrt(ex * ex + ey * ey), inv = 1.0 / sl;
                    const double tx = ex * inv, ty = ey * inv;
                    double pt[UM][6], x[UM], y[UM], be[UM], A[UM], xb[UM], yb[UM];
                    int ids[UM];
                    int k = 0;
                    for (unsigned m = mask; m; m &= m - 1) {
                        const int i = __ffs(m) - 1;
                        x[k] = (ox[i] - mx) * inv;
                        y[k] = (oy[i] - my) * inv;
                        pt[k][0] = 1.0; pt[k][1] = x[k]; pt[k][2] = y[k];
                        pt[k][3] = x[k] * x[k]; pt[k][4] = x[k] * y[k]; pt[k][5] = y[k] * y[k];
                        be[k] = ub[i];
                        ids[k++] = i;
                    }
                    const double bv[6] = {0.0, 0.0, 0.0, -0.5 * tx * tx, -0.5 * tx * ty, -0.5 * ty * ty};
                    const double ce = 2.0 * lam[e] * lam[f];
                    double bb[6], Be;
                    edge_adjoint_svd(k, pt, x, y, be, bv, ce, A, xb, yb, bb, Be);
                    for (int j = 0; j < k; ++j) uw[ids[j]] = fma(ce, A[j], uw[ids[j]]);
                    lbar[e] += 2.0 * lam[f] * Be;
                    lbar[f] += 2.0 * lam[e] * Be;
                    if (POS) {
                        // members: x = (o - m) / s; frame: m = (d_e + d_f) / 2, s = |d_e - d_f|
                        double mbx = 0.0, mby = 0.0, sb = 0.0;
                        for (int j = 0; j < k; ++j) {
                            udx[ids[j]] += xb[j] * inv;
                            udy[ids[j]] += yb[j] * inv;
                            mbx -= xb[j] * inv;
                            mby -= yb[j] * inv;
                            sb -= (xb[j] * x[j] + yb[j] * y[j]) * inv;
                        }
                        // b = -(1/2) [tx^2, tx ty, ty^2] with t = (d_e - d_f) / s
                        const double tbx = -tx * bb[3] - 0.5 * ty * bb[4];
                        const double tby = -0.5 * tx * bb[4] - ty * bb[5];
                        const double tt = tbx * tx + tby * ty;
                        const double ebx = (tbx - tt * tx) * inv + sb * tx;
                        const double eby = (tby - tt * ty) * inv + sb * ty;
                        udx[vi[e]] += 0.5 * mbx + ebx;
                        udy[vi[e]] += 0.5 * mby + eby;
                        udx[vi[f]] += 0.5 * mbx - ebx;
                        udy[vi[f]] += 0.5 * mby - eby;
                    }
                }
            if (POS) {
                // lambda_k = N_k / A2 with N_a = d_b x d_c, N_b = d_c x d_a, N_c = d_a x d_b
                const double Lam = lbar[0] * lam[0] + lbar[1] * lam[1] + lbar[2] * lam[2];
                const double n0 = (lbar[0] - Lam) / A2, n1 = (lbar[1] - Lam) / A2,
                             n2 = (lbar[2] - Lam) / A2;
                double gx[3] = {0.0, 0.0, 0.0}, gy[3] = {0.0, 0.0, 0.0};
                gx[1] += n0 * d[2][1];  gy[1] -= n0 * d[2][0];
                gx[2] -= n0 * d[1][1];  gy[2] += n0 * d[1][0];
                gx[2] += n1 * d[0][1];  gy[2] -= n1 * d[0][0];
                gx[0] -= n1 * d[2][1];  gy[0] += n1 * d[2][0];
                gx[0] += n2 * d[1][1];  gy[0] -= n2 * d[1][0];
                gx[1] -= n2 * d[0][1];  gy[1] += n2 * d[0][0];
                for (int e = 0; e < 3; ++e) {
                    udx[vi[e]] += gx[e];
                    udy[vi[e]] += gy[e];
                }
            }
        }
        if (st != 0) {
            if (st == -PFEM_FAR) st = -PFEM_ERR_CAPACITY;
            record_error(a.status, -st, node);
            nu = 0;
        }
        write_entries<R, double, POS>(b, node, nu, us, uw, udx, udy);
    }
}

// ---------------------------------------------------------------- transposed gather
// Two sources of entries: given weights [nodes, K] (-1: unused; entry id = node * K + k), counted by
// k_tr_count, and the entries that the node kernels wrote and counted (id = node << ENTRY_BITS | k).

__global__ void k_tr_count(long long E, const int *__restrict__ slot, int *__restrict__ count,
                           int *__restrict__ rank)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < E;
         e += (long long)gridDim.x * blockDim.x) {
        const int s = slot[e];
        rank[e] = s >= 0 ? atomicAdd(count + s, 1) : -1;
    }
}

__global__ void k_tr_scatter(long long E, const int *__restrict__ slot, const int *__restrict__ rank,
                             const int *__restrict__ start, int *__restrict__ order)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < E;
         e += (long long)gridDim.x * blockDim.x) {
        const int s = slot[e];
        if (s >= 0) order[__ldg(start + s) + rank[e]] = (int)e;
    }
}

__global__ void k_tr_scatter_nodes(long long nodes, const int *__restrict__ cnt, const int *__restrict__ slot,
                                   const int *__restrict__ rank, const int *__restrict__ start,
                                   int *__restrict__ order)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
         i += (long long)gridDim.x * blockDim.x) {
        const int nu = cnt[i];
        for (int k = 0; k < nu; ++k) {
            const long long e = k * nodes + i;
            order[__ldg(start + slot[e]) + rank[e]] = (int)(i << ENTRY_BITS | k);
        }
    }
}

// The ids of one particle's entries in increasing order (arrival order before): f(id) for each.
// Up to 16 are sorted in the thread by insertion, more in place by Shell's method (gaps of Ciura
// 2001): few particles on a fine mesh have hundreds of entries each, and the order in which the nodes'
// warps arrive leaves insertion a quarter of n^2 moves.
template <typename F> __device__ __forceinline__ void in_order(int *order, int n, F &&f)
{
    constexpr int LOCAL = 16;
    if (n <= LOCAL) {
        int v[LOCAL];
        for (int i = 0; i < n; ++i) {
            const int x = order[i];
            int j = i - 1;
            for (; j >= 0 && v[j] > x; --j) v[j + 1] = v[j];
            v[j + 1] = x;
        }
        for (int i = 0; i < n; ++i) f(v[i]);
        return;
    }
    int gap = 1;                                 // 1, 4, 10, 23, 57, 132, then by 2.25
    auto larger = [](int g) { return g == 1 ? 4 : g == 4 ? 10 : g == 10 ? 23 : g == 23 ? 57 : g == 57 ? 132 : g * 2 + g / 4; };
    auto smaller = [](int g) { return g > 132 ? max(132, (g * 4 + 8) / 9) : g == 132 ? 57 : g == 57 ? 23 : g == 23 ? 10 : g == 10 ? 4 : g == 4 ? 1 : 0; };
    while (gap < 1 << 24 && larger(gap) < n) gap = larger(gap);
    for (; gap > 0; gap = smaller(gap))
        for (int i = gap; i < n; ++i) {
            const int x = order[i];
            int j = i - gap;
            for (; j >= 0 && order[j] > x; j -= gap) order[j + gap] = order[j];
            order[j + gap] = x;
        }
    for (int i = 0; i < n; ++i) f(order[i]);
}

// grad_vals[particle] = sum_e w_e gbar_node(e); grad_pos[particle] = sum_e dpos_e.  NODES: the node
// kernels' entries (val: Entry<R> with POS, else R), otherwise given weights (val: R).
template <typename V, typename R, bool NODES, bool POS>
__global__ void k_tr_gather(long long N, int K, long long nodes, int C, const int *__restrict__ start,
                            int *order, const void *__restrict__ val, const V *__restrict__ grad_mesh,
                            const int *__restrict__ perm, V *__restrict__ grad_vals,
                            V *__restrict__ grad_pos)
{
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
         s += (long long)gridDim.x * blockDim.x) {
        R gv[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) gv[c] = R(0);
        R gx = R(0), gy = R(0);
        const int a = __ldg(start + s), b = __ldg(start + s + 1);
        in_order(order + a, b - a, [&](int id) {
            const long long node = NODES ? id >> ENTRY_BITS : id / K;
            const long long e = NODES ? (long long)(id & ((1 << ENTRY_BITS) - 1)) * nodes + node : id;
            R w;
            if constexpr (POS) {
                const Entry<R> v = ((const Entry<R> *)val)[e];
                w = v.w;
                gx += v.dx;
                gy += v.dy;
            } else {
                w = __ldg((const R *)val + e);
            }
            if (grad_vals)
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < C) gv[c] = fma(w, load_val<V, R>(grad_mesh + node * C + c), gv[c]);
        });
        const long long o = perm ? (long long)__ldg(perm + s) : s;
        if (grad_vals)
            for (int c = 0; c < C; ++c) store_val<V, R>(grad_vals + o * C + c, gv[c]);
        if (POS) {
            store_val<V, R>(grad_pos + 2 * o, gx);
            store_val<V, R>(grad_pos + 2 * o + 1, gy);
        }
    }
}

static unsigned grid1(long long work, int threads)
{
    long long b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > num_sms() * 64LL) b = num_sms() * 64LL;
    return (unsigned)b;
}

BwdLayout bwd_layout(int n, long long N, int Kw)
{
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    BwdLayout L;
    L.K = KBWD;
    const int K = Kw > KBWD ? Kw : KBWD;
    const long long E = (long long)n * n * K;
    size_t off = 256;
    L.e_slot = off;  off = al(off + 4 * (size_t)E);
    L.e_val = off;   off = al(off + 24 * (size_t)E);
    L.count = off;   off = al(off + 4 * (size_t)(N + 1));
    L.start = off;   off = al(off + 4 * (size_t)(N + 1));
    L.rank = off;    off = al(off + 4 * (size_t)E);
    L.order = off;   off = al(off + 4 * (size_t)E);
    L.scan = off;    off = al(off + 4 * scan_scratch_ints(N + 1));
    NodeRecs r;
    L.rec = off;     off = al(off + node_recs_layout(nullptr, (long long)n * n, &r));
    L.tab = off;     off = al(off + star_tab_bytes(N));
    L.queue = off;   off = al(off + 8 * (size_t)n * n);
    L.total = off;
    return L;
}

// Phase 2: the transposed index of the entries, whose counts per particle are in L.count, and the
// gather.
template <typename V, typename R>
static cudaError_t gather_nodes(const BwdArgs &b, long long N, int C, const int *perm, void *grad_vals,
                                void *grad_pos, const BwdLayout &L, char *ws, cudaStream_t s)
{
    int *start = (int *)(ws + L.start), *order = (int *)(ws + L.order);
    cudaError_t e = scan_exclusive(b.count, start, N + 1, (int *)(ws + L.scan), s);
    if (e != cudaSuccess) return e;
    k_tr_scatter_nodes<<<grid1(b.nodes, 128), 128, 0, s>>>(b.nodes, b.e_cnt, b.e_slot, b.e_rank, start, order);
    auto go = [&](auto pos) {
        k_tr_gather<V, R, true, decltype(pos)::value><<<grid1(N, 128), 128, 0, s>>>(
            N, b.K, b.nodes, C, start, order, b.e_val, (const V *)b.grad_mesh, perm, (V *)grad_vals,
            (V *)grad_pos);
    };
    if (grad_pos) go(std::true_type());
    else go(std::false_type());
    count_launch(2);
    return cudaGetLastError();
}

// The same from given weights [nodes, K]: the value gradient.
template <typename V, typename R>
static cudaError_t gather_weights(const BwdArgs &b, long long N, int K, int C, const int *w_idx, const R *w,
                                  const int *perm, void *grad_vals, const BwdLayout &L, char *ws,
                                  cudaStream_t s)
{
    const long long E = b.nodes * K;
    int *start = (int *)(ws + L.start), *order = (int *)(ws + L.order);
    cudaError_t e = cudaMemsetAsync(b.count, 0, 4 * (size_t)(N + 1), s);
    if (e != cudaSuccess) return e;
    k_tr_count<<<grid1(E, 256), 256, 0, s>>>(E, w_idx, b.count, b.e_rank);
    count_launch();
    e = scan_exclusive(b.count, start, N + 1, (int *)(ws + L.scan), s);
    if (e != cudaSuccess) return e;
    k_tr_scatter<<<grid1(E, 256), 256, 0, s>>>(E, w_idx, b.e_rank, start, order);
    k_tr_gather<V, R, false, false><<<grid1(N, 128), 128, 0, s>>>(N, K, b.nodes, C, start, order, w,
                                                                  (const V *)b.grad_mesh, perm,
                                                                  (V *)grad_vals, (V *)nullptr);
    count_launch(2);
    return cudaGetLastError();
}

template <typename P, typename V, typename R, typename S, int SHAPE>
static cudaError_t bwd_t(const GeoArgs &g, const int *perm, int C, const void *vals,
                         const void *grad_mesh, void *grad_vals, void *grad_pos, bool checkpoint,
                         const int *w_idx, const void *w, int Kw, const BwdLayout &L, char *ws,
                         cudaStream_t s)
{
    const int K = L.K;
    BwdArgs b;
    b.f.n = g.n;
    b.f.B.q = (const uint2 *)g.q_sorted;
    b.f.B.start = g.cell_start;
    b.f.B.nb = g.nb;
    b.f.B.rmax = g.rmax;
    b.f.B.dmax = g.dmax;
    b.f.B.kcap = g.kcap;
    b.f.B.walk_cap = g.walk_cap;
    b.f.B.last4 = g.N >= 4 ? (int)(g.N - 4) : -1;
    b.f.ucap = g.ucap;
    b.f.R0 = g.R0;
    b.f.pos = g.pos_sorted;
    b.f.perm = perm;
    b.f.vals = vals;
    b.f.C = C;
    b.f.out = nullptr;
    b.f.w_idx = nullptr;
    b.f.w = nullptr;
    b.f.K = 0;
    b.f.status = (DevStatus *)ws;
    b.grad_mesh = grad_mesh;
    b.K = K;
    b.nodes = (long long)g.n * g.n;
    b.e_slot = (int *)(ws + L.e_slot);
    b.e_rank = (int *)(ws + L.rank);
    b.e_val = ws + L.e_val;
    b.count = (int *)(ws + L.count);
    const dim3 grid((g.n + 15) / 16, (g.n + 7) / 8);
    // the nodes' records (quadratic shape functions); a node's entry count takes the place of its
    // record's head, which its thread has read by then
    NodeRecs recs;
    node_recs_layout(ws + L.rec, b.nodes, &recs);
    b.e_cnt = recs.meta;
    // the star table's queue counter sits in the status block, after the status word
    const StarTab tab = star_tab_layout(ws + L.tab, g.N, (int *)(ws + 64));   // (right before the fix-pass counter)
    // the fix-pass queue: its counter in the status block, one entry per node
    b.f.defer_count = (int *)(ws + 68);
    b.f.defer_list = (long long *)(ws + L.queue);
    b.f.defer_cap = (int)std::min(b.nodes, (long long)0x7fffffff);
    auto node_pass = [&](auto pos) {
        constexpr bool POS = decltype(pos)::value;
        cudaMemsetAsync(b.count, 0, 4 * (size_t)(g.N + 1), s);
        if constexpr (SHAPE == PFEM_SHAPE_QUADRATIC) {
            // a star that no node needs may fail unnoticed with FP64 systems, whose adjoint has always
            // looked at the needed ones only: a scratch status word
            DevStatus *st = sizeof(S) == 8 ? (DevStatus *)(ws + 128) : b.f.status;
            launch_star_table(b.f.B, g.R0, g.rmax_far, tab, st, s, 1);     // and the fix-pass counter
            k_p2m_geom<<<grid, 128, 0, s>>>(b.f, tab, recs);
            k_bwd_solve<P, V, R, S, POS><<<(unsigned)((b.nodes + 127) / 128), 128, 0, s>>>(b, recs);
            count_launch(2);
        } else {
            cudaMemsetAsync(b.f.defer_count, 0, sizeof(int), s);
            k_bwd_linear<P, V, R, POS><<<grid, 128, 0, s>>>(b);
            count_launch();
        }
        // the queued nodes: widest search radius, FP64 SVD adjoint
        BwdArgs bf = b;
        bf.f.B.rmax = std::max(g.rmax, g.rmax_far);
        k_bwd_fix<P, V, R, SHAPE, POS, SHAPE == PFEM_SHAPE_QUADRATIC && sizeof(S) == 8><<<num_sms() * 2, 64, 0, s>>>(bf);
        count_launch();
    };
    if (checkpoint) {
        // value gradient straight from the stored weights
        cudaError_t e = gather_weights<V, R>(b, g.N, Kw, C, w_idx, (const R *)w, perm, grad_vals, L, ws, s);
        if (e != cudaSuccess || !grad_pos) return e;
        node_pass(std::true_type());
        return gather_nodes<V, R>(b, g.N, C, perm, nullptr, grad_pos, L, ws, s);
    }
    if (grad_pos) node_pass(std::true_type());
    else node_pass(std::false_type());
    return gather_nodes<V, R>(b, g.N, C, perm, grad_vals, grad_pos, L, ws, s);
}

cudaError_t launch_p2m_backward(const GeoArgs &g, const int *perm, int C, const void *vals,
                                pfem_dtype val_t, pfem_shape shape, pfem_solve solve,
                                bool checkpoint, const int *w_idx, const void *w, int Kw,
                                const void *grad_mesh, void *grad_vals, void *grad_pos,
                                const BwdLayout &L, void *ws, cudaStream_t s)
{
    char *W = (char *)ws;
    const bool q = shape == PFEM_SHAPE_QUADRATIC;
    if (val_t == PFEM_F64) {
        if (q) return bwd_t<double, double, double, double, 1>(g, perm, C, vals, grad_mesh, grad_vals, grad_pos, checkpoint, w_idx, w, Kw, L, W, s);
        return bwd_t<double, double, double, double, 0>(g, perm, C, vals, grad_mesh, grad_vals, grad_pos, checkpoint, w_idx, w, Kw, L, W, s);
    }
    if (!q) return bwd_t<float, float, float, float, 0>(g, perm, C, vals, grad_mesh, grad_vals, grad_pos, checkpoint, w_idx, w, Kw, L, W, s);
    if (solve == PFEM_SOLVE_F64)
        return bwd_t<float, float, float, double, 1>(g, perm, C, vals, grad_mesh, grad_vals, grad_pos, checkpoint, w_idx, w, Kw, L, W, s);
    return bwd_t<float, float, float, float, 1>(g, perm, C, vals, grad_mesh, grad_vals, grad_pos, checkpoint, w_idx, w, Kw, L, W, s);
}

}  // namespace pfem
