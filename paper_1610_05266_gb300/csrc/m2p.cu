// m2p.cu -- mesh-to-particle interpolation (Sec. 2.2 eq. m2p) with linear FE shape functions
// on the fixed structured mesh, in the caller's particle order.
//
// The particle's cell (i, j) comes from its fixed-point coordinates (the same rule that bins
// the particles); local coordinates s = x/H - i, t = y/H - j select the triangle of the cell
// split along (i,j)->(i+1,j+1).  With hi = max(s, t), lo = min(s, t) the weights are 1 - hi on node
// (i,j), lo on (i+1,j+1) and hi - lo on (i+1,j) where s >= t, on (i,j+1) where s < t.
// Because the image row and column are stored, i+1 and j+1 never wrap.  The kernel is a
// bandwidth-bound gather: positions and outputs stream once; the mesh is read through L2.
#include <cmath>
#include <type_traits>

#include "internal.h"
#include "m2p.cuh"

namespace pfem {

// Particles a thread, 256 apart: their loads are in flight together.  8192^2 particles of one BF16
// component 632 -> 314 us with four (their bytes take 104 us), 1254^2 of three FP32 ones 18 -> 13
// us with two; the round trip of four FP32 ones at 1025^2 / 2048^2 1061 us with one and 1057 with two;
// four FP64 ones keep enough in flight with one.  FP64 positions in fixed point (m2p.cuh): 1024^2 of three 63 -> 26 us.
template <typename P, typename V, typename R, int CT, int U, bool FINE>
__global__ void __launch_bounds__(256) k_m2p(int n, long long N, const P *__restrict__ pos,
                                             int Crt, const V *__restrict__ mesh,
                                             V *__restrict__ vals)
{
    const long long m0 = blockIdx.x * (256LL * U) + threadIdx.x;
    m2p_particles<P, V, R, CT, U, FINE>(n, m0, N, pos, Crt, mesh, vals);
}

template <typename P, typename V, typename R>
static cudaError_t m2p_t(int n, long long N, const void *pos, int C, const void *mesh, void *vals,
                         cudaStream_t s)
{
    const bool aligned = ((reinterpret_cast<uintptr_t>(mesh) | reinterpret_cast<uintptr_t>(vals)) & 15) == 0;
    auto go = [&](auto ct, auto u) {
        constexpr int CT = decltype(ct)::value, U = decltype(u)::value;
        auto launch = [&](auto fine) {
            k_m2p<P, V, R, CT, U, decltype(fine)::value><<<(unsigned)((N + 256 * U - 1) / (256 * U)), 256, 0, s>>>(
                n, N, (const P *)pos, C, (const V *)mesh, (V *)vals);
        };
        // FP64 positions on fine meshes: another look at those near the origin (m2p.cuh), which costs the
        // others 4 % (2048^2 particles of one component on 1025^2 nodes 73 us, 76 with it)
        if (sizeof(P) == 8 && n > 2049) launch(std::integral_constant<bool, sizeof(P) == 8>());
        else launch(std::false_type());
    };
    // the components in registers up to four; four FP32 ones as one 16-byte access when the arrays
    // allow it
    if (C == 1) go(std::integral_constant<int, 1>(), std::integral_constant<int, 4>());
    else if (C == 2) go(std::integral_constant<int, 2>(), std::integral_constant<int, 4>());
    else if (C == 3) go(std::integral_constant<int, 3>(), std::integral_constant<int, 2>());
    else if (C == 4 && (aligned || sizeof(V) != 4)) go(std::integral_constant<int, 4>(), std::integral_constant<int, sizeof(R) == 8 ? 1 : 2>());
    else go(std::integral_constant<int, 0>(), std::integral_constant<int, 1>());
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_m2p(int n, long long N, const void *pos, pfem_dtype pos_t, int C,
                       const void *mesh, void *vals, pfem_dtype val_t, cudaStream_t s)
{
    if (N == 0) return cudaSuccess;
    if (val_t == PFEM_F64) {
        if (pos_t == PFEM_F64) return m2p_t<double, double, double>(n, N, pos, C, mesh, vals, s);
        return m2p_t<float, double, double>(n, N, pos, C, mesh, vals, s);
    }
    if (val_t == PFEM_F32) {
        if (pos_t == PFEM_F64) return m2p_t<double, float, float>(n, N, pos, C, mesh, vals, s);
        return m2p_t<float, float, float>(n, N, pos, C, mesh, vals, s);
    }
    if (pos_t == PFEM_F64) return m2p_t<double, __nv_bfloat16, float>(n, N, pos, C, mesh, vals, s);
    return m2p_t<float, __nv_bfloat16, float>(n, N, pos, C, mesh, vals, s);
}

// ---------------------------------------------------------------- adjoint of M2P

// grad_mesh[node] = sum over particles whose triangle uses this stored node of w * gbar.
// One thread per stored node; particles of the (up to four) cells around it are visited in
// bin order, so the sum order is fixed (no atomics).  Stored image entries receive only the
// reads that the forward made from them.
template <typename P, typename V, typename R>
__global__ void __launch_bounds__(128) k_m2p_bwd_mesh(int n, int nb, const P *__restrict__ pos,
                                                      const int *__restrict__ cell_start,
                                                      const int *__restrict__ perm, int C,
                                                      const V *__restrict__ gv,
                                                      V *__restrict__ gm)
{
    const int I = blockIdx.x * 16 + (threadIdx.x & 15);
    const int J = blockIdx.y * 8 + (threadIdx.x >> 4);
    if (I >= n || J >= n) return;
    const int nc = n - 1;
    const long long node = (long long)J * n + I;
    R acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = R(0);
    for (int cj = J - 1; cj <= J; ++cj) {
        if (cj < 0 || cj >= nc) continue;
        const long long ylo = bin_lo(cj, nc), yhi = bin_lo(cj + 1, nc);
        const int by0 = bin_of((uint32_t)ylo, nb), by1 = bin_of((uint32_t)(yhi - 1), nb);
        for (int ci = I - 1; ci <= I; ++ci) {
            if (ci < 0 || ci >= nc) continue;
            const long long xlo = bin_lo(ci, nc), xhi = bin_lo(ci + 1, nc);
            const int bx0 = bin_of((uint32_t)xlo, nb), bx1 = bin_of((uint32_t)(xhi - 1), nb);
            for (int by = by0; by <= by1; ++by) {
                const int s0 = __ldg(cell_start + (long long)by * nb + bx0);
                const int s1 = __ldg(cell_start + (long long)by * nb + bx1 + 1);
                for (int s = s0; s < s1; ++s) {
                    const int m = __ldg(perm + s);
                    P px, py;
                    load_pos(pos, m, px, py);
                    int i, j;
                    cell_index(px, py, nc, i, j);
                    if (i != ci || j != cj) continue;
                    const MeshCell<R> c = mesh_cell<P, R>(px, py, n);
                    const R w = node == c.n00 ? c.w0 : node == c.n00 + c.mid ? c.w1 : node == c.n00 + n + 1 ? c.w2 : R(0);
                    if (w == R(0)) continue;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k < C) acc[k] = fma(w, load_val<V, R>(gv + (long long)m * C + k), acc[k]);
                }
            }
        }
    }
    for (int c = 0; c < C; ++c) store_val<V, R>(gm + node * C + c, acc[c]);
}

// grad_pos[m] = sum_c gbar_c * grad f_c(r_m), f the linear FE interpolant of the mesh field.
template <typename P, typename V, typename R>
__global__ void __launch_bounds__(256) k_m2p_bwd_pos(int n, long long N, const P *__restrict__ pos,
                                                     int C, const V *__restrict__ mesh,
                                                     const V *__restrict__ gv, V *__restrict__ gp)
{
    const int nc = n - 1;
    for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < N;
         m += (long long)gridDim.x * blockDim.x) {
        P px, py;
        load_pos(pos, m, px, py);
        int i, j;
        const bool below = cell_index(px, py, nc, i, j);
        const long long n00 = (long long)j * n + i, n10 = n00 + 1, n11 = n00 + n + 1, n01 = n00 + n;
        R gx = R(0), gy = R(0);
        for (int c = 0; c < C; ++c) {
            const R g = load_val<V, R>(gv + m * C + c);
            const R f00 = load_val<V, R>(mesh + n00 * C + c), f10 = load_val<V, R>(mesh + n10 * C + c);
            const R f11 = load_val<V, R>(mesh + n11 * C + c), f01 = load_val<V, R>(mesh + n01 * C + c);
            R ds, dt;
            if (below) { ds = f10 - f00; dt = f11 - f10; }
            else        { ds = f11 - f01; dt = f01 - f00; }
            gx = fma(g, ds, gx);
            gy = fma(g, dt, gy);
        }
        store_val<V, R>(gp + 2 * m, gx * (R)nc);
        store_val<V, R>(gp + 2 * m + 1, gy * (R)nc);
    }
}

template <typename P, typename V, typename R>
static cudaError_t m2p_bwd_t(int n, int nb, long long N, const void *pos, const int *cell_start,
                             const int *perm, int C, const void *mesh, const void *gv, void *gm,
                             void *gp, cudaStream_t s)
{
    k_m2p_bwd_mesh<P, V, R><<<dim3((n + 15) / 16, (n + 7) / 8), 128, 0, s>>>(
        n, nb, (const P *)pos, cell_start, perm, C, (const V *)gv, (V *)gm);
    count_launch();
    if (gp && N > 0) {
        long long blocks = (N + 255) / 256;
        if (blocks > num_sms() * 16LL) blocks = num_sms() * 16LL;
        k_m2p_bwd_pos<P, V, R><<<(unsigned)blocks, 256, 0, s>>>(n, N, (const P *)pos, C,
                                                               (const V *)mesh, (const V *)gv,
                                                               (V *)gp);
        count_launch();
    }
    return cudaGetLastError();
}

cudaError_t launch_m2p_backward(int n, int nb, long long N, const void *pos, pfem_dtype pos_t,
                                const int *cell_start, const int *perm, int C, const void *mesh,
                                const void *gv, pfem_dtype val_t, void *gm, void *gp,
                                cudaStream_t s)
{
    if (val_t == PFEM_F64) {
        if (pos_t == PFEM_F64) return m2p_bwd_t<double, double, double>(n, nb, N, pos, cell_start, perm, C, mesh, gv, gm, gp, s);
        return m2p_bwd_t<float, double, double>(n, nb, N, pos, cell_start, perm, C, mesh, gv, gm, gp, s);
    }
    if (pos_t == PFEM_F64) return m2p_bwd_t<double, float, float>(n, nb, N, pos, cell_start, perm, C, mesh, gv, gm, gp, s);
    return m2p_bwd_t<float, float, float>(n, nb, N, pos, cell_start, perm, C, mesh, gv, gm, gp, s);
}

// ---------------------------------------------------------------- M2P with mesh QCSF
// Quadratically consistent mesh shape functions (App. B on the fixed mesh; the paper's
// projFEM6/projFEMq interpolate mesh -> particles with them, Table 1, and compute their
// coefficients once, Sec. 3.1).  With every cell split along (i,j)->(i+1,j+1), node (I,J) has
// neighbours (I+-1,J), (I,J+-1), (I+1,J+1), (I-1,J-1); an edge's stencil is the closed
// neighbourhood of both endpoints (10 nodes) and its minimum-norm coefficients depend only
// on the edge's direction.  For the triangle of a cell the host folds the three
// edges into one table: the coefficient of each stencil node in each edge.  Then
//   w_k = lambda_k [k vertex] + sum_e 2 lambda_P(e) lambda_Q(e) A_{k,e}.
// Node values are read at the unique nodes (I mod (n-1), J mod (n-1)).
//
// The triangle above the diagonal is the one below it with x and y exchanged, so the kernel
// works in coordinates (hi, lo) = (max, min) of the particle's cell coordinates, with vertices
// (0,0), (1,0), (1,1) and one table for both: its index is the same in every lane and the
// coefficients are operands from the constant bank.  (Two tables chosen per lane made every
// table read a divergent constant load: 140 us for 2048^2 particles on 1025^2 nodes, C = 4, FP32.)

// The 12 nodes around the triangle: its vertices, then the rest of their neighbours.
constexpr int MQ_NODES = 12;
__host__ __device__ constexpr int mq_x(int k)
{
    constexpr int X[MQ_NODES] = {0, 1, 1, 0, -1, 0, -1, 2, 1, 2, 1, 2};
    return X[k];
}
__host__ __device__ constexpr int mq_y(int k)
{
    constexpr int Y[MQ_NODES] = {0, 0, 1, 1, 0, -1, -1, 0, -1, 1, 2, 2};
    return Y[k];
}

// Is node k in the stencil of edge e?  (All but the two neighbours that only the vertex opposite
// the edge has.)
__host__ __device__ constexpr bool mq_in(int k, int e)
{
    return e == 0 ? k != 10 && k != 11 : e == 1 ? k != 4 && k != 6 : k != 7 && k != 8;
}

template <typename R> struct MQTable {
    R A[MQ_NODES][3];           // coefficient of node k in edge e, which joins vertices e and e + 1
};

// Minimum-norm coefficients of the mesh edge from (0,0) to (ex,ey) over its 10-node
// stencil, by the 6x6 normal equations (FP64 Cholesky).
static int mesh_edge_host(int ex, int ey, int S[16][2], double A[16])
{
    static const int NB[6][2] = {{1, 0}, {0, 1}, {-1, 0}, {0, -1}, {1, 1}, {-1, -1}};
    int k = 0;
    const int ends[2][2] = {{0, 0}, {ex, ey}};
    for (int e = 0; e < 2; ++e)
        for (int m = -1; m < 6; ++m) {
            const int x = ends[e][0] + (m < 0 ? 0 : NB[m][0]);
            const int y = ends[e][1] + (m < 0 ? 0 : NB[m][1]);
            bool dup = false;
            for (int i = 0; i < k; ++i) dup |= S[i][0] == x && S[i][1] == y;
            if (!dup) { S[k][0] = x; S[k][1] = y; ++k; }
        }
    const double s = std::sqrt((double)(ex * ex + ey * ey));
    double P[16][6], M[6][6] = {{0}};
    for (int i = 0; i < k; ++i) {
        const double x = (S[i][0] - 0.5 * ex) / s, y = (S[i][1] - 0.5 * ey) / s;
        const double p[6] = {1, x, y, x * x, x * y, y * y};
        for (int r = 0; r < 6; ++r) {
            P[i][r] = p[r];
            for (int c = 0; c < 6; ++c) M[r][c] += p[r] * p[c];
        }
    }
    const double tx = ex / s, ty = ey / s;
    double b[6] = {0, 0, 0, -0.5 * tx * tx, -0.5 * tx * ty, -0.5 * ty * ty};
    double L[6][6] = {{0}};
    for (int j = 0; j < 6; ++j) {
        double d = M[j][j];
        for (int q = 0; q < j; ++q) d -= L[j][q] * L[j][q];
        L[j][j] = std::sqrt(d);
        for (int i = j + 1; i < 6; ++i) {
            double t = M[i][j];
            for (int q = 0; q < j; ++q) t -= L[i][q] * L[j][q];
            L[i][j] = t / L[j][j];
        }
    }
    double z[6], y[6];
    for (int r = 0; r < 6; ++r) {
        double t = b[r];
        for (int q = 0; q < r; ++q) t -= L[r][q] * z[q];
        z[r] = t / L[r][r];
    }
    for (int r = 5; r >= 0; --r) {
        double t = z[r];
        for (int q = r + 1; q < 6; ++q) t -= L[q][r] * y[q];
        y[r] = t / L[r][r];
    }
    for (int i = 0; i < k; ++i) {
        double a = 0;
        for (int r = 0; r < 6; ++r) a += P[i][r] * y[r];
        A[i] = a;
    }
    return k;
}

template <typename R> static MQTable<R> build_mq_table()
{
    MQTable<R> T;
    const int E[3][4] = {{0, 0, 1, 0}, {1, 0, 0, 1}, {0, 0, 1, 1}};     // origin and direction
    for (int e = 0; e < 3; ++e) {
        int S[16][2];
        double A[16];
        const int K = mesh_edge_host(E[e][2], E[e][3], S, A);
        for (int k = 0; k < MQ_NODES; ++k) {
            T.A[k][e] = R(0);
            for (int i = 0; i < K; ++i)
                if (S[i][0] + E[e][0] == mq_x(k) && S[i][1] + E[e][1] == mq_y(k)) T.A[k][e] = (R)A[i];
        }
    }
    return T;
}

// built once per process (thread-safe initialisation of a function-local static)
template <typename R> static const MQTable<R> &mq_table()
{
    static const MQTable<R> T = build_mq_table<R>();
    return T;
}

// One particle per thread.  Bound by the L1: twelve gathers a particle, which neighbouring
// particles share; the weights are 30 FMAs with constant operands.  2048^2 particles on 1025^2
// nodes, C = 4, FP32: 49 us (17 us of it is what the bytes take); 58 us before the lanes of both
// triangles read the nodes they share together.
template <typename P, typename V, typename R, int CT>
__global__ void __launch_bounds__(256) k_m2p_q(int n, long long N, const P *__restrict__ pos, int Crt,
                                               const V *__restrict__ mesh, V *__restrict__ vals,
                                               const MQTable<R> T)
{
    const int C = CT > 0 ? CT : Crt;
    const int nc = n - 1;
    for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < N;
         m += (long long)gridDim.x * blockDim.x) {
        P px, py;
        load_pos(pos, m, px, py);
        const MeshCell<R> cell = mesh_cell<P, R>(px, py, n);
        const int i = cell.i, j = cell.j;
        const bool below = cell.mid == 1;
        const R lam[3] = {cell.w0, cell.w1, cell.w2};
        const R ce[3] = {R(2) * lam[0] * lam[1], R(2) * lam[1] * lam[2], R(2) * lam[2] * lam[0]};
        R w[MQ_NODES];
#pragma unroll
        for (int k = 0; k < MQ_NODES; ++k) {
            w[k] = R(0);
#pragma unroll
            for (int e = 0; e < 3; ++e)
                if (mq_in(k, e)) w[k] = fma(T.A[k][e], ce[e], w[k]);
            if (k < 3) w[k] += lam[k];
        }
        // the four columns and rows around the cell (unique nodes)
        int col[4];
        const V *row[4];
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            int I = i + d - 1, J = j + d - 1;
            I += I < 0 ? nc : 0;
            I -= I >= nc ? nc : 0;
            J += J < 0 ? nc : 0;
            J -= J >= nc ? nc : 0;
            col[d] = I * C;
            row[d] = mesh + (long long)J * n * C;
        }
        R acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = R(0);
#pragma unroll
        for (int k = 0; k < MQ_NODES; ++k) {
            // node k of the triangle's own coordinates is read together with its mirror image, so
            // that the lanes of both triangles read the nodes they share in the same instruction
            constexpr int MIRROR[MQ_NODES] = {0, 3, 2, 1, 5, 4, 6, -1, -1, 10, 9, 11};
            const int x = mq_x(k) + 1, y = mq_y(k) + 1;
            const V *mp;
            R wk;
            if (MIRROR[k] >= 0) {
                mp = row[y] + col[x];
                wk = below ? w[k] : w[MIRROR[k]];
            } else {
                mp = below ? row[y] + col[x] : row[x] + col[y];
                wk = w[k];
            }
            if constexpr (CT == 4 && sizeof(V) == 4 && sizeof(R) == 4) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(mp));
                acc[0] = fmaf(wk, v.x, acc[0]);
                acc[1] = fmaf(wk, v.y, acc[1]);
                acc[2] = fmaf(wk, v.z, acc[2]);
                acc[3] = fmaf(wk, v.w, acc[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < C) acc[c] = fma(wk, load_val<V, R>(mp + c), acc[c]);
            }
        }
        if constexpr (CT == 4 && sizeof(V) == 4 && sizeof(R) == 4)
            __stcs(reinterpret_cast<float4 *>(vals) + m, make_float4(acc[0], acc[1], acc[2], acc[3]));
        else
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < C) store_val<V, R>(vals + m * C + c, acc[c]);
    }
}

template <typename P, typename V, typename R>
static cudaError_t m2p_q_t(int n, long long N, const void *pos, int C, const void *mesh, void *vals,
                           cudaStream_t s)
{
    long long blocks = (N + 255) / 256;
    if (blocks > num_sms() * 16LL) blocks = num_sms() * 16LL;
    // the component loop unrolled; four FP32 components as one 16-byte access when the arrays allow it
    // (else the loop over eight with a test each)
    const bool aligned = ((reinterpret_cast<uintptr_t>(mesh) | reinterpret_cast<uintptr_t>(vals)) & 15) == 0;
    auto go = [&](auto ct) {
        k_m2p_q<P, V, R, decltype(ct)::value><<<(unsigned)blocks, 256, 0, s>>>(
            n, N, (const P *)pos, C, (const V *)mesh, (V *)vals, mq_table<R>());
    };
    switch (C == 4 && sizeof(V) == 4 && !aligned ? 0 : C) {
    case 1: go(std::integral_constant<int, 1>()); break;
    case 2: go(std::integral_constant<int, 2>()); break;
    case 3: go(std::integral_constant<int, 3>()); break;
    case 4: go(std::integral_constant<int, 4>()); break;
    case 5: go(std::integral_constant<int, 5>()); break;
    case 6: go(std::integral_constant<int, 6>()); break;
    case 7: go(std::integral_constant<int, 7>()); break;
    case 8: go(std::integral_constant<int, 8>()); break;
    default: go(std::integral_constant<int, 0>());
    }
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_m2p_quadratic(int n, long long N, const void *pos, pfem_dtype pos_t, int C,
                                 const void *mesh, void *vals, pfem_dtype val_t, cudaStream_t s)
{
    if (N == 0) return cudaSuccess;
    if (val_t == PFEM_F64 && pos_t == PFEM_F64) return m2p_q_t<double, double, double>(n, N, pos, C, mesh, vals, s);
    if (val_t == PFEM_F32 && pos_t == PFEM_F32) return m2p_q_t<float, float, float>(n, N, pos, C, mesh, vals, s);
    if (val_t == PFEM_BF16 && pos_t == PFEM_F32) return m2p_q_t<float, __nv_bfloat16, float>(n, N, pos, C, mesh, vals, s);
    return cudaErrorInvalidValue;
}

}  // namespace pfem
