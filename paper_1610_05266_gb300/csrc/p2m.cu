// p2m.cu -- launchers of the particle-to-mesh kernels (fused apply, explicit weights, apply
// from explicit weights) and of the Delaunay-star diagnostic.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "internal.h"
#include "p2m.cuh"

namespace pfem {

// The queue of nodes for the FP64 SVD pass lives in the workspace after the 256-byte status
// block: a counter at byte 256, node indices from byte 512.  A workspace of 256 bytes has no
// queue (such nodes then report PFEM_ERR_DEGENERATE).
static void set_queue(P2MArgs &a, void *ws, size_t ws_bytes)
{
    const long long nodes = (long long)a.n * a.n;
    const long long cap = ws_bytes >= 520 ? (long long)((ws_bytes - 512) / sizeof(long long)) : 0;
    a.defer_cap = (int)std::min(std::min(cap, nodes), (long long)INT_MAX);
    a.defer_count = a.defer_cap > 0 ? (int *)((char *)ws + 256) : nullptr;
    a.defer_list = a.defer_cap > 0 ? (long long *)((char *)ws + 512) : nullptr;
}

static P2MArgs make_args(const GeoArgs &g, DevStatus *st)
{
    P2MArgs a;
    a.n = g.n;
    a.B.q = (const uint2 *)g.q_sorted;
    a.B.start = g.cell_start;
    a.B.nb = g.nb;
    a.B.rmax = g.rmax;
    a.B.dmax = g.dmax;
    a.B.kcap = g.kcap;
    a.B.walk_cap = g.walk_cap;
    a.B.last4 = g.N >= 4 ? (int)(g.N - 4) : -1;
    a.R0 = g.R0;
    a.pos = g.pos_sorted;
    a.perm = nullptr;
    a.vals = nullptr;
    a.C = 0;
    a.out = nullptr;
    a.w_idx = nullptr;
    a.w = nullptr;
    a.K = 0;
    a.status = st;
    a.ucap = g.ucap;
    return a;
}

// Meshes of up to this many nodes per SM run four lanes a node: their warps are too few to cover one
// lane's serial work.  Round trips on 152 SMs (24,320 nodes at the line), one lane / four: 33^2 FP64
// 136 / 102 us, 129^2 113 / 102 (FP64 153 / 140), 138^2 123 / 111, 200^2 139 / 150, 257^2 three loop
// steps 523 / 600.
constexpr int TAB_QUAD_NODES = 160;

static dim3 node_grid(int n) { return dim3((n + 15) / 16, (n + 7) / 8); }

template <typename P, typename V, typename R, typename S, int REF, int SHAPE, bool W>
static cudaError_t go_fast(const P2MArgs &a, cudaStream_t s)
{
    if constexpr (SHAPE == PFEM_SHAPE_LINEAR) {
        k_p2m_linear<P, V, R, W><<<node_grid(a.n), 128, 0, s>>>(a);
    } else {
        // FP64 solves take the FP32 factor with the solution refined to FP64 (fix64.cuh)
        constexpr bool F64 = sizeof(S) == 8;
        k_p2m<P, V, R, std::conditional_t<F64, float, S>, F64 ? REFINE_FIX64 : REF, SHAPE, W>
            <<<node_grid(a.n), 128, 0, s>>>(a);
    }
    count_launch();
    return cudaGetLastError();
}

static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace layout of P2M after the 256-byte status block: the fix-pass queue counter at byte
// 256 and the star-table queue counter right before it, the fix-pass queue from byte 512 (8 bytes
// per node), then 136 bytes a node that pfem_workspace_size includes and nothing uses, and the star
// table.
static size_t table_offset(long long nodes) { return al256(512 + 8 * (size_t)nodes) + al256(136 * (size_t)nodes); }

size_t p2m_ws_bytes(long long nodes, long long N) { return table_offset(nodes) + star_tab_bytes(N); }

// Star table in ws, when it has room for it.
static bool set_table(StarTab &t, void *ws, size_t ws_bytes, long long nodes, long long N)
{
    if (ws_bytes < p2m_ws_bytes(nodes, N)) return false;
    t = star_tab_layout((char *)ws + table_offset(nodes), N, (int *)((char *)ws + 252));
    return true;
}

// P2M: the fast pass over all nodes, then the fix pass over the nodes it queued.  With quadratic
// shape functions, the apply form and room for the table, the fast pass is the star table and
// then k_p2m_tab (location, edge solves and apply per node); otherwise one kernel that searches the
// stars per node.
// Stage events (when the caller's context has them): 0 before the fast pass, 1 after the star
// table, 2 right before k_p2m_tab, 3 after it, 4 after the fix pass.
template <typename P, typename V, typename R, typename S, int REF, int SHAPE, bool W>
static cudaError_t go(const GeoArgs &g, const P2MArgs &a, cudaStream_t s,
                      const StarTab *tab = nullptr)
{
    const int R0 = g.R0, rmax_far = g.rmax_far;
    cudaError_t e;
    stage_event(g, 0, s);
    // the star table's launcher clears both queue counters, which lie side by side
    if (a.defer_cap > 0 && !(SHAPE == PFEM_SHAPE_QUADRATIC && tab)) {
        e = cudaMemsetAsync(a.defer_count, 0, sizeof(int), s);
        if (e != cudaSuccess) return e;
    }
    if (SHAPE == PFEM_SHAPE_QUADRATIC && W && tab) {
        if constexpr (SHAPE == PFEM_SHAPE_QUADRATIC && W) {
            // a star that no node needs may fail unnoticed, as where each node searches its own: a
            // scratch status word
            e = launch_star_table(a.B, R0, rmax_far, *tab, (DevStatus *)((char *)a.status + 128), s, 1);
            if (e != cudaSuccess) return e;
            const bool vec = a.K % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.w_idx) | reinterpret_cast<uintptr_t>(a.w)) & 31) == 0;
            k_shape_tab<P, R, sizeof(S) == 8 ? REFINE_FIX64 : REF><<<node_grid(a.n), 128, 0, s>>>(a, *tab, vec);
            count_launch();
            e = cudaGetLastError();
        }
    } else if (SHAPE == PFEM_SHAPE_QUADRATIC && !W && tab) {
        e = launch_star_table(a.B, R0, rmax_far, *tab, a.status, s, 1);
        if (e != cudaSuccess) return e;
        stage_event(g, 1, s);
        stage_event(g, 2, s);
        e = wait_values(g, s);
        if (e != cudaSuccess) return e;
        constexpr int TREF = sizeof(S) == 8 ? REFINE_FIX64 : REF;
        if ((long long)a.n * a.n <= (long long)TAB_QUAD_NODES * num_sms())
            k_p2m_tab<P, V, R, float, TREF, 4><<<dim3((a.n + 7) / 8, (a.n + 3) / 4), 128, 0, s>>>(a, *tab);
        else
            k_p2m_tab<P, V, R, float, TREF, 1><<<node_grid(a.n), 128, 0, s>>>(a, *tab);
        count_launch();
        e = cudaGetLastError();
        stage_event(g, 3, s);
    } else {
        if (!W) {
            e = wait_values(g, s);
            if (e != cudaSuccess) return e;
        }
        e = go_fast<P, V, R, S, REF, SHAPE, W>(a, s);
    }
    if (e != cudaSuccess || a.defer_cap <= 0) return e;
    P2MArgs f = a;
    f.B.rmax = rmax_far > a.B.rmax ? rmax_far : a.B.rmax;
    if (SHAPE == PFEM_SHAPE_QUADRATIC && !W && tab)
        k_p2m_fix_tab<P, V, R><<<num_sms() * 2, 128, 0, s>>>(f, *tab);
    else
        k_p2m_fix<P, V, R, SHAPE, W><<<num_sms(), 128, 0, s>>>(f);
    count_launch();
    stage_event(g, 4, s);
    return cudaGetLastError();
}

// Compute type S and refinement of each solve for FP32 arithmetic.
template <typename P, typename V, int SHAPE, bool W>
static cudaError_t go_solve(pfem_solve solve, const GeoArgs &g, const P2MArgs &a, cudaStream_t s,
                            const StarTab *t)
{
    switch (solve) {
    case PFEM_SOLVE_F64: return go<P, V, float, double, REFINE_NONE, SHAPE, W>(g, a, s, t);
    case PFEM_SOLVE_F32: return go<P, V, float, float, REFINE_NONE, SHAPE, W>(g, a, s, t);
    default: return go<P, V, float, float, REFINE_FIX, SHAPE, W>(g, a, s, t);   // both refined solves
    }
}

cudaError_t launch_p2m(const GeoArgs &g, const int *perm, int C, const void *vals,
                       pfem_dtype val_t, pfem_shape shape, pfem_solve solve, void *out,
                       DevStatus *st, size_t ws_bytes, cudaStream_t s)
{
    P2MArgs a = make_args(g, st);
    set_queue(a, st, ws_bytes);
    a.perm = perm;
    a.vals = vals;
    a.C = C;
    a.out = out;
    const bool q = shape == PFEM_SHAPE_QUADRATIC;
    StarTab tab;
    const StarTab *t = set_table(tab, st, ws_bytes, (long long)g.n * g.n, g.N) ? &tab : nullptr;
    if (val_t == PFEM_F64) {   // positions FP64, arithmetic FP64
        if (!q) return go<double, double, double, double, REFINE_NONE, 0, false>(g, a, s);
        return go<double, double, double, double, REFINE_NONE, 1, false>(g, a, s, t);
    }
    if (val_t == PFEM_F32) {   // positions FP32, arithmetic FP32
        if (!q) return go<float, float, float, float, REFINE_NONE, 0, false>(g, a, s);
        return go_solve<float, float, 1, false>(solve, g, a, s, t);
    }
    if (!q) return go<float, __nv_bfloat16, float, float, REFINE_NONE, 0, false>(g, a, s);
    return go_solve<float, __nv_bfloat16, 1, false>(solve, g, a, s, t);
}

cudaError_t launch_shape(const GeoArgs &g, pfem_shape shape, pfem_solve solve, int K, int *w_idx,
                         void *w, pfem_dtype w_t, DevStatus *st, size_t ws_bytes, cudaStream_t s)
{
    P2MArgs a = make_args(g, st);
    set_queue(a, st, ws_bytes);
    a.K = K;
    a.w_idx = w_idx;
    a.w = w;
    const bool q = shape == PFEM_SHAPE_QUADRATIC;
    StarTab tab;
    const StarTab *t = q && set_table(tab, st, ws_bytes, (long long)g.n * g.n, g.N) ? &tab : nullptr;
    if (w_t == PFEM_F64) {
        if (!q) return go<double, double, double, double, REFINE_NONE, 0, true>(g, a, s);
        return go<double, double, double, double, REFINE_NONE, 1, true>(g, a, s, t);
    }
    if (!q) return go<float, float, float, float, REFINE_NONE, 0, true>(g, a, s);
    return go_solve<float, float, 1, true>(solve, g, a, s, t);
}

// alpha_i = sum_k w[i,k] alpha[w_idx[i,k]] (explicit-weight P2M)
template <typename V, typename R>
__global__ void __launch_bounds__(256) k_apply(long long nodes, int K, const int *__restrict__ w_idx,
                                               const R *__restrict__ w, const int *__restrict__ perm,
                                               int C, const V *__restrict__ vals, V *__restrict__ out,
                                               bool vec)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
         i += (long long)gridDim.x * blockDim.x) {
        R acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = R(0);
        for (int k = 0; k < K; k += 4) {
            // four entries at a time (their loads in flight together), one 16-byte load of the slots
            // where the rows allow it
            int s[4];
            if (vec) {
                const int4 q = __ldg(reinterpret_cast<const int4 *>(w_idx + i * K + k));
                s[0] = q.x; s[1] = q.y; s[2] = q.z; s[3] = q.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) s[j] = k + j < K ? __ldg(w_idx + i * K + k + j) : -1;
            }
            // the row ends at its first -1
#pragma unroll
            for (int j = 1; j < 4; ++j) s[j] = s[j - 1] < 0 ? -1 : s[j];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (s[j] < 0) continue;
                const R wk = __ldg(w + i * K + k + j);
                R v[8];
                load_vals<V, R>(vals, perm, s[j], C, v);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < C) acc[c] = fma(wk, v[c], acc[c]);
            }
            if (s[3] < 0) break;
        }
        store_vals<V, R>(out, i, C, acc);
    }
}

cudaError_t launch_apply(int n, const int *perm, int C, const void *vals, pfem_dtype val_t,
                         const int *w_idx, const void *w, int K, pfem_dtype w_t, void *out,
                         cudaStream_t s)
{
    const long long nodes = (long long)n * n;
    long long blocks = (nodes + 255) / 256;
    if (blocks > num_sms() * 16LL) blocks = num_sms() * 16LL;
    const bool vec = K % 4 == 0 && (reinterpret_cast<uintptr_t>(w_idx) & 15) == 0;
    if (val_t == PFEM_F64 && w_t == PFEM_F64)
        k_apply<double, double><<<(unsigned)blocks, 256, 0, s>>>(
            nodes, K, w_idx, (const double *)w, perm, C, (const double *)vals, (double *)out, vec);
    else if (val_t == PFEM_F32 && w_t == PFEM_F32)
        k_apply<float, float><<<(unsigned)blocks, 256, 0, s>>>(
            nodes, K, w_idx, (const float *)w, perm, C, (const float *)vals, (float *)out, vec);
    else if (val_t == PFEM_BF16 && w_t == PFEM_F32)
        k_apply<__nv_bfloat16, float><<<(unsigned)blocks, 256, 0, s>>>(
            nodes, K, w_idx, (const float *)w, perm, C, (const __nv_bfloat16 *)vals,
            (__nv_bfloat16 *)out, vec);
    else
        return cudaErrorInvalidValue;
    count_launch();
    return cudaGetLastError();
}

// The star table written straight into the caller's arrays, then padded: unused entries -1 and
// a failed star's count 0 (its error is in the status word).
__global__ void k_stars_pad(long long N, int *nbrs, int *counts)
{
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
         v += (long long)gridDim.x * blockDim.x) {
        const int w = (int)((unsigned)counts[v] & 255u) - 128;   // drop the table's stamp
        const int c = w < 0 ? 0 : w;
        for (int k = c; k < KMAX; ++k) nbrs[v * KMAX + k] = -1;
        counts[v] = c;
    }
}

// Workspace bytes of pfem_delaunay_stars: the status block and the retry queue.
size_t stars_ws_bytes(long long N) { return 256 + 4 * (size_t)(N > 0 ? N : 1); }

cudaError_t launch_stars(const GeoArgs &g, int *nbrs, int *counts, DevStatus *st, cudaStream_t s)
{
    P2MArgs a = make_args(g, st);
    StarTab t;
    t.nbr = nbrs;
    t.cnt = counts;
    t.queue = (int *)((char *)st + 256);
    t.qcount = (int *)((char *)st + 64);
    t.N = g.N;
    t.gen = next_tab_gen();
    cudaError_t e = launch_star_table(a.B, g.R0, g.rmax_far, t, st, s);
    if (e != cudaSuccess) return e;
    long long blocks = (g.N + 255) / 256;
    if (blocks > num_sms() * 16LL) blocks = num_sms() * 16LL;
    if (blocks < 1) blocks = 1;
    k_stars_pad<<<(unsigned)blocks, 256, 0, s>>>(g.N, nbrs, counts);
    count_launch();
    return cudaGetLastError();
}

}  // namespace pfem
