// startab.cuh -- the Delaunay star of every particle (App. B: the particles joined to it by a
// Delaunay edge), computed once per projection call and kept in a table that the per-node
// kernels read instead of searching.
//
// A mesh node needs the stars of the three vertices of its Delaunay triangle, and neighbouring
// nodes need different particles; searching stars per node makes every thread of a warp run its
// own gift-wrapping, of its own length, over its own candidate list.  Here every particle's star
// is computed by one thread of a particle-parallel kernel, so the threads of a warp do the same
// work on neighbouring particles (consecutive slots share bins), with the candidate lists in
// shared memory.  Stars the list attempt cannot certify (an empty circle wider than the
// candidate cutoff, a list overflow) are queued and computed by a second kernel that searches
// growing regions.  The table is then a plain array: slot v's star is nbr[v * PFEM_KMAX + k],
// k < cnt[v], counter-clockwise from its nearest neighbour.
#pragma once

#include "geom.cuh"

namespace pfem {

struct StarTab {
    int *nbr;           // [N][KMAX] slots
    int *cnt;           // [N] stamped count (tab_pack): star size, -1 while queued, or -PFEM_ERR_*
    int *queue;         // [N] slots whose list attempt failed
    int *qcount;        // number of queued slots
    long long N;
    unsigned gen;       // stamp of this call's entries (1 .. 2^24 - 1)
};

// A count entry carries the stamp of the call that wrote it, so that an entry left by an
// earlier call (or not yet written by this one) reads as "not available" (-1) instead of as a
// star: (gen << 8) | (value + 128).
__device__ __forceinline__ int tab_pack(unsigned gen, int v)
{
    return (int)((gen << 8) | (unsigned)((v + 128) & 255));
}

__device__ __forceinline__ int tab_count(const StarTab &t, int v)
{
    const unsigned w = (unsigned)__ldg(t.cnt + v);
    return (w >> 8) == t.gen ? (int)(w & 255u) - 128 : -1;
}

// Star of slot v read from the table (entries through the read-only cache).
struct TabStar {
    const int *p;
    int n;
    __device__ __forceinline__ int operator[](int i) const { return __ldg(p + i); }
};

__device__ __forceinline__ TabStar tab_star(const StarTab &t, int v)
{
    return {t.nbr + (long long)v * KMAX, tab_count(t, v)};
}

// Apex of the Delaunay triangle to the left of the directed edge u -> w: the neighbour that
// follows w counter-clockwise in u's star.  -PFEM_ERR_DEGENERATE if w is not in u's star (the
// table is then inconsistent, which exact predicates rule out), or u's star's error.
__device__ __forceinline__ int tab_apex(const StarTab &t, int u, int w)
{
    const TabStar s = tab_star(t, u);
    if (s.n < 0) return s.n;
    for (int k = 0; k < s.n; ++k)
        if (s[k] == w) return s[k + 1 == s.n ? 0 : k + 1];
    return -PFEM_ERR_DEGENERATE;
}

// Locate fixed-point point p with the table's stars: nearest particle, the sector of its fan,
// else a visibility walk whose steps are table lookups.  Returns 0 or -PFEM_ERR_* / -PFEM_FAR.
static __device__ __noinline__ int locate_tab(const Bins &B, const StarTab &t, uint2 p, int R0,
                                              int tri[3])
{
    const int v0 = nearest_particle(B, p, R0);
    if (v0 < 0) return v0;
    const TabStar s0 = tab_star(t, v0);
    if (s0.n < 0) return s0.n == -1 ? -PFEM_FAR : s0.n;
    return fan_walk(B, p, v0, s0, s0.n, [&](int u, int w) { return tab_apex(t, u, w); }, tri);
}

// Threads per block and candidate-list capacity of the list kernels.  The lists live in shared
// memory, one column per thread (16 candidates and two entries that take what is not kept, 12
// bytes each, x 128 threads = 27 KB per block: eight blocks fill an SM's shared memory).
// Jittered lattices at jitter 0.25 have at most 16 particles within the 2-spacing cutoff (rarely
// 17 at jitter 0.3); longer lists go to the retry kernel.
constexpr int STAR_TPB = 128;
constexpr int STAR_KL = 16;
#ifndef PFEM_STAR_MIN_BLOCKS
#define PFEM_STAR_MIN_BLOCKS 8
#endif

// A thread's candidate list for the hull star: coordinates relative to v (FP32) and slots, entry
// k of the thread's column at k * S.  Lists longer than 16 keep their order and stack, which 16
// entries leave to registers, as bytes beside them.
template <int KLC, int S> struct HullListT {
    static constexpr int K = KLC, STRIDE = S, ROWS = KLC + 2;
    static constexpr int BYTES = ROWS * S * 12 + (KLC > 16 ? 2 * KLC * S : 0);    // of S columns
    float2 *xy;
    int *s;
    unsigned char *ord, *stk;
    // column `lane` of BYTES bytes of shared memory
    static __device__ __forceinline__ HullListT at(void *mem, int lane)
    {
        float2 *x = (float2 *)mem;
        int *i = (int *)(x + ROWS * S);
        unsigned char *b = (unsigned char *)(i + ROWS * S);
        return {x + lane, i + lane, b + lane, b + KLC * S + lane};
    }
};
using HullList = HullListT<STAR_KL, STAR_TPB>;

// The key of candidate k, packed for sorting: the pseudo-angle of (x, y), monotone in the polar
// angle, in 26-bit fixed point (a full turn is 2^26 units) above the 5-bit list index.  With p = y /
// (|x| + |y|) in [-1, 1] and 2^24 units a quadrant it is p where x >= 0 and half a turn less p where
// x < 0, modulo a turn: half a turn is the sign bit of the key shifted up by one.  The key's error
// is below 17 units (1e-6 of a quadrant), so keys that differ by more than KEY_NEAR units are in
// the right order; closer ones are ordered exactly.
constexpr unsigned KEY_NEAR = 67;    // 4e-6 * 2^24
constexpr unsigned KEY_TURN = 1u << 26;
__device__ __forceinline__ float rcp_approx(float x)     // within 1 ulp; x not denormal
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// The pseudo-angle in the upper 26 bits.
__device__ __forceinline__ unsigned angle_key(float x, float y)
{
    const float r = copysignf(16777216.0f * rcp_approx(fabsf(x) + fabsf(y)), x);
    return ((unsigned)__float2int_rn(y * r) << 6) ^ (__float_as_uint(x) & 0x80000000u);
}

// Sort KLC packed keys (bitonic network, unrolled: the array stays in registers; Batcher's
// odd-even merge network, 63 instead of 80 compare-exchanges for 16 keys, measured slower).
template <int KLC> __device__ __forceinline__ void sort_keys(unsigned (&w)[KLC])
{
#pragma unroll
    for (int size = 2; size <= KLC; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int i = 0; i < KLC; ++i) {
                const int j = i ^ stride;
                if (j > i) {
                    const unsigned a = w[i], b = w[j];
                    const unsigned lo = min(a, b), hi = max(a, b);
                    const bool up = (i & size) == 0;
                    w[i] = up ? lo : hi;
                    w[j] = up ? hi : lo;
                }
            }
}

// The rare parts of the hull star, out of line: they would only lengthen its code, which the
// warps of an SM, each at another step of it, read through one instruction cache.

// Exact offset of list entry k from v.
template <typename List>
__device__ __forceinline__ int2 list_exact(const Bins &B, uint2 pv, const List &L, int k)
{
    return rel(__ldg(B.q + L.s[k * List::STRIDE]), pv);
}

// The list's nearest candidate by exact distance, the lowest slot among equals.
template <typename List>
static __device__ __noinline__ int nearest_exact(const Bins &B, uint2 pv, List L, int cnt)
{
    long long best = 0x7fffffffffffffffLL;
    int s0 = 0x7fffffff, u0 = 0;
    for (int k = 0; k < cnt; ++k) {
        const int2 d = list_exact(B, pv, L, k);
        const long long d2 = (long long)d.x * d.x + (long long)d.y * d.y;
        const int s = L.s[k * List::STRIDE];
        if (d2 < best || (d2 == best && s < s0)) { best = d2; s0 = s; u0 = k; }
    }
    return u0;
}

// The candidates in angular order from u0 where keys are too close: 4 bits an entry, u0 lowest.
// Insertion sort with near-equal angles by the half turn from u0 and the exact cross product; on
// one ray the farther particle first (its image lies inside the hull and the scan removes it),
// which on u0's own ray puts the farther particles at the end.
static __device__ __noinline__ unsigned long long order_exact(const Bins &B, uint2 pv, HullList L,
                                                              int cnt, int u0)
{
    const int2 d0 = list_exact(B, pv, L, u0);
    auto key = [&](int k) {
        const float2 c = L.xy[k * STAR_TPB], o = L.xy[u0 * STAR_TPB];
        return (angle_key(c.x, c.y) - angle_key(o.x, o.y)) >> 6;
    };
    auto half = [&](int k, int2 d) {
        if (k == u0) return 0;
        const long long cr = cross(d0, d);
        if (cr != 0) return cr > 0 ? 1 : 2;
        return (long long)d0.x * d.x + (long long)d0.y * d.y < 0 ? 2 : 3;
    };
    auto after = [&](int a, int b) -> bool {   // should candidate a come after b?
        const unsigned ka = key(a), kb = key(b);
        if (min(ka, kb) > KEY_NEAR && max(ka, kb) < KEY_TURN - KEY_NEAR) {
            if (ka > kb + KEY_NEAR) return true;
            if (kb > ka + KEY_NEAR) return false;
        }
        const int2 da = list_exact(B, pv, L, a), db = list_exact(B, pv, L, b);
        const int ha = half(a, da), hb = half(b, db);
        if (ha != hb) return ha > hb;
        const long long cr = cross(da, db);
        if (cr != 0) return cr < 0;
        return (long long)da.x * da.x + (long long)da.y * da.y < (long long)db.x * db.x + (long long)db.y * db.y;
    };
    unsigned long long o = 0;
    for (int i = 0; i < cnt; ++i) {
        int j = i;                             // entry i goes before the last ones it precedes
        while (j > 0 && after((int)(o >> (4 * (j - 1))) & 15, i)) --j;
        const unsigned long long low = (1ull << (4 * j)) - 1;
        o = (o & low) | ((unsigned long long)i << (4 * j)) | ((o & ~low) << 4);
    }
    return o;
}

// The certificate of a triangle thin at v (star_hull), list entries a and b: the same bound from
// the exact offsets (64-bit integers, products in FP64 within 1e-15).
template <typename List>
static __device__ __noinline__ bool certify_thin(const Bins &B, uint2 pv, float D, List L, int a, int b)
{
    const int2 ea = list_exact(B, pv, L, a), eb = list_exact(B, pv, L, b);
    const long long Ke = cross(ea, eb);
    if (Ke <= 0) return false;
    const long long ex = (long long)ea.x - eb.x, ey = (long long)ea.y - eb.y;
    const double lae = (double)((long long)ea.x * ea.x + (long long)ea.y * ea.y);
    const double lbe = (double)((long long)eb.x * eb.x + (long long)eb.y * eb.y);
    const double labe = ((double)(ex * ex) + (double)(ey * ey)) / ((double)D * (double)D);
    const double Kd = (double)Ke;
    return !(lae * lbe * labe > 0.997 * Kd * Kd);
}

// The certificate where the region does not hold the disk of radius D about v: the circle through
// v, a, b has centre -(P, Q) / 2K and passes through v; its radius r must satisfy r + err <= every
// clearance measured from the centre and <= D / 2.
static __device__ __noinline__ bool certify_region(const Region &g, float D, HullList L,
                                                   unsigned long long star, int sp)
{
    auto at = [&](int j) { return L.xy[((int)(star >> (4 * j)) & 15) * STAR_TPB]; };
    for (int j = 0; j < sp; ++j) {
        const float2 a = at(j), b = at(j + 1 == sp ? 0 : j + 1);
        const FCirc cb = make_fcirc(a.x, a.y, b.x, b.y);
        if (!(cb.K > 1e-3f * cb.Ka)) return false;
        const float ik = __frcp_rn(cb.K);
        const float ccx = -0.5f * cb.P * ik, ccy = -0.5f * cb.Q * ik;
        const float err = (1e-4f * (cb.Pa + cb.Qa + (fabsf(cb.P) + fabsf(cb.Q)) * cb.Ka * ik)) * ik + 64.f;
        const float room = fminf(fminf(fminf(g.cl_hi_x - ccx, g.cl_lo_x + ccx),
                                       fminf(g.cl_hi_y - ccy, g.cl_lo_y + ccy)),
                                 0.49995f * D) - err;
        if (!(room > 0.f) || fmaf(ccx, ccx, ccy * ccy) > room * room * 0.9999f) return false;
    }
    return true;
}

// The Delaunay star of v from the candidates within distance D (at most STAR_KL), by the convex
// hull of the candidates inverted about v.  Inversion c -> c/|c|^2 maps the circles through v
// to lines, so an empty circle through v, a, b becomes a hull edge between the images of a
// and b; and the orientation of three images is the sign of the lifted incircle determinant of
// (v, a, b, c) -- the predicate of the gift-wrapping search, with the same tie-break.  So the
// hull's vertices in counter-clockwise order are v's star.  Returns the count, -1 (list overflow
// or not certified: the caller retries wider) or -PFEM_ERR_*.  B.last4 >= 0.
//
// The kernel is bound by instruction issue, and a warp's 32 stars differ in their data, so the
// steps are laid out as loops of the same length in every lane with predicated bodies:
//  1. Gather: one distance test per particle of the region; those within D are appended to the
//     list and nothing else is done there, because some lane of a warp accepts almost every one.
//  2. Over the list (unrolled, registers): nearest candidate u0, always a Delaunay neighbour, and
//     angular keys; the keys turned so that u0 comes first, through the sorting network.
//  3. One pass that drops every candidate whose image lies inside the triangle of v and the images
//     of the two candidates beside it in angular order: such a candidate is not on the hull,
//     whether or not the two are.  About half of the list goes.  (Where the two are 180 degrees
//     or more apart the test drops nothing, unless a neighbouring gap is that wide: then v has
//     no closed star within D, and the certificate fails with or without the candidate.)
//  4. A Graham scan of the rest, a push or a pop per iteration, its stack and the candidates'
//     order 4-bit entries of 64-bit registers.
//  5. Certify every triangle as the gift-wrapping search does (circumcircle inside the searched
//     region and within D of v).
template <typename List>
__device__ __forceinline__ int star_hull(const Bins &B, int v, uint2 pv, const Region &g, float D,
                                         const List &L, int *row)
{
    constexpr int S = List::STRIDE, KLC = List::K;
    constexpr bool SHORT = KLC == 16;
    constexpr unsigned IDS = SHORT ? 15u : 31u;     // index bits
    static_assert(KLC == 16 || KLC == 32, "the keys hold a 5-bit list index");
    const float D2 = D * D;
    int cnt = 0;
    auto take = [&](int s, uint2 qs, bool in) {
        const int2 d = rel(qs, pv);
        const float fx = (float)d.x, fy = (float)d.y;
        const float l = fmaf(fx, fx, fy * fy);
        // written in any case and kept by moving on, without a branch
        L.xy[cnt * S] = make_float2(fx, fy);
        L.s[cnt * S] = s;
        cnt = min(cnt + (in && s != v && l <= D2 ? 1 : 0), KLC + 1);
    };
    // the region's slot runs, four loads in flight at a time
    for_region_runs(B, g, [&](int a, int e) {
        int s = a;
        for (; s < e && s <= B.last4; s += 4) {
            const uint2 *q = B.q + s;
            const uint2 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3);
            const int left = e - s;
            take(s, q0, true);
            take(s + 1, q1, left > 1);
            take(s + 2, q2, left > 2);
            take(s + 3, q3, left > 3);
        }
        for (; s < e; ++s) take(s, __ldg(B.q + s), true);
    });
    if (cnt > KLC || cnt == 0) return -1;
    // nearest candidate: FP32 squared distances with the index in the low bits; the two
    // smallest tell whether the rounding could have mixed them up (each is within 6 units of the
    // last place of its true value: 2 of the 16-unit steps at most)
    unsigned w[KLC], m1 = 0xffffffffu, m2 = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < KLC; ++k) {
        const float2 c = L.xy[k * S];
        const float l = fmaf(c.x, c.x, c.y * c.y);
        // past the list (whatever its padding holds): all ones, by arithmetic, since a select
        // becomes a branch around the load and the key
        const unsigned d = (__float_as_uint(l) & ~IDS) | (unsigned)k | (unsigned)((cnt - 1 - k) >> 31);
        w[k] = angle_key(c.x, c.y);
        m2 = min(m2, max(m1, d));
        m1 = min(m1, d);
    }
    int u0 = (int)(m1 & IDS);
    if (m2 != 0xffffffffu && (m2 >> (SHORT ? 4 : 5)) - (m1 >> (SHORT ? 4 : 5)) <= 2u) u0 = nearest_exact(B, pv, L, cnt);
    const float2 c0 = L.xy[u0 * S];
    const float l0 = fmaf(c0.x, c0.x, c0.y * c0.y);
    if (l0 == 0.f) return -PFEM_ERR_DEGENERATE;
    // Angular order from u0: the keys less u0's above the 5-bit list index, through the network.
    // The list's padding sorts behind them as further entries of u0, the first a full turn from
    // it and the rest well apart, so that one look at the differences of adjacent keys finds
    // those closer than KEY_NEAR, u0's neighbours across the turn among them: such a star takes
    // the exact order.
    const unsigned k0 = angle_key(c0.x, c0.y);
    // (bit 4 of a short list's padding keeps the first one beyond the turn)
    const unsigned pad = (KEY_TURN << 5) + (SHORT ? 16u : 32u) + (unsigned)u0 - ((unsigned)cnt << 20);
#pragma unroll
    for (int k = 0; k < KLC; ++k)
        w[k] = k < cnt ? ((w[k] - k0) >> 1) + (unsigned)k : pad + ((unsigned)k << 20);
    sort_keys<KLC>(w);
    unsigned gap = (KEY_TURN << 5) - w[KLC - 1];        // a full list; else above 2^31
#pragma unroll
    for (int k = 0; k + 1 < KLC; ++k) gap = min(gap, w[k + 1] - w[k]);
    const bool near = gap < ((KEY_NEAR + 1) << 5);
    if constexpr (SHORT) {
        if (near) {
            const unsigned long long o = order_exact(B, pv, L, cnt, u0);
#pragma unroll
            for (int k = 0; k < KLC; ++k) w[k] = k < cnt ? (unsigned)(o >> (4 * k)) & 15u : (unsigned)u0;
        }
    } else if (near) {
        return -1;                               // left to the warp search
    }
    // Is the image of c to the left of the images of a -> b, i.e. c outside the circle through v,
    // a, b?  FP32 filter on det = la (b x c) - lb (a x c) + lc (a x b), whose terms are bounded by
    // la lb + lc (la + lb) <= 3 D^4 (|p x q| <= (lp + lq) / 2, every l <= D^2): one bound for the
    // whole star, 2^-19 of that; the exact predicate when undecided.
    const float bnd = 5.7220458984375e-06f * D2 * D2;    // 3 x 2^-19 x D^4
    // drop what is certainly inside, from the last candidate to the first so that the first ends
    // in the lowest bits of ord: c between p, the one before it, and n, the one kept after it (u0
    // at the end)
    unsigned long long ord = 0;
    int rem = 0, oi = KLC;                       // long lists: L.ord from entry oi on
    {
        float nx = c0.x, ny = c0.y, nl = l0, cx = c0.x, cy = c0.y, cl = l0, cn = 0.f;
        unsigned id = 0;
#pragma unroll
        for (int k = KLC - 1; k >= 0; --k) {
            const unsigned pid = w[k] & IDS;
            const float2 p = L.xy[pid * S];
            const float pl = fmaf(p.x, p.x, p.y * p.y);
            const float pc = fmaf(p.x, cy, -p.y * cx), pn = fmaf(p.x, ny, -p.y * nx);
            const float det = fmaf(pl, cn, fmaf(-cl, pn, nl * pc));
            const bool keep = det > -bnd;
            if (keep && k + 1 < cnt) {
                if constexpr (SHORT) ord = (ord << 4) | id;
                else L.ord[--oi * S] = (unsigned char)id;
                ++rem;
            }
            nx = keep ? cx : nx;
            ny = keep ? cy : ny;
            nl = keep ? cl : nl;
            cn = keep ? pc : pn;
            cx = p.x;
            cy = p.y;
            cl = pl;
            id = pid;
        }
    }
    if (rem < 2) return -1;
    // Graham scan from u0 over the rest and back to u0, a push or a pop an iteration (below 2 KLC)
    unsigned long long stk = 0;
    int sp = 2;
    // the candidate after the next one; the stack's entry d below its top
    auto upcoming = [&](int d) { return SHORT ? (int)(ord >> (4 * d)) & 15 : (int)L.ord[(oi + d) * S]; };
    auto below = [&](int d) { return SHORT ? (int)(stk >> (4 * d)) & 15 : (int)L.stk[max(sp - 1 - d, 0) * S]; };
    {
        const int ib = upcoming(0);
        int ic = upcoming(1);
        const float2 b0 = L.xy[ib * S], s0 = L.xy[ic * S];
        if constexpr (SHORT) {
            stk = (unsigned long long)((unsigned)u0 << 4 | (unsigned)ib);
            ord >>= 8;
        } else {
            L.stk[0] = (unsigned char)u0;
            L.stk[S] = (unsigned char)ib;
            oi += 2;
        }
        --rem;
        float ax = c0.x, ay = c0.y, la = l0, bx = b0.x, by = b0.y, lb = fmaf(bx, bx, by * by);
        float cx = s0.x, cy = s0.y, lc = fmaf(cx, cx, cy * cy), ab = fmaf(ax, by, -ay * bx);
        for (int it = 0; it < 2 * KLC; ++it) {
            const float bc = fmaf(bx, cy, -by * cx), ac = fmaf(ax, cy, -ay * cx);
            const float det = fmaf(la, bc, fmaf(-lb, ac, lc * ab));
            bool keep = det > bnd;
            if (!keep && det >= -bnd) {
                const uint2 qa = __ldg(B.q + L.s[below(1) * S]), qb = __ldg(B.q + L.s[below(0) * S]),
                            qc = __ldg(B.q + L.s[ic * S]);
                keep = incircle_exact(rel(qa, pv), rel(qb, pv), rel(qc, pv), pv, qa, qb, qc) < 0;
            }
            keep = keep || sp < (rem == 0 ? 3 : 2);
            if (keep && rem == 0) break;
            const int id = keep ? (rem > 1 ? upcoming(0) : u0) : below(2);
            const float2 t = L.xy[id * S];
            const float lt = fmaf(t.x, t.x, t.y * t.y);
            if constexpr (SHORT) {
                stk = keep ? (stk << 4) | (unsigned)ic : stk >> 4;
                ord = keep ? ord >> 4 : ord;
            } else {
                if (keep) L.stk[sp * S] = (unsigned char)ic;
                oi = min(oi + (keep ? 1 : 0), KLC - 1);
            }
            sp += keep ? 1 : -1;
            rem -= keep ? 1 : 0;
            const float tax = ax, tay = ay, tla = la;
            ax = keep ? bx : t.x; ay = keep ? by : t.y; la = keep ? lb : lt;
            bx = keep ? cx : tax; by = keep ? cy : tay; lb = keep ? lc : tla;
            cx = keep ? t.x : cx; cy = keep ? t.y : cy; lc = keep ? lt : lc;
            ic = keep ? id : ic;
            ab = fmaf(ax, by, -ay * bx);
        }
    }
    if (sp < 3) return -1;
    // the star from u0 on, the first entry lowest: the stack's 4-bit entries in reverse
    unsigned long long star = 0;
    if constexpr (SHORT) {
        star = __brevll(stk) >> (64 - 4 * sp);
        star = (star & 0x5555555555555555ull) << 1 | (star >> 1 & 0x5555555555555555ull);
        star = (star & 0x3333333333333333ull) << 2 | (star >> 2 & 0x3333333333333333ull);
    }
    auto member = [&](int j) { return SHORT ? (int)(star >> (4 * j)) & 15 : (int)L.stk[j * S]; };
    // certify every triangle (v, w_j, w_j+1): counter-clockwise, circumcircle inside the region
    // and within D of v (then no particle outside the list can lie inside it).
    if (fminf(fminf(g.cl_lo_x, g.cl_hi_x), fminf(g.cl_lo_y, g.cl_hi_y)) >= 0.9995f * D) {
        // The region holds the disk of radius 0.9995 D about v.  A circle through v of radius
        // r = |a| |b| |a - b| / (2 |a x b|) lies within 2r of v, so 4 r^2 <= 0.997 D^2, i.e.
        // la lb |a - b|^2 <= 0.997 D^2 K^2, keeps it inside both.  Each FP32 offset carries
        // at most one rounding (2^-24, none below 2^24 units).  With K > 1e-3 of its summed
        // magnitudes, K^2 is within 4e-4 of its exact value, and a and b are then at least
        // 7e-4 rad apart as seen from v, so |a - b|^2 is within 4e-4 as well: the true 2r stays
        // below 0.9989 D, inside the region, and every particle within the circle has an FP32
        // squared distance below D^2, i.e. is in the list.
        const float iD2 = __frcp_rn(D2);
        float2 b = c0;
        float lb = l0;
        unsigned long long rest = star >> 4;
        for (int j = 0; j < sp; ++j) {
            const float2 a = b;
            const float la = lb;
            b = j + 1 == sp ? c0 : L.xy[(SHORT ? (int)rest & 15 : member(j + 1)) * S];
            rest >>= 4;
            lb = fmaf(b.x, b.x, b.y * b.y);
            const float k1 = a.x * b.y, k2 = a.y * b.x;
            const float K = k1 - k2;
            const float dx = a.x - b.x, dy = a.y - b.y;
            const float lab = fmaf(dx, dx, dy * dy) * iD2;
            const bool thin = !(K > 1e-3f * (fabsf(k1) + fabsf(k2)));
            if (thin ? !certify_thin(B, pv, D, L, member(j), member(j + 1 == sp ? 0 : j + 1))
                     : la * lb * lab > 0.997f * K * K)
                return -1;
        }
    } else if constexpr (SHORT) {
        if (!certify_region(g, D, L, star, sp)) return -1;
    } else {
        return -1;
    }
    if (sp > B.kcap) return -PFEM_ERR_CAPACITY;
    // the row (64-byte aligned) in whole 32-byte sectors by 16-byte stores, -1 after the star:
    // a partly written sector would cost the memory system a read to complete it
    const int nq = ((sp + 7) >> 3) << 1;
    for (int q = 0; q < nq; ++q) {
        const unsigned m = (unsigned)star;
        int e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            e[i] = L.s[(SHORT ? (int)(m >> (4 * i) & 15u) : member(min(4 * q + i, sp - 1))) * S];
            if (4 * q + i >= sp) e[i] = -1;
        }
        star >>= 16;
        reinterpret_cast<int4 *>(row)[q] = make_int4(e[0], e[1], e[2], e[3]);
    }
    return sp;
}

// The list attempt for slot v (candidates in L): its star into the table, or v queued.
__device__ __forceinline__ void star_list_slot(const Bins &B, int R0, const StarTab &t, long long v,
                                               const HullList &L, DevStatus *st)
{
    const uint2 pv = __ldg(B.q + v);
    int *out = t.nbr + v * KMAX;
    int c = -1;
    if (B.dmax > 0.f && B.last4 >= 0)
        c = star_hull(B, (int)v, pv, make_region(B, pv, R0), B.dmax, L, out);
    if (c == -1) {
        t.cnt[v] = tab_pack(t.gen, -1);
        t.queue[atomicAdd(t.qcount, 1)] = (int)v;   // at most N entries: each slot once
        return;
    }
    t.cnt[v] = tab_pack(t.gen, c);
    if (c < 0) record_error(st, -c, v);
}

// ---------------------------------------------------------------- queued stars, a warp each
// The stars whose list attempt failed: twelve of the jittered 2048^2 lattice's four million, more
// than half of a uniform random set's.  One warp computes one star by gift wrapping, its lanes
// sharing the candidates, so that a short queue takes the latency of one star's steps and a long
// one keeps the lanes busy.  (A thread per star, over lists in shared and local memory, took 32 us
// for the lattice's twelve and 1.77 ms for 590,000 of 1024^2 uniform random particles.)

// Candidates of a warp in shared memory: offsets from v and slots, in rows of 32 that lie STRIDE
// apart (32: one array).
constexpr int WSTAR_CAP = 96;
template <int STRIDE> struct WarpListT {
    int2 *d;
    int *s;
    static __device__ __forceinline__ int at(int k) { return STRIDE == 32 ? k : (k >> 5) * STRIDE + (k & 31); }
};
using WarpList = WarpListT<32>;
using HullWarpList = WarpListT<HullList::STRIDE>;      // in the lists of the warp's lanes

// An int whose order is the float's.
__device__ __forceinline__ int ordered(float x)
{
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}

// The apex of the Delaunay triangle to the left of v -> w among the warp's candidates: scan(f)
// calls f(d, slot) for each candidate of the calling lane.  The apex has the widest angle
// above the edge, i.e. the smallest cotangent t = c . (c - w) / (w x c); FP32 with an error bound,
// and the exact incircle predicate (with its tie-break) between candidates whose bounds overlap.
// All lanes return the same slot (-1: none) and offset.
template <typename Scan>
__device__ __forceinline__ int apex_warp(uint2 pv, int2 dw, Scan &&scan, int2 &best)
{
    const unsigned full = 0xffffffffu;
    const uint2 pw = make_uint2(pv.x + (unsigned)dw.x, pv.y + (unsigned)dw.y);
    auto inside = [&](int2 b, int2 c) {      // c inside the circle through v, w, b
        return incircle_exact(dw, b, c, pv, pw, make_uint2(pv.x + (unsigned)b.x, pv.y + (unsigned)b.y),
                              make_uint2(pv.x + (unsigned)c.x, pv.y + (unsigned)c.y)) > 0;
    };
    const float wx = (float)dw.x, wy = (float)dw.y;
    int2 bd = make_int2(0, 0);
    int bs = -1;
    float bt = 0.f, be = 0.f;
    scan([&](int2 d, int s) {
        const float cx = (float)d.x, cy = (float)d.y;
        const float o1 = wx * cy, o2 = wy * cx, oa = fabsf(o1) + fabsf(o2);
        const float X = o1 - o2;
        float t = 0.f, e = __int_as_float(0x7f800000);
        if (X > 4.76837158203125e-07f * oa) {
            // the inputs carry a rounding of 2^-24 each: N is within 4 of them of its terms'
            // magnitudes, X within 3 of oa (so at least 0.62 X is left), the quotient within 1
            const float inv = __fdividef(1.f, X);
            t = fmaf(cx, cx - wx, cy * (cy - wy)) * inv;
            const float mag = fmaf(fabsf(cx), fabsf(cx) + fabsf(wx), fabsf(cy) * (fabsf(cy) + fabsf(wy)));
            e = 2e-6f * fmaf(fabsf(t), oa, mag) * inv;
        } else if (X < -4.76837158203125e-07f * oa || cross(dw, d) <= 0) {
            return;                             // not strictly left of v -> w
        }
        if (bs >= 0) {
            if (t - e > bt + be) return;
            if (!(t + e < bt - be) && !inside(bd, d)) return;
        }
        bd = d;
        bs = s;
        bt = t;
        be = e;
    });
    const int lim = __reduce_min_sync(full, bs >= 0 ? ordered(bt + be) : 0x7fffffff);
    unsigned open = __ballot_sync(full, bs >= 0 && ordered(bt - be) <= lim);
    if (open == 0) return -1;
    int win = __ffs(open) - 1;
    for (open &= open - 1; open; open &= open - 1) {
        const int j = __ffs(open) - 1;
        const int2 b = make_int2(__shfl_sync(full, bd.x, win), __shfl_sync(full, bd.y, win));
        const int2 c = make_int2(__shfl_sync(full, bd.x, j), __shfl_sync(full, bd.y, j));
        if (inside(b, c)) win = j;
    }
    best = make_int2(__shfl_sync(full, bd.x, win), __shfl_sync(full, bd.y, win));
    return __shfl_sync(full, bs, win);
}

// The star of v by gift wrapping over the candidates of scan, from the nearest one u0 on, every
// triangle certified as apex_search does (its circumcircle inside the region, and with a cutoff
// D > 0, whose disk about v the region holds, within D of v).  Lane k receives entry k.  Returns the count, -1 (not certified) or
// -PFEM_ERR_CAPACITY.
template <typename Scan>
__device__ __forceinline__ int wrap_warp(const Bins &B, uint2 pv, const Region &g, float D, int u0,
                                         int2 d0, Scan &&scan, int &entry)
{
    const int lane = threadIdx.x & 31;
    const float iD2 = D > 0.f ? __frcp_rn(D * D) : 0.f;
    int cur = u0, n = 0;
    int2 dw = d0;
    for (;;) {
        if (n == B.kcap) return -PFEM_ERR_CAPACITY;
        if (lane == n) entry = cur;
        ++n;
        int2 da;
        const int a = apex_warp(pv, dw, scan, da);
        if (a < 0) return -1;
        // as in star_hull where the region holds the disk of radius D
        const float wx = (float)dw.x, wy = (float)dw.y, ax = (float)da.x, ay = (float)da.y;
        const float k1 = wx * ay, k2 = wy * ax, K = k1 - k2;
        if (D > 0.f && K > 1e-3f * (fabsf(k1) + fabsf(k2))) {
            const float dx = ax - wx, dy = ay - wy;
            const float lw = fmaf(wx, wx, wy * wy), la = fmaf(ax, ax, ay * ay);
            if (la * lw * (fmaf(dx, dx, dy * dy) * iD2) > 0.997f * K * K) return -1;
        } else {
            const Circ cb = make_circ(dw, da);
            const float inv2k = 0.5f / cb.K;
            const float cx = -cb.P * inv2k, cy = -cb.Q * inv2k;
            const float ext = sqrtf(fmaf(cx, cx, cy * cy)) + 1e-5f * (cb.Pa + cb.Qa) * (2.f * inv2k) + 64.f;
            if (cx - ext < -g.cl_lo_x || cx + ext > g.cl_hi_x || cy - ext < -g.cl_lo_y || cy + ext > g.cl_hi_y)
                return -1;
            if (D > 0.f && 2.f * ext > D * 0.9999f) return -1;
        }
        if (a == u0) return n >= 3 ? n : -1;
        cur = a;
        dw = da;
    }
}

// Star of slot v by the calling warp: list attempts with wider cutoffs (on uniform random
// particles 44 % of the stars have a circumcircle wider than 2 mean spacings, 0.3 % wider than
// 3.5), then every particle of growing regions up to B.rmax.  Lane k receives entry k.  Returns
// the count or -PFEM_ERR_* / -PFEM_FAR, the same in every lane.
template <typename List>
__device__ __forceinline__ int star_warp(const Bins &B, int v, uint2 pv, int R0, const List &L,
                                             int &entry)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    long long d2b;
    int u0;
    int2 d0;
    auto nearer = [&](int2 d, int s) {
        const long long d2 = (long long)d.x * d.x + (long long)d.y * d.y;
        if (d2 < d2b || (d2 == d2b && s < u0)) { d2b = d2; u0 = s; d0 = d; }
    };
    auto reset = [&]() { d2b = 0x7fffffffffffffffLL; u0 = 0x7fffffff; d0 = make_int2(0, 0); };
    auto nearest = [&]() {                       // over the lanes
        for (int o = 16; o > 0; o >>= 1) {
            const long long e = __shfl_xor_sync(full, d2b, o);
            const int s = __shfl_xor_sync(full, u0, o);
            const int2 d = make_int2(__shfl_xor_sync(full, d0.x, o), __shfl_xor_sync(full, d0.y, o));
            if (e < d2b || (e == d2b && s < u0)) { d2b = e; u0 = s; d0 = d; }
        }
    };
    if (B.dmax > 0.f)
        for (float f = 1.75f; f < 3.f; f += 0.75f) {
            const float D = f * B.dmax, D2 = D * D;
            const int R = max(R0, (int)ceilf(D * (float)B.nb * 2.3283064365386963e-10f));
            if (R > B.rmax) break;
            const Region g = make_region(B, pv, R);
            if (fminf(fminf(g.cl_lo_x, g.cl_hi_x), fminf(g.cl_lo_y, g.cl_hi_y)) < 0.9995f * D) break;
            int m = 0;
            reset();
            __syncwarp();
            for_region_runs(B, g, [&](int a, int e) {
                for (int s0 = a; s0 < e; s0 += 32) {
                    const int s = s0 + lane;
                    int2 d = make_int2(0, 0);
                    bool in = s < e && s != v;
                    if (in) {
                        d = rel(__ldg(B.q + s), pv);
                        const float fx = (float)d.x, fy = (float)d.y;
                        in = fmaf(fx, fx, fy * fy) <= D2;
                    }
                    const unsigned got = __ballot_sync(full, in);
                    const int at = m + __popc(got & ((1u << lane) - 1u));
                    if (in) {
                        nearer(d, s);
                        if (at < WSTAR_CAP) {
                            L.d[L.at(at)] = d;
                            L.s[L.at(at)] = s;
                        }
                    }
                    m += __popc(got);
                }
            });
            __syncwarp();
            nearest();
            if (m > 0 && d2b == 0) return -PFEM_ERR_DEGENERATE;
            if (m > WSTAR_CAP) break;
            if (m == 0) continue;
            const int c = wrap_warp(B, pv, g, D, u0, d0, [&](auto &&f) {
                for (int k = lane; k < m; k += 32) f(L.d[L.at(k)], L.s[L.at(k)]);
            }, entry);
            if (c != -1) return c;
        }
    for (int R = R0; R <= B.rmax; R = next_radius(R, R0)) {
        const Region g = make_region(B, pv, R);
        auto scan = [&](auto &&f) {
            for_region_runs(B, g, [&](int a, int e) {
                for (int s = a + lane; s < e; s += 32)
                    if (s != v) f(rel(__ldg(B.q + s), pv), s);
            });
        };
        reset();
        scan(nearer);
        nearest();
        if (d2b == 0) return -PFEM_ERR_DEGENERATE;
        if (u0 == 0x7fffffff) continue;
        const int c = wrap_warp(B, pv, g, 0.f, u0, d0, scan, entry);
        if (c != -1) return c;
    }
    return -PFEM_FAR;
}

// star_warp out of line, for kernels whose lanes have their registers for the hull attempt.
static __device__ __noinline__ int star_warp_call(const Bins &B, int v, int R0, HullWarpList L, int &entry)
{
    return star_warp(B, v, __ldg(B.q + v), R0, L, entry);
}

// Locate fixed-point point p as locate() does, the star of its nearest particle by the hull over the
// calling thread's list.  Where that cannot certify the star (more than half of a uniform random set's)
// the warp searches it together, its candidates in the lists' memory: every lane of the warp calls,
// `mine` where it has a point.  (Gift wrapping a lane instead keeps its candidates in local memory, for
// which the lists leave no L1: linear P2M of 1024^2 uniform random particles onto 257^2 nodes 1257 us,
// by gift wrapping alone 780, so 300.)
static __device__ __forceinline__ int locate_hull(const Bins &B, bool mine, uint2 p, int R0, const HullList &L,
                                                  int tri[3])
{
    static_assert((WSTAR_CAP + 31) / 32 <= HullList::ROWS, "a warp's candidates fit its lists");
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int v0 = mine ? nearest_particle(B, p, R0) : -1;
    __align__(16) int star[KMAX];
    int c = v0;
    if (v0 >= 0) {
        c = -1;
        const uint2 pv = __ldg(B.q + v0);
        if (B.dmax > 0.f && B.last4 >= 0) c = star_hull(B, v0, pv, make_region(B, pv, R0), B.dmax, L, star);
    }
    __syncwarp();
    const HullWarpList W{reinterpret_cast<int2 *>(L.xy - lane), L.s - lane};
    for (unsigned left = __ballot_sync(full, v0 >= 0 && c == -1); left; left &= left - 1) {
        const int j = __ffs(left) - 1;
        int entry = -1;
        const int n = star_warp_call(B, __shfl_sync(full, v0, j), R0, W, entry);
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            const int x = __shfl_sync(full, entry, k);
            if (lane == j) star[k] = x;
        }
        if (lane == j) c = n;
    }
    if (c < 0) return c;
    return fan_walk(B, p, v0, ArrStar{star, c}, c, [&](int u, int w) { return apex_of(B, u, w, R0); }, tri);
}

// Store a queued slot's star (entry of the calling lane) or record its error (an exhausted region as
// PFEM_ERR_CAPACITY).
__device__ __forceinline__ void star_retry_slot(const Bins &B, int R0, const StarTab &t, int v,
                                                const WarpList &L, DevStatus *st)
{
    const int lane = threadIdx.x & 31;
    int entry = -1;
    int c = star_warp(B, v, __ldg(B.q + v), R0, L, entry);
    if (c == -PFEM_FAR) c = -PFEM_ERR_CAPACITY;
    if (c > 0 && lane < ((c + 7) & ~7)) t.nbr[(long long)v * KMAX + lane] = lane < c ? entry : -1;
    if (lane == 0) {
        if (c < 0) record_error(st, -c, v);
        t.cnt[v] = tab_pack(t.gen, c);
    }
}

// Threads per block of the retry kernels and blocks per SM (31 KB of lists each): the queue length is
// known only on the device, so the grid covers what the SMs hold at once.
constexpr int RETRY_TPB = 64;
constexpr int RETRY_BLOCKS = 6;
using HullListLong = HullListT<32, RETRY_TPB>;

// A hull attempt at a queued star over a list of 32 at 1.375 times the cutoff: true when it is done.
__device__ __forceinline__ bool star_retry_hull(const Bins &B, int R0, const StarTab &t, int v,
                                                const HullListLong &L, DevStatus *st)
{
    if (!(B.dmax > 0.f) || B.last4 < 0) return false;
    const float D = 1.375f * B.dmax;
    const int R = max(R0, (int)ceilf(D * (float)B.nb * 2.3283064365386963e-10f));
    if (R > B.rmax) return false;
    const uint2 pv = __ldg(B.q + v);
    const int c = star_hull(B, v, pv, make_region(B, pv, R), D, L, t.nbr + (long long)v * KMAX);
    if (c == -1) return false;
    t.cnt[v] = tab_pack(t.gen, c);
    if (c < 0) record_error(st, -c, v);
    return true;
}

// The queue: a warp takes one star at a time while the queue is short, else 32, a lane each for a hull
// attempt and the rest one after the other.  1024^2 uniform random particles (590,000 queued): 1387 us
// with a warp for every star; round trip with the hull attempt at 1.25, 1.375, 1.5 times the cutoff
// 2141, 2033, 2297 us.  bins(v): the bins and first radius of slot v's problem.
template <typename BinsOf>
__device__ __forceinline__ void star_retry(const StarTab &t, void *mem, const WarpList &W, DevStatus *st,
                                           BinsOf &&bins)
{
    const int n = min(*t.qcount, (int)min(t.N, (long long)0x7fffffff));
    const int warps = gridDim.x * (RETRY_TPB / 32), w = blockIdx.x * (RETRY_TPB / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (n <= 4 * warps) {
        for (int i = w; i < n; i += warps) {
            const int v = t.queue[i];
            int R0;
            const Bins B = bins(v, R0);
            star_retry_slot(B, R0, t, v, W, st);
        }
        return;
    }
    const HullListLong L = HullListLong::at(mem, threadIdx.x);
    for (long long i0 = 32LL * w; i0 < n; i0 += 32LL * warps) {
        const bool mine = i0 + lane < n;
        const int v = mine ? t.queue[i0 + lane] : 0;
        bool done = true;
        if (mine) {
            int R0;
            const Bins B = bins(v, R0);
            done = star_retry_hull(B, R0, t, v, L, st);
        }
        __syncwarp();
        for (unsigned left = __ballot_sync(0xffffffffu, !done); left; left &= left - 1) {
            const int u = __shfl_sync(0xffffffffu, v, __ffs(left) - 1);
            int R0;
            const Bins B = bins(u, R0);
            star_retry_slot(B, R0, t, u, W, st);
        }
    }
}

}  // namespace pfem
