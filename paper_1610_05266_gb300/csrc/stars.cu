// stars.cu -- the star table (startab.cuh): the Delaunay star of every particle, one thread per
// particle, then the particles whose list attempt failed by a region search.
#include <algorithm>
#include <atomic>

#include "internal.h"
#include "startab.cuh"

namespace pfem {

__global__ void __launch_bounds__(STAR_TPB, PFEM_STAR_MIN_BLOCKS) k_star_list(Bins B, int R0, StarTab t,
                                                                              DevStatus *st)
{
    __shared__ __align__(16) unsigned char lists[HullList::BYTES];
    const long long v = blockIdx.x * (long long)STAR_TPB + threadIdx.x;
    if (v >= t.N) return;
    star_list_slot(B, R0, t, v, HullList::at(lists, threadIdx.x), st);
}

// The queued particles, with the radius of B (the launcher passes the widest one).
__global__ void __launch_bounds__(RETRY_TPB, RETRY_BLOCKS) k_star_retry(Bins B, int R0, StarTab t,
                                                                        DevStatus *st)
{
    __shared__ __align__(16) unsigned char lists[HullListLong::BYTES];
    __shared__ int2 sd[RETRY_TPB / 32 * WSTAR_CAP];
    __shared__ int ss[RETRY_TPB / 32 * WSTAR_CAP];
    const int w = threadIdx.x >> 5;
    star_retry(t, lists, WarpList{sd + w * WSTAR_CAP, ss + w * WSTAR_CAP}, st, [&](int, int &r) {
        r = R0;
        return B;
    });
}

size_t star_tab_bytes(long long N)
{
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t n = (size_t)(N > 0 ? N : 1);
    return al(n * KMAX * sizeof(int)) + al(n * sizeof(int)) + al(n * sizeof(int));
}

// A fresh stamp for each table build (1 .. 2^24 - 1, cycling).
unsigned next_tab_gen()
{
    static std::atomic<unsigned> gen{0};
    unsigned g;
    do {
        g = (gen.fetch_add(1, std::memory_order_relaxed) + 1) & 0xffffffu;
    } while (g == 0);
    return g;
}

StarTab star_tab_layout(char *base, long long N, int *qcount)
{
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t n = (size_t)(N > 0 ? N : 1);
    StarTab t;
    t.nbr = (int *)base;
    t.cnt = (int *)(base + al(n * KMAX * sizeof(int)));
    t.queue = (int *)(base + al(n * KMAX * sizeof(int)) + al(n * sizeof(int)));
    t.qcount = qcount;
    t.N = N;
    t.gen = next_tab_gen();
    return t;
}

cudaError_t launch_star_table(const Bins &B, int R0, int rmax_far, const StarTab &t,
                              DevStatus *st, cudaStream_t s, int also)
{
    if (t.N <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(t.qcount, 0, sizeof(int) * (size_t)(1 + also), s);
    if (e != cudaSuccess) return e;
    k_star_list<<<(unsigned)((t.N + STAR_TPB - 1) / STAR_TPB), STAR_TPB, 0, s>>>(B, R0, t, st);
    Bins Bf = B;
    Bf.rmax = std::max(B.rmax, rmax_far);
    k_star_retry<<<num_sms() * RETRY_BLOCKS, RETRY_TPB, 0, s>>>(Bf, R0, t, st);
    count_launch(2);
    return cudaGetLastError();
}

}  // namespace pfem
