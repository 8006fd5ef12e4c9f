// ma_small_grid.cuh -- grids of n <= 17 points a side held by one thread block:
// index arithmetic and the colour phases of their sweeps.
//
// A sweep of a small grid is a chain of colour phases, each as long as one
// point's dependent chain (loads, Hessian, the Newton steps of the root) and a
// barrier; the points of a phase fill few warps.  So a phase runs on no more
// warps than it has points for (a whole block's barrier, and idle warps at
// it, cost more than the phase), a point's position comes from multiplications
// by reciprocals in place of integer divisions, and what no phase
// writes is loaded one phase ahead.
#pragma once

#include <cuda_runtime.h>

namespace ma {
namespace small {

// Index arithmetic of a grid of n <= 17 points a side.  t / d as
// t (65536 / d + 1) >> 16: exact for t d <= 65536.
struct SmallGrid {
    int n, a, b, ma, mb, mi, mn;   // a, b: interior indices of parity 0, 1; m*: reciprocals of a, b, n - 2, n
    __device__ __forceinline__ explicit SmallGrid(int n_) : n(n_), a((n_ - 3) / 2), b((n_ - 1) / 2)
    {
        auto set = [this](int a_, int b_, int i_, int n_) { ma = a_; mb = b_; mi = i_; mn = n_; };
        switch (n) {   // the sizes of a hierarchy's levels without a division
        case 3: set(0, 65537, 65537, 65536 / 3 + 1); break;
        case 5: set(65537, 65536 / 2 + 1, 65536 / 3 + 1, 65536 / 5 + 1); break;
        case 9: set(65536 / 3 + 1, 65536 / 4 + 1, 65536 / 7 + 1, 65536 / 9 + 1); break;
        case 17: set(65536 / 7 + 1, 65536 / 8 + 1, 65536 / 15 + 1, 65536 / 17 + 1); break;
        default: set(65536 / a + 1, 65536 / b + 1, 65536 / (n - 2) + 1, 65536 / n + 1);
        }
    }
    __device__ __forceinline__ int count(int c) const
    {
        return ((c & 1) ? b : a) * ((c & 2) ? b : a) * ((c & 4) ? b : a);
    }
    __device__ __forceinline__ int offset(int c) const   // cm_offset
    {
        const int sj = (c & 2) ? b : a, sk = (c & 4) ? b : a;
        return ((c & 4) ? (a + b) * (a + b) * a : 0) + ((c & 2) ? (a + b) * a * sk : 0) + ((c & 1) ? a * sj * sk : 0);
    }
    // linear index of point t of colour c
    __device__ __forceinline__ int point(int c, int t) const
    {
        const bool pi = c & 1, pj = c & 2, pk = c & 4;
        const int y0 = (t * (pi ? mb : ma)) >> 16, x = t - y0 * (pi ? b : a);
        const int z = (y0 * (pj ? mb : ma)) >> 16, y = y0 - z * (pj ? b : a);
        return (((pk ? 1 : 2) + 2 * z) * n + (pj ? 1 : 2) + 2 * y) * n + (pi ? 1 : 2) + 2 * x;
    }
    // interior point q in natural order: (i, j, k), its linear index returned
    __device__ __forceinline__ int interior(int q, int* i, int* j, int* k) const
    {
        const int y0 = (q * mi) >> 16, z = (y0 * mi) >> 16;
        *i = 1 + q - y0 * (n - 2);
        *j = 1 + y0 - z * (n - 2);
        *k = 1 + z;
        return (*k * n + *j) * n + *i;
    }
    // colour-major slot and colour count of interior point (i, j, k)
    __device__ __forceinline__ int slot(int i, int j, int k, int* cnt, int* off) const
    {
        const int c = (i & 1) | ((j & 1) << 1) | ((k & 1) << 2);
        const int ni = (i & 1) ? b : a, nj = (j & 1) ? b : a;
        *cnt = count(c);
        *off = offset(c);
        return (((k - 1) >> 1) * nj + ((j - 1) >> 1)) * ni + ((i - 1) >> 1);
    }
};

// Warps that run a grid's colour phases, and their barrier: one warp up to
// 5^3 (at most 9 points a phase), four up to 9^3 (at most 91), the block above.
__device__ __forceinline__ int phase_threads(int n, int block) { return n <= 5 ? 32 : (n <= 9 ? 128 : block); }

__device__ __forceinline__ void phase_barrier(int n)
{
    if (n <= 5) __syncwarp();
    else if (n <= 9) asm volatile("bar.sync 1, 128;" ::: "memory");
    else __syncthreads();
}

// Phase q of a sweep: in colour pairs (c, c ^ 7) for c = 0 .. 3, or in
// ascending order in 7 phases: colours 3 and 4 differ in all three parities,
// so they are independent and share one.
__device__ __forceinline__ int phases_of(bool pairs) { return pairs ? 4 : 7; }
__device__ __forceinline__ int phase_first(bool pairs, int q) { return pairs || q <= 3 ? q : q + 1; }
__device__ __forceinline__ int phase_second(bool pairs, int q) { return pairs ? q ^ 7 : (q == 3 ? 4 : -1); }

// Linear index and slot of a phase's point t, packed; -1 where it has none.
__device__ __forceinline__ int phase_point(const SmallGrid& G, bool pairs, int q, int t)
{
    int c = phase_first(pairs, q);
    const int d = phase_second(pairs, q), nc = G.count(c);
    if (t >= nc) {
        if (d < 0) return -1;
        t -= nc;
        c = d;
        if (t >= G.count(d)) return -1;
    }
    return G.point(c, t) | (G.offset(c) + t) << 16;
}

// The points of grids up to 9^3, at most one a thread in each phase, worked
// out once: entry [phase][thread].
constexpr int kPhaseTab = 7 * 128;

__device__ __forceinline__ void fill_phase_tab(int* tab, int n, bool pairs)
{
    if (n > 9 || n < 5) return;
    const SmallGrid G(n);
    const int lt = n <= 5 ? 5 : 7;   // log2 of the threads
    for (int x = threadIdx.x; x < phases_of(pairs) << lt; x += blockDim.x)
        tab[x] = phase_point(G, pairs, x >> lt, x & ((1 << lt) - 1));
}

// The phase tables of the 9^3 and 5^3 grids.
constexpr int kTailTab = kPhaseTab + 7 * 32;
__device__ __forceinline__ int* tail_tab(int* tab, int n) { return n == 9 ? tab : tab + kPhaseTab; }

}  // namespace small
}  // namespace ma
