// ma_kernels_f64.cu -- FP64 kernels of the FAS V-cycle (Algorithm 1 of Liu,
// Froese, Oberman, Xiao) on one level grid of n^3 doubles, [k][j][i] order,
// boundary shell included.
//
//   smoother        Section 2: 8-colour nonlinear Gauss-Seidel, smallest root
//   residual        Algorithm 1 step 3 (r = rhs - det D^2_h u), norm partials
//   restriction     Section 3: half/full weighting, injection (steps 3-4)
//   coarse rhs      Algorithm 1 step 5 (tau correction)
//   prolongation    Section 3 trilinear, Algorithm 1 steps 7-8
//   coarsest solve  Algorithm 1 step 1, one thread block
//
// GB300 issues FP64 at about 1/70 of its FP32 rate.  The cycles' sweeps,
// residuals and coarse right-hand sides therefore take integer differences and
// two floats (ma_smooth_f2.cuh, ma_residual.cuh), two or three FP64 operations a
// point.  The single steps ma_smooth and ma_residual are FP64 throughout
// (ma_point.cuh), and bound by that pipe, as are the transfers.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <vector>

#include "ma.h"
#include "ma_internal.h"
#include "ma_batched.cuh"
#include "ma_point.cuh"
#include "ma_transfer.cuh"
#include "ma_residual.cuh"
#include "ma_small_grid.cuh"
#include "ma_smooth_f2.cuh"

namespace ma {

namespace {

using namespace small;

constexpr int BX = 32, BY = 4;

// Grids of kF2MinN points a side and more take the two-float forms of the
// point update, the residual and the coarse right-hand side; the one unknown of
// a 3^3 grid, which FP64 solves to a few ulps of the root, does not.
constexpr int kF2MinN = 5;
// ... with det3's sums unnormalised from here up, where its error stays below an ulp of u
constexpr int kUnormMinN = 33;

__device__ __forceinline__ long long lin(int i, int j, int k, int n)
{
    return ((long long)k * n + j) * n + i;
}

// ---------------------------------------------------------------------------
// Smoother: one colour phase.  Colour c = (i&1) | (j&1)<<1 | (k&1)<<2; the
// interior points of parity p along an axis start at 1 (p = 1) or 2 (p = 0).
// Every stencil neighbour differs from the centre in at least one index
// parity, so the points of one colour are independent and one launch may
// update them all in parallel.
// ---------------------------------------------------------------------------
template <int PI, int PJ, int PK>
__device__ __forceinline__ void smooth_colour_block(double* u, const double* __restrict__ rhs, int n, double h6,
                                                    unsigned long long* events, uint3 bid)
{
    const int i = (PI ? 1 : 2) + 2 * (int)(bid.x * BX + threadIdx.x);
    const int j = (PJ ? 1 : 2) + 2 * (int)(bid.y * BY + threadIdx.y);
    const int k = (PK ? 1 : 2) + 2 * (int)bid.z;
    if (i > n - 2 || j > n - 2 || k > n - 2) return;
    const long long sy = n, sz = (long long)n * n;
    const long long p = lin(i, j, k, n);
    const double v0 = u[p];
    const HessS H = gather_hess(u, p, sy, sz, v0);
    bool nonconvex = false;
    const double z = smallest_root(H, __dmul_rn(h6, rhs[p]), &nonconvex);   // h6 = 64 h^6: the 4 Hs scaling
    u[p] = fma(0.125, z, v0);
    if (nonconvex && events) atomicAdd(events, 1ull);
}

template <int PI, int PJ, int PK>
__global__ void __launch_bounds__(BX * BY) k_smooth_colour(double* u, const double* __restrict__ rhs, int n,
                                                            double h6, unsigned long long* events)
{
    smooth_colour_block<PI, PJ, PK>(u, rhs, n, h6, events, blockIdx);
}

// Interior indices of one parity along an axis of n points (n odd).
__host__ __device__ __forceinline__ int colour_count(int n, int parity) { return parity ? (n - 1) / 2 : (n - 3) / 2; }

template <int C>
cudaError_t launch_colour(double* u, const double* rhs, int n, double h6, unsigned long long* ev, cudaStream_t s)
{
    constexpr int PI = C & 1, PJ = (C >> 1) & 1, PK = (C >> 2) & 1;
    const int ni = colour_count(n, PI), nj = colour_count(n, PJ), nk = colour_count(n, PK);
    if (ni <= 0 || nj <= 0 || nk <= 0) return cudaSuccess;
    dim3 grid((ni + BX - 1) / BX, (nj + BY - 1) / BY, nk);
    count_launches(1);
    k_smooth_colour<PI, PJ, PK><<<grid, dim3(BX, BY), 0, s>>>(u, rhs, n, h6, ev);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The same sweep with the point update of ma_smooth_f2.cuh.  Colours 3 and 4
// follow each other in the order and differ in all three parities, a corner
// offset the stencil lacks, so they are independent and one launch sweeps both: blocks with z below nk0 take colour C, the rest colour
// D.  NN > 0 fixes the grid size at compile time for the sizes that stream
// from HBM: the 18 neighbour offsets become immediates of the loads.
// ---------------------------------------------------------------------------
template <int C, int NN, bool UNORM>
__device__ __forceinline__ void smooth_f2_block(double* u, const double* __restrict__ rhs, int n_rt,
                                                const smoothf2::Params& P, unsigned long long* events, int bz)
{
    const int n = NN > 0 ? NN : n_rt;
    const int i = ((C & 1) ? 1 : 2) + 2 * (int)(blockIdx.x * BX + threadIdx.x);
    const int j = ((C & 2) ? 1 : 2) + 2 * (int)(blockIdx.y * BY + threadIdx.y);
    const int k = ((C & 4) ? 1 : 2) + 2 * bz;
    if (i > n - 2 || j > n - 2 || k > n - 2) return;
    smoothf2::point<UNORM, UNORM ? resid::kDirect : resid::kSmall, long long>(u, rhs, lin(i, j, k, n), n, (long long)n * n, P, events);
}

template <int C, int D, int NN, bool UNORM>
__global__ void __launch_bounds__(BX * BY) k_smooth_f2(double* u, const double* __restrict__ rhs, int n,
                                                        smoothf2::Params P, unsigned long long* events, int nk0)
{
    const int bz = blockIdx.z;
    if (C == D || bz < nk0) smooth_f2_block<C, NN, UNORM>(u, rhs, n, P, events, bz);
    else smooth_f2_block<D, NN, UNORM>(u, rhs, n, P, events, bz - nk0);
}

template <int C, int D>
cudaError_t launch_smooth_f2(double* u, const double* rhs, int n, const smoothf2::Params& P, unsigned long long* ev,
                             cudaStream_t s)
{
    // colour 3 holds the larger i and j ranges of the pair (3, 4)
    const int ni = colour_count(n, C & 1), nj = colour_count(n, (C >> 1) & 1), nk0 = colour_count(n, (C >> 2) & 1);
    const int nk = nk0 + (C == D ? 0 : colour_count(n, (D >> 2) & 1));
    const dim3 grid((ni + BX - 1) / BX, (nj + BY - 1) / BY, nk), blk(BX, BY);
    count_launches(1);
    switch (n) {
    case 129: k_smooth_f2<C, D, 129, true><<<grid, blk, 0, s>>>(u, rhs, n, P, ev, nk0); break;
    case 257: k_smooth_f2<C, D, 257, true><<<grid, blk, 0, s>>>(u, rhs, n, P, ev, nk0); break;
    case 513: k_smooth_f2<C, D, 513, true><<<grid, blk, 0, s>>>(u, rhs, n, P, ev, nk0); break;
    default:
        if (n < kUnormMinN) k_smooth_f2<C, D, 0, false><<<grid, blk, 0, s>>>(u, rhs, n, P, ev, nk0);
        else k_smooth_f2<C, D, 0, true><<<grid, blk, 0, s>>>(u, rhs, n, P, ev, nk0);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sweeps of a 33^3 grid in one cluster of 16 thread blocks.  A phase there is
// one point's dependent chain (3400 cycles with the general gather, of which
// 1900 the gather) and a launch: 7 launches a sweep, 2.7 us each.  Two sweeps in
// one launch: 38 -> 29 us.  Block m holds planes 2m .. 2m + 3 of u in shared memory
// and owns the middle two, an odd and an even one; a point's new value also
// goes to the neighbour that holds its plane, and a cluster barrier ends the
// phase.  Rows are kept with the even i first, so that the points of a phase
// are contiguous.  Same point update in the same order as the launches, whose
// gather may take the other exact form.
// ---------------------------------------------------------------------------
namespace sweep33 {

constexpr int N = 33, KC = 16, TC = 512;
constexpr int RS = 34, PS = N * RS;      // row: 17 even places, then 16 odd ones
constexpr int kSmem = 6 * PS * (int)sizeof(double);

__device__ __forceinline__ int place(int i) { return (i & 1) * 17 + (i >> 1); }

// The value at offset o = di + N dj + N^2 dk of a point, all in -1 .. 1: q is
// the point's row, x its place and xm, xp those of i - 1 and i + 1.
struct At {
    const double* q;
    int x, xm, xp;
    __device__ __forceinline__ double operator()(int o) const
    {
        const int w = o + 1 + N + N * N, di = w % N - 1, dj = w / N % N - 1, dk = w / (N * N) - 1;
        return q[dk * PS + dj * RS + (di == 0 ? x : (di < 0 ? xm : xp))];
    }
};

__device__ __noinline__ double point_f64(At at, double rhs6, bool* nonconvex)
{
    const double v0 = at(0);
    const HessS H = gather_hess_of(at, N, N * N, v0);
    return fma(0.125, smallest_root(H, rhs6, nonconvex), v0);
}

__device__ __forceinline__ unsigned rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void store_remote(const double* smem, unsigned block, double v)
{
    unsigned a = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;\n" : "+r"(a) : "r"(block));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

__global__ void __launch_bounds__(TC, 1) k_sweeps(double* u, const double* __restrict__ rhs, smoothf2::Params P,
                                                  int nsweeps, unsigned long long* events)
{
    extern __shared__ double csm[];
    double *su = csm, *sr = csm + 4 * PS;
    const int m = (int)rank();
    for (int t = threadIdx.x; t < 4 * N * N; t += TC) {
        const int lp = t / (N * N), r = t - lp * N * N, j = r / N, i = r - j * N, k = 2 * m + lp;
        if (k >= N) continue;
        const int at = j * RS + place(i);
        su[lp * PS + at] = u[k * N * N + r];
        if (lp == 1 || lp == 2) sr[(lp - 1) * PS + at] = __ldg(rhs + k * N * N + r);
    }
    barrier();   // every block is running before another writes to it
    const int half = threadIdx.x >> 8, a = threadIdx.x & 15, b = (threadIdx.x >> 4) & 15;
    unsigned long long ev = 0;
    for (int q = 0, w = 0; q < 7 * nsweeps; ++q, w = w == 6 ? 0 : w + 1) {
        const int c = half == 0 ? phase_first(false, w) : phase_second(false, w);
        const int i = ((c & 1) ? 1 : 2) + 2 * a, j = ((c & 2) ? 1 : 2) + 2 * b, lp = (c & 4) ? 1 : 2;
        if (c >= 0 && i <= N - 2 && j <= N - 2 && 2 * m + lp <= N - 2) {
            const At at{su + lp * PS + j * RS, place(i), place(i - 1), place(i + 1)};
            const double bv = sr[(lp - 1) * PS + j * RS + at.x];
            double v;
            if (!smoothf2::update<true, resid::kSmall, int>(
                    [&](int o) -> long long { return __double_as_longlong(at(o)); }, N, N * N, bv, P, &v)) {
                bool nonconvex = false;
                v = point_f64(at, __dmul_rn(P.h6, bv), &nonconvex);
                ev += nonconvex ? 1 : 0;
            }
            double* p = su + lp * PS + j * RS + at.x;
            *p = v;
            if (lp == 1 && m > 0) store_remote(p + 2 * PS, m - 1, v);
            if (lp == 2 && m < KC - 1) store_remote(p - 2 * PS, m + 1, v);
        }
        barrier();
    }
    for (int t = threadIdx.x; t < 2 * N * N; t += TC) {
        const int lp = 1 + t / (N * N), r = t - (lp - 1) * N * N, j = r / N, i = r - j * N, k = 2 * m + lp;
        if (i < 1 || j < 1 || i > N - 2 || j > N - 2 || k > N - 2) continue;
        u[k * N * N + r] = su[lp * PS + j * RS + place(i)];
    }
    if (events && ev) atomicAdd(events, ev);
}

cudaLaunchConfig_t config(cudaLaunchAttribute* at, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(KC);
    cfg.blockDim = dim3(TC);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = KC;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Whether the current device runs such a cluster; the answer and the kernel's
// limits are set once per device.
bool ready()
{
    static std::atomic<signed char> known[64];   // 0: not asked, 1: yes, -1: no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    signed char k = known[dev].load(std::memory_order_acquire);
    if (k == 0) {
        cudaLaunchAttribute at{};
        const cudaLaunchConfig_t cfg = config(&at, nullptr);
        int clusters = 0;
        const bool ok =
            cudaFuncSetAttribute(k_sweeps, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) == cudaSuccess &&
            cudaFuncSetAttribute(k_sweeps, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k_sweeps, &cfg) == cudaSuccess && clusters > 0;
        if (!ok) (void)cudaGetLastError();
        k = ok ? 1 : -1;
        known[dev].store(k, std::memory_order_release);
    }
    return k > 0;
}

cudaError_t launch(double* u, const double* rhs, const smoothf2::Params& P, int nsweeps, unsigned long long* events,
                   cudaStream_t s)
{
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config(&at, s);
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, k_sweeps, u, rhs, P, nsweeps, events);
}

}  // namespace sweep33

// ---------------------------------------------------------------------------
// Block reduction of (max |x|, sum x^2) in a fixed order (deterministic).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void block_reduce_store(unsigned long long mx, double ss, double* partials, int slot)
{
    __shared__ unsigned long long smx[BX * BY / 32];
    __shared__ double sss[BX * BY / 32];
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_down_sync(0xffffffffu, mx, o));
        ss += __shfl_down_sync(0xffffffffu, ss, o);
    }
    const int t = threadIdx.y * BX + threadIdx.x;
    if ((t & 31) == 0) { smx[t >> 5] = mx; sss[t >> 5] = ss; }
    __syncthreads();
    if (t == 0) {
        unsigned long long m = smx[0];
        double q = sss[0];
        for (int w = 1; w < BX * BY / 32; ++w) { m = max(m, smx[w]); q += sss[w]; }
        partials[2 * slot] = __longlong_as_double((long long)m);
        partials[2 * slot + 1] = q;
    }
}

// x in FP64, by integer operations where it is normal or zero
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    return b == 0 || b - 0x00800000u < 0x7f000000u ? f2d(x) : (double)x;
}

constexpr int KZ = 16;   // z-blocks of the reduction grids; each loops over k

dim3 reduce_grid(int n) { return dim3((n + BX - 1) / BX, (n + BY - 1) / BY, n < KZ ? n : KZ); }

template <typename T>
__device__ __forceinline__ void norm_partials_block(const T* __restrict__ v, int n, double* partials, uint3 bid,
                                                    uint3 gdim)
{
    const int i = bid.x * BX + threadIdx.x;
    const int j = bid.y * BY + threadIdx.y;
    unsigned long long mx = 0;
    double ss = 0.0;
    if (i > 0 && j > 0 && i < n - 1 && j < n - 1) {
        for (int k = bid.z == 0 ? (int)gdim.z : (int)bid.z; k < n - 1; k += gdim.z) {
            const double x = widen(v[lin(i, j, k, n)]);
            mx = resid::max_bits(mx, x);
            ss = fma(x, x, ss);
        }
    }
    block_reduce_store(mx, ss, partials, (bid.z * gdim.y + bid.y) * gdim.x + bid.x);
}

template <typename T>
__global__ void __launch_bounds__(BX * BY) k_norm_partials(const T* __restrict__ v, int n, double* partials)
{
    norm_partials_block<T>(v, n, partials, blockIdx, gridDim);
}

// One block folds the partials in a fixed order: out2 = (max, sqrt(h^3 sum)).
__global__ void __launch_bounds__(resid::NF) k_norm_final(const double* __restrict__ partials, int count, double h3,
                                                          double* out2)
{
    resid::norm_final_block(partials, count, h3, out2);
}

// b_H = det(D^2_H w_H) + r_H on the interior, 0 on the shell.
__device__ __forceinline__ void coarse_rhs_block(const double* __restrict__ wc, const double* __restrict__ rc,
                                                 double* __restrict__ bc, int nc, double inv_H6, uint3 bid)
{
    const int I = bid.x * BX + threadIdx.x;
    const int J = bid.y * BY + threadIdx.y;
    const int K = bid.z;
    if (I >= nc || J >= nc) return;
    const long long p = lin(I, J, K, nc);
    double b = 0.0;
    if (I > 0 && J > 0 && K > 0 && I < nc - 1 && J < nc - 1 && K < nc - 1) {
        const HessS H = gather_hess(wc, p, nc, (long long)nc * nc, wc[p]);
        b = fma(det0(H), inv_H6, rc[p]);
    }
    bc[p] = b;
}

__global__ void __launch_bounds__(BX * BY) k_coarse_rhs(const double* __restrict__ wc, const double* __restrict__ rc,
                                                        double* __restrict__ bc, int nc, double inv_H6)
{
    coarse_rhs_block(wc, rc, bc, nc, inv_H6, blockIdx);
}

// r + det(D^2_h u) (SIGN = 1, the coarse right-hand side) or r - det (SIGN = -1,
// the residual) at a point, with exact integer second differences and a
// two-float determinant, added to r in FP64; ld as gather_f2_of takes it, q the
// centre's place.
template <int SIGN, bool UNORM, int FORM, typename Idx, typename Ld>
__device__ __forceinline__ double operator_of(Ld ld, const double* q, Idx sy, Idx sz, double rv, const resid::Scaling& P)
{
    using namespace resid;
    f2::F2 H[6];
    long long b0;
    if (P.kexp != kNone && gather_f2_of<FORM, Idx>(ld, sy, sz, P.kexp, H, &b0)) {
        const f2::F2 d = f2::det3<UNORM>(H[0], H[1], H[2], H[3], H[4], H[5]);
        if (usable(d, rv)) return fma(SIGN * (f2d(d.hi) + f2d(d.lo)), P.inv_c, rv);
    }
    return operator_f64(q, sy, sz, rv, P.inv_h6, SIGN);
}

// At a point of a grid in shared memory (q points at it).
template <int SIGN, bool UNORM>
__device__ __forceinline__ double operator_point(const double* q, int sy, int sz, double rv, const resid::Scaling& P)
{
    return operator_of<SIGN, UNORM, resid::kSmall, int>(
        [q](int o) -> long long { return __double_as_longlong(q[o]); }, q, sy, sz, rv, P);
}

// Over a grid, 0 on the shell: one point a thread, the grid size at compile time
// for the sizes of a hierarchy's larger levels.  The FP64 forms of the two were
// bound by the FP64 pipe (257^3: 754 us residual, 800 us right-hand side); this
// one by issue, 240 us at 257^3, 35 against 98 at 129^3, 8.7 against 22 at 65^3,
// 3.9 against 7.2 at 33^3 (Example 4, graph replay; nine resident blocks, 56
// registers and 8 bytes of spills, against eight: 253 us at 257^3).  Runs of
// planes a thread, as the residual with norms walks them, keep more values live
// (76 registers for 64): 297 us.
template <int NN, int SIGN, bool UNORM>
__global__ void __launch_bounds__(BX * BY, NN > 0 ? 9 : (UNORM ? 8 : 6))
    k_operator_f2(const double* __restrict__ u, const double* __restrict__ r, double* __restrict__ out, int n_rt,
                  resid::Scaling P)
{
    const int n = NN > 0 ? NN : n_rt;
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= n || j >= n) return;
    const long long p = lin(i, j, k, n), sz = (long long)n * n;
    if (i == 0 || j == 0 || k == 0 || i == n - 1 || j == n - 1 || k == n - 1) {
        out[p] = 0.0;
        return;
    }
    const long long* q = reinterpret_cast<const long long*>(u) + p;
    out[p] = operator_of<SIGN, UNORM, UNORM ? resid::kDirect : resid::kSmall, long long>(
        [q](long long o) -> long long { return __ldg(q + o); }, u + p, n, sz, __ldg(r + p), P);
}

template <int SIGN>
cudaError_t launch_operator_f2(const double* u, const double* r, double* out, int n, const resid::Scaling& P,
                               cudaStream_t s)
{
    const dim3 g = xfer::grid_of(n), b(BX, BY);
    switch (n) {
    case 33: k_operator_f2<33, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P); break;
    case 65: k_operator_f2<65, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P); break;
    case 129: k_operator_f2<129, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P); break;
    case 257: k_operator_f2<257, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P); break;
    case 513: k_operator_f2<513, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P); break;
    default:
        if (n < kUnormMinN) k_operator_f2<0, SIGN, false><<<g, b, 0, s>>>(u, r, out, n, P);
        else k_operator_f2<0, SIGN, true><<<g, b, 0, s>>>(u, r, out, n, P);
    }
    return cudaGetLastError();
}

// rhs := f, u := g (whole grids); counts interior points with f not finite
// or f <= 0 and shell points with g not finite.
__global__ void k_copy_rhs_bc(const double* __restrict__ f, const double* __restrict__ g, double* __restrict__ rhs,
                              double* __restrict__ u, int n, int* bad)
{
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= n || j >= n) return;
    const long long p = lin(i, j, k, n);
    const double fv = f[p], gv = g[p];
    rhs[p] = fv;
    u[p] = gv;
    const bool interior = i > 0 && j > 0 && k > 0 && i < n - 1 && j < n - 1 && k < n - 1;
    const bool ok = interior ? (isfinite(fv) && fv > 0.0 && isfinite(gv)) : isfinite(gv);
    if (!ok) atomicAdd(bad, 1);
}

// ---------------------------------------------------------------------------
// Grids of n <= 17 in one thread block (ma_small_grid.cuh): sweeps, the
// coarsest solve, the fused tail.  From 5^3 up the points take the two-float
// forms, as the separate launches do: one warp's chain of 47 FP64 operations
// holds its scheduler's FP64 unit for about 3000 cycles a phase, the two-float
// chain takes about 1100.
// ---------------------------------------------------------------------------
constexpr int COARSE_THREADS = 256;

struct Grid64 {
    double* u;
    const double* rhs;
    const int* tab;          // phase table (ascending order), n <= 9
    smoothf2::Params P;
};

// A point's new value in FP64 throughout, with a second Newton step: the root to a few ulps.
__device__ __noinline__ double point_precise(const double* q, int sy, int sz, double rhs6, bool* nonconvex)
{
    const double v0 = q[0];
    const HessS H = gather_hess_of([&](int o) { return q[o]; }, sy, sz, v0);
    return fma(0.125, smallest_root_precise(H, rhs6, nonconvex), v0);
}

// nsw sweeps in ascending order; each(p, old, new) sees every update.  The
// grid's phase threads enter.  PRECISE: the points by point_precise.
template <bool PRECISE, typename Each>
__device__ __forceinline__ void run_sweeps64(const SmallGrid& G, const Grid64& S, int nsw, int nt,
                                             unsigned long long* ev, Each each)
{
    const int n = G.n, tid = threadIdx.x;
    auto update = [&](int p) {
        const double v0 = S.u[p];
        bool nonconvex = false;
        const double v = PRECISE ? point_precise(S.u + p, n, n * n, __dmul_rn(S.P.h6, S.rhs[p]), &nonconvex)
                                 : smoothf2::point_sm(S.u + p, n, n * n, S.rhs[p], S.P, &nonconvex);
        S.u[p] = v;
        *ev += nonconvex ? 1ull : 0ull;
        each(v0, v);
    };
    if (n <= 9) {
        int cur = S.tab[tid];
        for (int q = 0, w = 0; q < 7 * nsw; ++q) {
            w = w == 6 ? 0 : w + 1;
            const int nxt = S.tab[w * nt + tid];
            if (cur >= 0) update(cur & 0xffff);
            phase_barrier(n);
            cur = nxt;
        }
        return;
    }
    for (int q = 0, w = 0; q < 7 * nsw; ++q, w = w == 6 ? 0 : w + 1) {
        const int c = phase_first(false, w), d = phase_second(false, w);
        const int tot = G.count(c) + (d >= 0 ? G.count(d) : 0);
        for (int t = tid; t < tot; t += nt) update(phase_point(G, false, w, t) & 0xffff);
        phase_barrier(n);
    }
}

// Newton's method on the 5^3 grid (27 unknowns) by one warp, from the current
// iterate: the sweeps converge by a factor of 0.6, 40 - 70 of them to 1e-14,
// each 7 phases long.  Lane = interior point.  The residuals and their FP32
// Jacobian come from the two-float Hessian; the Jacobian is inverted in place
// (Gauss-Jordan) and kept while an iteration cuts the residual fourfold.  It
// starts from an iterate whose points are all positive definite, with positive
// right-hand sides; where they are not positive definite (FMG's zero interior)
// from the solution of the Poisson equation with right-hand side
// 3 rhs^(1/3), which a convex solution exceeds and mostly lies near.  If the
// residual does not fall, or a step leaves a point that is not positive definite
// or out of range, the iterate is put back.  True
// when the changes that a sweep would make (each point's residual over its
// derivative) are at most 1e-14 max |u|, the sweeps' own rule; otherwise the
// caller's sweeps decide as they would have.  finest: the grid is no other's
// correction, and the last step takes its residual in FP64 (3000 cycles), which on
// 5^3 rounds less than the two-float determinant does.  J: 27 x kJ floats.
constexpr int kJ = 29;   // an odd stride: a lane's row and a column of it meet no bank conflicts

__device__ __forceinline__ bool newton5(double* u, const double* rhs, const smoothf2::Params& P, float* J, bool finest)
{
    using namespace resid;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool on = lane < 27;
    const int a = on ? lane : 0;
    const int i = 1 + a % 3, j = 1 + (a / 3) % 3, k = 1 + a / 9, p = (k * 5 + j) * 5 + i;
    const double b = rhs[p], start = u[p];
    const f2::F2 r6 = f2::from_f64(__dmul_rn(P.c, b));
    float last = 0.0f;
    bool moved = false, laplace = false;
    auto step = [&](float g) {   // u -= J^-1 g
        float d = 0.0f;
        for (int c = 0; c < 27; ++c) {
            const float gc = __shfl_sync(FULL, g, c);
            if (on) d = fmaf(-J[lane * kJ + c], gc, d);
        }
        __syncwarp();   // every lane has read what it needs of u
        if (on) u[p] = fma(8.0 * P.kz, f2d(d), u[p]);
        __syncwarp();
    };
    for (int it = 0; it < 24; ++it) {
        f2::F2 H[6];
        long long b0;
        auto ld = [&](int o) -> long long { return __double_as_longlong(u[p + o]); };
        bool usable = gather_f2_of<kSmall, int>(ld, 5, 25, P.kexp, H, &b0);
        if (!usable && ((ld(0) | ld(1) | ld(-1) | ld(5) | ld(-5) | ld(25) | ld(-25)) << 1) == 0) {
            usable = true;   // a zero interior's centre: no Hessian there, which is a Laplacian of 0
            H[0] = H[1] = H[2] = H[3] = H[4] = H[5] = f2::F2{0.0f, 0.0f};
        }
        usable = usable && __double_as_longlong(b) > 0;
        bool ok = usable;
        float g = 0.0f, m = 0.0f;
        if (ok) {
            const f2::F2 d = f2::det3(H[0], H[1], H[2], H[3], H[4], H[5]);
            const f2::F2 e = f2::add(d, f2::neg(r6));
            g = e.hi + e.lo;
            HessSf F;
            F.A = H[0].hi; F.B = H[1].hi; F.C = H[2].hi;
            F.R = H[3].hi; F.S = H[4].hi; F.T = H[5].hi;
            const float scale = fabsf(F.A) + fabsf(F.B) + fabsf(F.C) + fabsf(F.R) + fabsf(F.S) + fabsf(F.T);
            m = minors_shift_f(F, 0.0f);
            ok = is_pd<HessSf, float>(F, d.hi) && m > 0.05f * scale * scale && scale > 9.5e-7f &&
                 scale < 1.0e9f && isfinite(g);
        }
        float worst = fabsf(g);
        for (int o = 16; o > 0; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(FULL, worst, o));
        const bool bad = __any_sync(FULL, on && !ok);
        const bool start_laplace = bad && !moved && !laplace && __all_sync(FULL, !on || usable);
        if (!start_laplace && (bad || (moved && !(worst < last)))) {
            // not a point Newton can be trusted from (its residual is not known), or the residual no longer falls:
            // put the iterate back, unless that is round-off
            if (bad || !__all_sync(FULL, !on || worst <= 1e-11f * fabsf(r6.hi))) {
                __syncwarp();
                if (on) u[p] = start;
                __syncwarp();
                return false;
            }
            double big = on ? fabs(__longlong_as_double(b0)) : 0.0;
            for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(FULL, big, o));
            const bool done = __all_sync(FULL, !on || fabsf(g) * (float)P.kz <= 1e-14f * (float)big * m);
            if (done && finest) {
                const HessS G = gather_hess_of([&](int o) { return u[p + o]; }, 5, 25, u[p]);
                step((float)fma(det0(G), P.kh * P.kh * P.kh, -__dmul_rn(P.c, b)));
            }
            return done;
        }
        if (start_laplace) g = H[0].hi + H[1].hi + H[2].hi - 3.0f * cbrtf(r6.hi);
        if (!moved || worst > 0.25f * last) {
            // row of the Jacobian: the cofactors times the stencil's weights, 2^k taken out
            const float A = H[0].hi, B = H[1].hi, C = H[2].hi, R = H[3].hi, S = H[4].hi, T = H[5].hi;
            const bool lp = start_laplace;
            const float cA = lp ? 1.0f : B * C - T * T, cB = lp ? 1.0f : A * C - S * S, cC = lp ? 1.0f : A * B - R * R;
            const float cR = lp ? 0.0f : S * T - R * C, cS = lp ? 0.0f : R * T - S * B, cT = lp ? 0.0f : R * S - T * A;
            float* row = J + lane * kJ;
            if (on) {
                for (int c = 0; c < 27; ++c) row[c] = 0.0f;
                auto add = [&](int di, int dj, int dk, float w) {
                    const int x = i + di, y = j + dj, z = k + dk;
                    if (x >= 1 && x <= 3 && y >= 1 && y <= 3 && z >= 1 && z <= 3)
                        row[(x - 1) + 3 * (y - 1) + 9 * (z - 1)] = w;
                };
                add(0, 0, 0, -8.0f * (cA + cB + cC));
                add(1, 0, 0, 4.0f * cA); add(-1, 0, 0, 4.0f * cA);
                add(0, 1, 0, 4.0f * cB); add(0, -1, 0, 4.0f * cB);
                add(0, 0, 1, 4.0f * cC); add(0, 0, -1, 4.0f * cC);
                add(1, 1, 0, 2.0f * cR); add(-1, -1, 0, 2.0f * cR); add(1, -1, 0, -2.0f * cR); add(-1, 1, 0, -2.0f * cR);
                add(1, 0, 1, 2.0f * cS); add(-1, 0, -1, 2.0f * cS); add(1, 0, -1, -2.0f * cS); add(-1, 0, 1, -2.0f * cS);
                add(0, 1, 1, 2.0f * cT); add(0, -1, -1, 2.0f * cT); add(0, 1, -1, -2.0f * cT); add(0, -1, 1, -2.0f * cT);
            }
            __syncwarp();
            for (int q = 0; q < 27; ++q) {   // in-place Gauss-Jordan; no pivoting: the matrix is near a definite one
                const float piv = __fdividef(1.0f, J[q * kJ + q]);
                const float f = on ? row[q] : 0.0f;
                __syncwarp();
                if (lane < 27) J[q * kJ + lane] = lane == q ? piv : J[q * kJ + lane] * piv;   // the pivot's row
                __syncwarp();
                if (on && lane != q) {
#pragma unroll 9
                    for (int c = 0; c < 27; ++c) row[c] = c == q ? -f * piv : fmaf(-f, J[q * kJ + c], row[c]);
                }
                __syncwarp();
            }
        }
        step(g);
        if (start_laplace) {
            laplace = true;
            continue;
        }
        last = worst;
        moved = true;
    }
    return false;
}

// The coarsest grid in shared memory: sweeps until max |du| <= 1e-14 max |u| (at
// most 100), or a fixed count; on 5^3 Newton's method first, again after every
// eighth sweep where it did not finish.  A fixed count's sweeps, and the one unknown
// of 3^3, have a second Newton step in FP64 (smallest_root_precise): one leaves
// 1e-15 of u behind on 5^3 while the points still move, which sweeps to
// convergence do not see.  Every thread of the block
// enters; ends with a block barrier.  J: 27 kJ floats.
__device__ __forceinline__ void coarsest64_sm(const Grid64& S, int n, int sweeps, bool finest, float* J,
                                              unsigned long long* ev)
{
    const int max_sweeps = sweeps > 0 ? sweeps : 100;
    const int nt = phase_threads(n, (int)blockDim.x);
    __shared__ double red[32][2];
    if (n == 3) {
        if (threadIdx.x == 0) {
            double v = S.u[13];
            for (int s = 0; s < max_sweeps; ++s) {
                const double v0 = v;
                const HessS H = gather_hess_of([&](int o) { return S.u[13 + o]; }, 3, 9, v0);
                bool nonconvex = false;
                const double z = smallest_root_precise(H, __dmul_rn(S.P.h6, S.rhs[13]), &nonconvex);
                v = fma(0.125, z, v0);
                *ev += nonconvex ? 1ull : 0ull;
                if (sweeps == 0 && fabs(v - v0) <= 1e-14 * fabs(v)) break;
            }
            S.u[13] = v;
        }
    } else if ((int)threadIdx.x < nt) {
        const SmallGrid G(n);
        if (sweeps > 0) run_sweeps64<true>(G, S, sweeps, nt, ev, [](double, double) {});
        for (int s = 0; s < max_sweeps && sweeps == 0; ++s) {
            if (n == 5 && (s & 7) == 0 && S.P.kexp != smoothf2::kNone && newton5(S.u, S.rhs, S.P, J, finest))
                break;
            double du = 0.0, um = 0.0;
            run_sweeps64<false>(G, S, 1, nt, ev, [&](double v0, double v) {
                du = fmax(du, fabs(v - v0));
                um = fmax(um, fabs(v));
            });
            for (int o = 16; o > 0; o >>= 1) {
                du = fmax(du, __shfl_xor_sync(0xffffffffu, du, o));
                um = fmax(um, __shfl_xor_sync(0xffffffffu, um, o));
            }
            if (nt > 32) {
                if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = du; red[threadIdx.x >> 5][1] = um; }
                phase_barrier(n);
                du = um = 0.0;
                for (int w = 0; w < nt / 32; ++w) { du = fmax(du, red[w][0]); um = fmax(um, red[w][1]); }
                phase_barrier(n);   // red is free again
            }
            if (du <= 1e-14 * um) break;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void coarsest64_body(double* u, const double* __restrict__ rhs, int n,
                                                const smoothf2::Params& P, int sweeps, bool finest,
                                                unsigned long long* events)
{
    extern __shared__ double sm[];
    __shared__ int tab[kPhaseTab];
    __shared__ float J[27 * kJ];
    const int m = n * n * n;
    double* su = sm;
    double* sr = sm + m;
    for (int q = threadIdx.x; q < m; q += COARSE_THREADS) { su[q] = u[q]; sr[q] = rhs[q]; }
    fill_phase_tab(tab, n, false);
    __syncthreads();
    unsigned long long ev = 0;
    coarsest64_sm(Grid64{su, sr, tab, P}, n, sweeps, finest, J, &ev);
    for (int q = threadIdx.x; q < m; q += COARSE_THREADS) u[q] = su[q];
    if (events && ev) atomicAdd(events, ev);
}

__global__ void __launch_bounds__(COARSE_THREADS) k_coarsest(double* u, const double* __restrict__ rhs, int n,
                                                             smoothf2::Params P, int sweeps, bool finest,
                                                             unsigned long long* events)
{
    coarsest64_body(u, rhs, n, P, sweeps, finest, events);
}

// ---------------------------------------------------------------------------
// The tail of an FP64 V-cycle in one block: every level with n <= 17, from
// the level the cycle enters there down to the coarsest grid and back, with
// u, w, r and rhs of those levels in shared memory.  Each step repeats the
// per-point arithmetic of its separate kernel -- the colour sweeps, the
// residual and the tau-corrected right-hand side, the restriction of
// xfer::k_restrict, the coarsest solve of k_coarsest, the prolongation of
// xfer::k_prolong -- so the result is the same bits; it replaces the ~100
// launches these latency-bound levels take by one.  FMG runs such a cycle
// from every level, so it pays most there.
// ---------------------------------------------------------------------------
constexpr int T64 = 512;

struct Tail64Level {
    int n;
    smoothf2::Params P;
    double* u;           // global iterate (read on the top level, written back there)
    const double* rhs;   // global right-hand side (read on the top level)
    int ou, ow, orr, orhs;   // places of the level's fields in shared memory, in doubles
};

struct Tail64Args {
    int nlev;
    Tail64Level lev[4];
    int nu1, nu2, kind, approx, coarse_sweeps, finest;
    unsigned long long* events;
};

__host__ __device__ inline int tail64_level_doubles(int n, bool top)
{
    const int m = n * n * n;
    return m /* u */ + (top ? 0 : m) /* w */ + m /* r */ + m /* rhs */;
}

inline void set_tail64_offsets(Tail64Args* A)
{
    int q = 0;
    for (int l = 0; l < A->nlev; ++l) {
        Tail64Level& V = A->lev[l];
        const int m = V.n * V.n * V.n;
        V.ou = q; q += m;
        V.ow = q; q += l > 0 ? m : 0;
        V.orr = q; q += m;
        V.orhs = q; q += m;
    }
}

struct Tail64Smem {
    double *u, *w, *r, *rhs;
};

__device__ __forceinline__ Tail64Smem tail64_fields(const Tail64Args& A, double* sm, int l)
{
    const Tail64Level& V = A.lev[l];
    return Tail64Smem{sm + V.ou, sm + V.ow, sm + V.orr, sm + V.orhs};
}

__device__ __forceinline__ void tail64_smooth(const Grid64& S, int n, int nsw, unsigned long long* ev)
{
    const int nt = phase_threads(n, T64);
    if ((int)threadIdx.x < nt && nsw > 0) run_sweeps64<false>(SmallGrid(n), S, nsw, nt, ev, [](double, double) {});
    __syncthreads();
}

// d: the coarse values u_H - w_H
__device__ __forceinline__ double tail64_line(const double* d, int nc, int Ic, int J0, int K0, int oj, int ok, double w)
{
    const double* q = d + (K0 * nc + J0) * nc + Ic;
    double s = 0.0 + q[0];
    if (oj) s += q[nc];
    if (ok) {
        s += q[nc * nc];
        if (oj) s += q[nc * nc + nc];
    }
    return s * w;
}

__device__ __forceinline__ void vcycle_tail_body(const Tail64Args& A)
{
    extern __shared__ double t64sm[];
    __shared__ int tab[kTailTab];
    __shared__ float J[27 * kJ];
    // inputs: the top level's iterate and right-hand side
    {
        const Tail64Smem S = tail64_fields(A, t64sm, 0);
        const int m = A.lev[0].n * A.lev[0].n * A.lev[0].n;
        for (int q = threadIdx.x; q < m; q += T64) { S.u[q] = A.lev[0].u[q]; S.rhs[q] = A.lev[0].rhs[q]; }
    }
    for (int l = 0; l < A.nlev; ++l) fill_phase_tab(tail_tab(tab, A.lev[l].n), A.lev[l].n, false);
    __syncthreads();
    unsigned long long ev = 0;
    const int L = A.nlev;
    auto grid = [&](int l) {
        const Tail64Smem S = tail64_fields(A, t64sm, l);
        return Grid64{S.u, S.rhs, tail_tab(tab, A.lev[l].n), A.lev[l].P};
    };
    for (int l = 0; l < L - 1; ++l) {
        const Tail64Smem F = tail64_fields(A, t64sm, l);
        const Tail64Smem C = tail64_fields(A, t64sm, l + 1);
        const int nf = A.lev[l].n, nc = A.lev[l + 1].n, ni = nc - 2;
        const SmallGrid GF(nf), GC(nc);
        tail64_smooth(grid(l), nf, A.nu1, &ev);                                              // (2)
        for (int q = threadIdx.x; q < (nf - 2) * (nf - 2) * (nf - 2); q += T64) {        // (3)
            int i, j, k;
            const int p = GF.interior(q, &i, &j, &k);
            F.r[p] = operator_point<-1, false>(F.u + p, nf, nf * nf, F.rhs[p], A.lev[l].P);
        }
        __syncthreads();
        // (3)-(4): the interior's two restrictions side by side (both are FP64 sums), the shell's injection
        for (int q = threadIdx.x; q < 2 * ni * ni * ni; q += T64) {
            const bool of_u = q >= ni * ni * ni;
            int I, Jc, K;
            const int pc = GC.interior(of_u ? q - ni * ni * ni : q, &I, &Jc, &K);
            const double* v = (of_u ? F.u : F.r) + ((2 * K) * nf + 2 * Jc) * nf + 2 * I;
            const double x = of_u && A.approx != 1
                                 ? v[0]
                                 : xfer::restrict_of<double>(
                                       [&](int di, int dj, int dk) -> double { return v[(dk * nf + dj) * nf + di]; },
                                       A.kind);
            if (of_u) {
                C.w[pc] = x;
                C.u[pc] = x;
            } else {
                C.r[pc] = x;
            }
        }
        for (int pc = threadIdx.x; pc < nc * nc * nc; pc += T64) {
            const int J0 = (pc * GC.mn) >> 16, K = (J0 * GC.mn) >> 16, I = pc - J0 * nc, Jc = J0 - K * nc;
            if (I > 0 && Jc > 0 && K > 0 && I < nc - 1 && Jc < nc - 1 && K < nc - 1) continue;
            const double w = F.u[((2 * K) * nf + 2 * Jc) * nf + 2 * I];
            C.w[pc] = w;
            C.u[pc] = w;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < ni * ni * ni; q += T64) {                            // (5)
            int i, j, k;
            const int p = GC.interior(q, &i, &j, &k);
            if (nc >= kF2MinN) {
                C.rhs[p] = operator_point<1, false>(C.w + p, nc, nc * nc, C.r[p], A.lev[l + 1].P);
            } else {
                const HessS H = gather_hess_of([&](int o) { return C.w[p + o]; }, nc, nc * nc, C.w[p]);
                C.rhs[p] = fma(det0(H), A.lev[l + 1].P.inv_h6, C.r[p]);
            }
        }
        __syncthreads();
    }
    coarsest64_sm(grid(L - 1), A.lev[L - 1].n, A.coarse_sweeps, A.finest != 0, J, &ev);                     // (1)
    for (int l = L - 2; l >= 0; --l) {
        const Tail64Smem F = tail64_fields(A, t64sm, l);
        const Tail64Smem C = tail64_fields(A, t64sm, l + 1);
        const int nf = A.lev[l].n, nc = A.lev[l + 1].n;
        const SmallGrid GF(nf);
        // (7)-(8) u_h += I(u_H - w_H) on the fine interior, each value formed as xfer::k_prolong forms it
        for (int q = threadIdx.x; q < nc * nc * nc; q += T64) C.w[q] = C.u[q] - C.w[q];
        __syncthreads();
        for (int q = threadIdx.x; q < (nf - 2) * (nf - 2) * (nf - 2); q += T64) {
            int i, j, k;
            const int p = GF.interior(q, &i, &j, &k);
            const int J0 = j >> 1, K0 = k >> 1, oj = j & 1, ok = k & 1;
            const double w = oj + ok == 2 ? 0.25 : (oj + ok == 1 ? 0.5 : 1.0);
            double v;
            if (i & 1) {
                const int I = i >> 1;
                const double a = tail64_line(C.w, nc, I, J0, K0, oj, ok, w);
                const double b = tail64_line(C.w, nc, I + 1, J0, K0, oj, ok, w);
                v = (a + b) * 0.5;
            } else {
                v = tail64_line(C.w, nc, i >> 1, J0, K0, oj, ok, w);
            }
            F.u[p] = F.u[p] + v;
        }
        __syncthreads();
        tail64_smooth(grid(l), nf, A.nu2, &ev);                                             // (9)
    }
    const int m0 = A.lev[0].n * A.lev[0].n * A.lev[0].n;
    for (int q = threadIdx.x; q < m0; q += T64) A.lev[0].u[q] = t64sm[A.lev[0].ou + q];
    if (A.events && ev) atomicAdd(A.events, ev);
}

__global__ void __launch_bounds__(T64, 1) k_vcycle_tail(const __grid_constant__ Tail64Args A) { vcycle_tail_body(A); }

int tail64_smem_bytes(const int* ns, int nlev)
{
    int d = 0;
    for (int l = 0; l < nlev; ++l) d += tail64_level_doubles(ns[l], l == 0);
    return d * (int)sizeof(double);
}

}  // namespace

// ---------------------------------------------------------------------------
// Batched FP64 launches (the start of a shared per-level batch): the norms
// of f and the FMG pass of Algorithm 2 over several hierarchies at once.
// With one coarsest grid size for all of them, FMG step j works on the level
// of size 2^j (coarsest_n - 1) + 1 in every hierarchy that has it, so the
// V-cycles of a step have the same level sizes everywhere.
// ---------------------------------------------------------------------------
namespace {

using batched::split_block;
using batched::TableBuilder;

enum F64OpId {
    F_PROLONG = batched::kF64Ops, F_CUBIC0, F_CUBIC1, F_CUBIC2, F_INJECT, F_ZERO, F_COARSEST, F_NORMPART
};

// add != 0: uf += I(uc - wc); add == 0: uf = I(uc) (trilinear)
struct OpProlong64 {
    static constexpr int NT = BX * BY, MINB = 1;
    struct Job {
        int inst, nc, nf, add, gx, gy;
        const double* uc;
        const double* wc;
        double* uf;
    };
    static __device__ __forceinline__ void run(const Job& J, int q)
    {
        xfer::prolong_block<double>(J.uc, J.wc, J.nc, J.uf, J.nf, J.add, split_block(q, J.gx, J.gy));
    }
};

struct CubicJob {
    int inst, nc, ox, oy, oz, interior_only, gx, gy;
    const double* in;
    double* out;
};

template <int AX>
struct OpCubic {
    static constexpr int NT = BX * BY, MINB = 1;
    using Job = CubicJob;
    static __device__ __forceinline__ void run(const Job& J, int q)
    {
        xfer::cubic_pass_block<AX>(J.in, J.out, J.nc, J.ox, J.oy, J.oz, J.interior_only, split_block(q, J.gx, J.gy));
    }
};

struct OpInject64 {
    static constexpr int NT = BX * BY, MINB = 1;
    struct Job {
        int inst, nf, nc, gx, gy;
        const double* vf;
        double* vc;
    };
    static __device__ __forceinline__ void run(const Job& J, int q)
    {
        xfer::inject_block<double>(J.vf, J.nf, J.vc, J.nc, split_block(q, J.gx, J.gy));
    }
};

struct OpZero64 {
    static constexpr int NT = BX * BY, MINB = 1;
    struct Job {
        int inst, n, gx, gy;
        double* u;
    };
    static __device__ __forceinline__ void run(const Job& J, int q)
    {
        xfer::zero_interior_block<double>(J.u, J.n, split_block(q, J.gx, J.gy));
    }
};

struct OpCoarsest64 {
    static constexpr int NT = COARSE_THREADS, MINB = 1;
    struct Job {
        int inst, n, sweeps, finest;
        smoothf2::Params P;
        double* u;
        const double* rhs;
        unsigned long long* events;
    };
    static __device__ __forceinline__ void run(const Job& J, int)
    {
        coarsest64_body(J.u, J.rhs, J.n, J.P, J.sweeps, J.finest != 0, J.events);
    }
};

struct OpNormPart64 {
    static constexpr int NT = BX * BY, MINB = 1;
    struct Job {
        int inst, n, gx, gy, gz;
        const double* v;
        double* partials;
    };
    static __device__ __forceinline__ void run(const Job& J, int q)
    {
        norm_partials_block<double>(J.v, J.n, J.partials, split_block(q, J.gx, J.gy),
                                    make_uint3((unsigned)J.gx, (unsigned)J.gy, (unsigned)J.gz));
    }
};

dim3 grid2(int n) { return dim3((n + BX - 1) / BX, (n + BY - 1) / BY, n); }

}  // namespace

void emit_rhs_partials_f64(TableBuilder& T, const BatchInstance* in, int count)
{
    std::vector<OpNormPart64::Job> jobs;
    std::vector<int> blocks;
    for (int b = 0; b < count; ++b) {
        const BatchLevel& F = in[b].lev[0];
        const dim3 g = reduce_grid(F.n);
        jobs.push_back(OpNormPart64::Job{in[b].id, F.n, (int)g.x, (int)g.y, (int)g.z, F.rhs, in[b].partials});
        blocks.push_back((int)(g.x * g.y * g.z));
    }
    T.emit(F_NORMPART, jobs, blocks, 0);
}

// Algorithm 2 as fmg(H, false) runs it: inject f and the data down, solve the
// coarsest grid from a zero interior, then up the levels: interpolate and one
// V-cycle from that level, the finest level receiving the interpolation only.
void emit_fmg_f64(TableBuilder& T, const BatchInstance* in, int count, const BatchParams& p,
                  const std::function<void(const std::vector<std::pair<int, int>>&)>& level_step)
{
    int Lmax = 0;
    for (int b = 0; b < count; ++b) Lmax = std::max(Lmax, in[b].L);
    for (int d = 0; d + 1 < Lmax; ++d)
        for (int field = 0; field < 2; ++field) {   // f, then the iterate (its shell carries g)
            std::vector<OpInject64::Job> jobs;
            std::vector<int> blocks;
            for (int b = 0; b < count; ++b) {
                if (d + 1 >= in[b].L) continue;
                const BatchLevel& F = in[b].lev[d];
                const BatchLevel& C = in[b].lev[d + 1];
                const dim3 g = grid2(C.n);
                jobs.push_back(OpInject64::Job{in[b].id, F.n, C.n, (int)g.x, (int)g.y, field ? F.u : F.rhs,
                                               field ? C.u : C.rhs});
                blocks.push_back((int)(g.x * g.y * g.z));
            }
            T.emit(F_INJECT, jobs, blocks, 0);
        }
    {
        std::vector<OpZero64::Job> zj;
        std::vector<OpCoarsest64::Job> kj;
        std::vector<int> zb, kb;
        int ksmem = 0;
        for (int b = 0; b < count; ++b) {
            const BatchLevel& V = in[b].lev[in[b].L - 1];
            const dim3 g = grid2(V.n);
            zj.push_back(OpZero64::Job{in[b].id, V.n, (int)g.x, (int)g.y, V.u});
            zb.push_back((int)(g.x * g.y * g.z));
            kj.push_back(OpCoarsest64::Job{in[b].id, V.n, p.coarse_sweeps, in[b].L == 1, smoothf2::make_params(V.h), V.u,
                                           V.rhs, in[b].events});
            kb.push_back(1);
            ksmem = std::max(ksmem, (int)(2 * sizeof(double) * (size_t)V.n * V.n * V.n));
        }
        T.emit(F_ZERO, zj, zb, 0);
        T.emit(F_COARSEST, kj, kb, ksmem);
    }
    for (int j = 1; j < Lmax; ++j) {
        // interpolation into level l = L - 1 - j of every hierarchy that has it
        std::vector<OpProlong64::Job> lj;
        std::vector<CubicJob> c0, c1, c2;
        std::vector<int> lb, b0, b1, b2;
        std::vector<std::pair<int, int>> E;
        for (int b = 0; b < count; ++b) {
            const int l = in[b].L - 1 - j;
            if (l < 0) continue;
            const BatchLevel& F = in[b].lev[l];
            const BatchLevel& C = in[b].lev[l + 1];
            const int nc = C.n, nf = F.n;
            if (p.fmg_interp == MA_FMG_CUBIC) {
                double* t1 = F.r;                              // the fine level's r is free here
                double* t2 = F.r + (size_t)nf * nc * nc;
                auto cj = [&](const double* src, double* dst, int ox, int oy, int oz, int io) {
                    return CubicJob{in[b].id, nc, ox, oy, oz, io, (ox + BX - 1) / BX, (oy + BY - 1) / BY, src, dst};
                };
                c0.push_back(cj(C.u, t1, nf, nc, nc, 0));
                b0.push_back(c0.back().gx * c0.back().gy * nc);
                c1.push_back(cj(t1, t2, nf, nf, nc, 0));
                b1.push_back(c1.back().gx * c1.back().gy * nc);
                c2.push_back(cj(t2, F.u, nf, nf, nf, 1));
                b2.push_back(c2.back().gx * c2.back().gy * nf);
            } else {
                const dim3 g = xfer::prolong_grid(nf);
                lj.push_back(OpProlong64::Job{in[b].id, nc, nf, 0, (int)g.x, (int)g.y, C.u, nullptr, F.u});
                lb.push_back((int)(g.x * g.y * g.z));
            }
            if (l >= 1) E.emplace_back(b, l);
        }
        T.emit(F_PROLONG, lj, lb, 0);
        T.emit(F_CUBIC0, c0, b0, 0);
        T.emit(F_CUBIC1, c1, b1, 0);
        T.emit(F_CUBIC2, c2, b2, 0);
        if (!E.empty()) level_step(E);
    }
}

cudaError_t batch_launch_f64(const char* tables, const batched::BLaunch& L, const int* active, cudaStream_t s)
{
    using batched::launch;
    const dim3 b2(BX, BY);
    switch (L.op) {
    case F_PROLONG: return launch<OpProlong64>(tables, L, b2, active, s);
    case F_CUBIC0: return launch<OpCubic<0>>(tables, L, b2, active, s);
    case F_CUBIC1: return launch<OpCubic<1>>(tables, L, b2, active, s);
    case F_CUBIC2: return launch<OpCubic<2>>(tables, L, b2, active, s);
    case F_INJECT: return launch<OpInject64>(tables, L, b2, active, s);
    case F_ZERO: return launch<OpZero64>(tables, L, b2, active, s);
    case F_COARSEST: return launch<OpCoarsest64>(tables, L, dim3(COARSE_THREADS), active, s);
    case F_NORMPART: return launch<OpNormPart64>(tables, L, b2, active, s);
    default: return cudaErrorInvalidValue;
    }
}

static std::atomic<unsigned long long> g_launches{0};
void count_launches(unsigned long long k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
void uncount_launches(unsigned long long k) { g_launches.fetch_sub(k, std::memory_order_relaxed); }
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// 64 h^6: determinants of the 4 Hs matrices the gathers return are 64 h^6 det(D^2 u).
static inline double pow6(double h) { const double h2 = h * h; return 64.0 * h2 * h2 * h2; }

cudaError_t launch_smooth(double* u, const double* rhs, int n, double h, int nsweeps,
                          unsigned long long* events, cudaStream_t s)
{
    const smoothf2::Params P = smoothf2::make_params(h);
    if (n >= kF2MinN && P.kexp != smoothf2::kNone) {
        if (n == sweep33::N && nsweeps > 0 && sweep33::ready()) return sweep33::launch(u, rhs, P, nsweeps, events, s);
        for (int sw = 0; sw < nsweeps; ++sw) {
            cudaError_t e;
            if ((e = launch_smooth_f2<0, 0>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<1, 1>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<2, 2>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<3, 4>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<5, 5>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<6, 6>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
            if ((e = launch_smooth_f2<7, 7>(u, rhs, n, P, events, s)) != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    return launch_smooth_f64(u, rhs, n, h, nsweeps, events, s);
}

cudaError_t launch_smooth_f64(double* u, const double* rhs, int n, double h, int nsweeps,
                              unsigned long long* events, cudaStream_t s)
{
    const double h6 = pow6(h);
    for (int sw = 0; sw < nsweeps; ++sw) {
        cudaError_t e;
        if ((e = launch_colour<0>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<1>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<2>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<3>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<4>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<5>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<6>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
        if ((e = launch_colour<7>(u, rhs, n, h6, events, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int residual_partial_count(int n)
{
    const dim3 g = reduce_grid(n);
    return (int)(g.x * g.y * g.z);
}

int norm_partial_count(int n) { return residual_partial_count(n); }

cudaError_t launch_residual(const double* u, const double* rhs, double* r, int n, double h,
                            double* partials, cudaStream_t s)
{
    const resid::Scaling P = resid::make_scaling(h);
    if (n >= kF2MinN && P.kexp != resid::kNone) {
        const dim3 g = reduce_grid(n);
        const int kchunk = (n + (int)g.z - 1) / (int)g.z;
        count_launches(1);
        if (!partials) return launch_operator_f2<-1>(u, rhs, r, n, P, s);
        const dim3 gk = resid::grid_for(n, g.z);
        if (n < kUnormMinN)
            resid::launch_k_residual_f2(gk, s, u, rhs, resid::NaturalF2Out<false>{r}, n, P, partials, kchunk);
        else
            resid::launch_k_residual_f2(gk, s, u, rhs, resid::NaturalF2Out<true>{r}, n, P, partials, kchunk);
        return cudaGetLastError();
    }
    return launch_residual_f64(u, rhs, r, n, h, partials, s);
}

cudaError_t launch_residual_f64(const double* u, const double* rhs, double* r, int n, double h, double* partials,
                                cudaStream_t s)
{
    count_launches(1);
    const dim3 g = reduce_grid(n);
    const int kchunk = (n + (int)g.z - 1) / (int)g.z;
    resid::k_residual_col<resid::NaturalF64Out><<<resid::grid_for(n, g.z), dim3(resid::RX, resid::RY), 0, s>>>(
        u, rhs, resid::NaturalF64Out{r}, n, 1.0 / pow6(h), partials, kchunk);
    return cudaGetLastError();
}

cudaError_t launch_norm_partials(const double* v, int n, double* partials, cudaStream_t s)
{
    count_launches(1);
    k_norm_partials<double><<<reduce_grid(n), dim3(BX, BY), 0, s>>>(v, n, partials);
    return cudaGetLastError();
}

cudaError_t launch_norm_partials_f32(const float* v, int n, double* partials, cudaStream_t s)
{
    count_launches(1);
    k_norm_partials<float><<<reduce_grid(n), dim3(BX, BY), 0, s>>>(v, n, partials);
    return cudaGetLastError();
}

cudaError_t launch_norm_final(const double* partials, int count, double h, double* out2, cudaStream_t s)
{
    count_launches(1);
    k_norm_final<<<1, resid::NF, 0, s>>>(partials, count, h * h * h, out2);
    return cudaGetLastError();
}

using xfer::grid_of;

cudaError_t launch_restrict_residual(const double* rf, int nf, double* rc, int kind, cudaStream_t s)
{
    const int nc = (nf + 1) / 2;
    count_launches(1);
    xfer::k_restrict<double><<<grid_of(nc), dim3(BX, BY), 0, s>>>(nullptr, rf, nf, nullptr, nullptr, rc, nc, kind, 0);
    return cudaGetLastError();
}

cudaError_t launch_restrict_solution(const double* uf, int nf, double* uc, int approx, int kind, cudaStream_t s)
{
    const int nc = (nf + 1) / 2;
    count_launches(1);
    xfer::k_restrict<double><<<grid_of(nc), dim3(BX, BY), 0, s>>>(uf, nullptr, nf, nullptr, uc, nullptr, nc, kind, approx);
    return cudaGetLastError();
}

cudaError_t launch_restrict_level(const double* uf, const double* rf, int nf, double* wc, double* uc, double* rc,
                                  int kind, int approx, cudaStream_t s)
{
    const int nc = (nf + 1) / 2;
    count_launches(1);
    xfer::k_restrict<double><<<grid_of(nc), dim3(BX, BY), 0, s>>>(uf, rf, nf, wc, uc, rc, nc, kind, approx);
    return cudaGetLastError();
}

cudaError_t launch_coarse_rhs(const double* wc, const double* rc, double* bc, int nc, double H, cudaStream_t s)
{
    count_launches(1);
    const resid::Scaling P = resid::make_scaling(H);
    if (nc >= kF2MinN && P.kexp != resid::kNone) return launch_operator_f2<1>(wc, rc, bc, nc, P, s);
    k_coarse_rhs<<<grid_of(nc), dim3(BX, BY), 0, s>>>(wc, rc, bc, nc, P.inv_h6);
    return cudaGetLastError();
}

cudaError_t launch_prolong_add(const double* uc, const double* wc, int nc, double* uf, cudaStream_t s)
{
    const int nf = 2 * nc - 1;
    count_launches(1);
    xfer::k_prolong<double><<<xfer::prolong_grid(nf), dim3(BX, BY), 0, s>>>(uc, wc, nc, uf, nf, 1);
    return cudaGetLastError();
}

cudaError_t launch_interpolate(const double* uc, int nc, double* uf, cudaStream_t s)
{
    const int nf = 2 * nc - 1;
    count_launches(1);
    xfer::k_prolong<double><<<xfer::prolong_grid(nf), dim3(BX, BY), 0, s>>>(uc, nullptr, nc, uf, nf, 0);
    return cudaGetLastError();
}

size_t interpolate_cubic_scratch(int nc)
{
    const size_t nf = 2 * (size_t)nc - 1;
    return sizeof(double) * (nf * nc * nc + nf * nf * nc);
}

// Tricubic interpolation (Algorithm 2 step 4): passes x, y, z through the
// scratch t (interpolate_cubic_scratch(nc) bytes); the fine shell is kept.
cudaError_t launch_interpolate_cubic(const double* uc, int nc, double* uf, double* t, cudaStream_t s)
{
    const int nf = 2 * nc - 1;
    double* t1 = t;                                  // nc x nc x nf
    double* t2 = t + (size_t)nf * nc * nc;           // nc x nf x nf
    auto grid = [](int ox, int oy, int oz) { return dim3((ox + BX - 1) / BX, (oy + BY - 1) / BY, oz); };
    count_launches(3);
    xfer::k_cubic_pass<0><<<grid(nf, nc, nc), dim3(BX, BY), 0, s>>>(uc, t1, nc, nf, nc, nc, 0);
    xfer::k_cubic_pass<1><<<grid(nf, nf, nc), dim3(BX, BY), 0, s>>>(t1, t2, nc, nf, nf, nc, 0);
    xfer::k_cubic_pass<2><<<grid(nf, nf, nf), dim3(BX, BY), 0, s>>>(t2, uf, nc, nf, nf, nf, 1);
    return cudaGetLastError();
}

cudaError_t launch_inject(const double* vf, int nf, double* vc, cudaStream_t s)
{
    const int nc = (nf + 1) / 2;
    count_launches(1);
    xfer::k_inject<double><<<grid_of(nc), dim3(BX, BY), 0, s>>>(vf, nf, vc, nc);
    return cudaGetLastError();
}

cudaError_t launch_zero_interior(double* u, int n, cudaStream_t s)
{
    count_launches(1);
    xfer::k_zero_interior<double><<<grid_of(n), dim3(BX, BY), 0, s>>>(u, n);
    return cudaGetLastError();
}

cudaError_t launch_copy_rhs_bc(const double* f, const double* g, double* rhs, double* u, int n, int* bad,
                               cudaStream_t s)
{
    count_launches(1);
    k_copy_rhs_bc<<<grid_of(n), dim3(BX, BY), 0, s>>>(f, g, rhs, u, n, bad);
    return cudaGetLastError();
}

cudaError_t launch_coarsest(double* u, const double* rhs, int n, double h, int sweeps, bool finest,
                            unsigned long long* events, cudaStream_t s)
{
    const size_t smem = 2 * sizeof(double) * (size_t)n * n * n;
    count_launches(1);
    k_coarsest<<<1, COARSE_THREADS, smem, s>>>(u, rhs, n, smoothf2::make_params(h), sweeps, finest, events);
    return cudaGetLastError();
}

// Largest level of the fused FP64 tail.  At 17^3 one SM's phases (512 points,
// a warp's chain on every scheduler four deep) take longer than 7 launches a
// sweep spread over the GPU, at 9^3 and below (91 points) the launches do.  FP64
// solves to 1e-10 with a bound of 5 / 9 / 17, ms: 33^3 2.95 / 2.54 / 2.90, 65^3 4.75 /
// 4.25 / 4.69, 129^3 8.95 / 8.47 / 8.94, 257^3 30.5 / 30.0 / 30.6.
constexpr int kVTailDefault = 9;
static std::atomic<int> g_vtail_max{kVTailDefault};

int vcycle_tail_max_n() { return g_vtail_max.load(std::memory_order_relaxed); }

bool set_vcycle_tail(int max_n)
{
    if (max_n == 1) max_n = kVTailDefault;
    if (!(max_n == 0 || max_n == 3 || max_n == 5 || max_n == 9 || max_n == 17)) return false;
    g_vtail_max.store(max_n, std::memory_order_relaxed);
    return true;
}

cudaError_t launch_vcycle_tail(const TailSpec64* lv, int nlev, int nu1, int nu2, int kind, int approx,
                               int coarse_sweeps, bool finest, unsigned long long* events, cudaStream_t s)
{
    if (nlev < 1 || nlev > 4) return cudaErrorInvalidValue;
    Tail64Args A{};
    A.nlev = nlev;
    int ns[4];
    for (int l = 0; l < nlev; ++l) {
        if (lv[l].n > 17 || (l > 0 && lv[l].n != (lv[l - 1].n + 1) / 2)) return cudaErrorInvalidValue;
        A.lev[l].n = ns[l] = lv[l].n;
        A.lev[l].P = smoothf2::make_params(lv[l].h);
        A.lev[l].u = lv[l].u;
        A.lev[l].rhs = lv[l].rhs;
    }
    set_tail64_offsets(&A);
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.kind = kind;
    A.approx = approx;
    A.coarse_sweeps = coarse_sweeps;
    A.finest = finest;
    A.events = events;
    count_launches(1);
    k_vcycle_tail<<<1, T64, tail64_smem_bytes(ns, nlev), s>>>(A);
    return cudaGetLastError();
}

cudaError_t prepare_coarsest_f64()
{
    (void)sweep33::ready();   // asked and set up here, outside any capture
    cudaError_t e = cudaFuncSetAttribute(k_coarsest, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(2 * sizeof(double) * 17 * 17 * 17));
    if (e != cudaSuccess) return e;
    const int tail_ns[4] = {17, 9, 5, 3};
    if ((e = cudaFuncSetAttribute(k_vcycle_tail, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  tail64_smem_bytes(tail_ns, 4))) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(batched::k_batched<OpCoarsest64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(2 * sizeof(double) * 17 * 17 * 17));
}

}  // namespace ma
