// ma_transfer.cuh -- grid transfers of the FAS V-cycle (Section 3 of Liu,
// Froese, Oberman, Xiao), templated on the element type so the FP64 cycle and
// the FP32 correction cycle run the same code.  Grids are n^3 values in
// [k][j][i] order, boundary shell included; coarse point (I, J, K) sits on fine
// point (2I, 2J, 2K), nf = 2 nc - 1.
#pragma once

#include <cuda_runtime.h>

namespace ma {
namespace xfer {

constexpr int BX = 32, BY = 4;

__device__ __forceinline__ long long lin(int i, int j, int k, int n)
{
    return ((long long)k * n + j) * n + i;
}

__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }

// Restriction I_h^H at a fine point p with strides sy, sz.  kind 0: the
// printed 7-point half weighting (6 centre + 6 faces) / 12; kind 1: 27-point
// full weighting, separable (1 2 1)/4 along each axis.  Written with explicit
// fused multiply-adds in a fixed order so that every kernel that inlines it
// rounds identically.
// at(di, dj, dk) reads the value at an offset from the point.
template <typename T, typename At>
__device__ __forceinline__ T restrict_of(At at, int kind)
{
    if (kind == 0) {
        const T faces = (at(1, 0, 0) + at(-1, 0, 0)) + (at(0, 1, 0) + at(0, -1, 0)) + (at(0, 0, 1) + at(0, 0, -1));
        return fma_t(T(6), at(0, 0, 0), faces) * (T(1) / T(12));
    }
    T acc = T(0);
#pragma unroll
    for (int dk = -1; dk <= 1; ++dk) {
        T plane = T(0);
#pragma unroll
        for (int dj = -1; dj <= 1; ++dj) {
            const T row = fma_t(T(2), at(0, dj, dk), at(-1, dj, dk) + at(1, dj, dk));
            plane = fma_t(dj == 0 ? T(2) : T(1), row, plane);
        }
        acc = fma_t(dk == 0 ? T(2) : T(1), plane, acc);
    }
    return acc * (T(1) / T(64));
}

template <typename T>
__device__ __forceinline__ T weighted_restrict(const T* __restrict__ v, long long p, long long sy, long long sz,
                                               int kind)
{
    return restrict_of<T>([&](int di, int dj, int dk) -> T { return v[p + dk * sz + dj * sy + di]; }, kind);
}

// The 27-point weighting of doubles of one sign and one binade: the weighted sum
// of the bit patterns is exact in int64, and so is its 64th, rounded once (to
// even).  The FP64 form is 28 operations on a pipe of 1/64 of the FP32 rate:
// 257^3 -> 129^3, u and r together: all the levels of a 257^3 solve 2220 us;
// with u this way 1450.  false where the values differ in sign or exponent, or are zero, denormal or not finite.
__device__ __forceinline__ bool restrict_binade(const double* __restrict__ v, long long p, long long sy, long long sz,
                                                double* out)
{
    const long long* q = reinterpret_cast<const long long*>(v) + p;
    const long long b0 = __ldg(q);
    const unsigned h0 = (unsigned)(b0 >> 32);
    unsigned diff = 0;
    long long sum = 0;   // of the differences from b0: below 2^58
#pragma unroll
    for (int dk = -1; dk <= 1; ++dk)
#pragma unroll
        for (int dj = -1; dj <= 1; ++dj) {
            const long long* row = q + dk * sz + dj * sy;
            const long long a = __ldg(row - 1), b = dj == 0 && dk == 0 ? b0 : __ldg(row), c = __ldg(row + 1);
            diff |= ((unsigned)(a >> 32) ^ h0) | ((unsigned)(b >> 32) ^ h0) | ((unsigned)(c >> 32) ^ h0);
            sum += ((a - b0) + (c - b0) + 2 * (b - b0)) << ((dj == 0) + (dk == 0));
        }
    const int E = (int)((h0 >> 20) & 0x7ff);
    if ((diff >> 20) != 0 || E == 0 || E == 0x7ff) return false;
    const long long f = sum >> 6, up = (sum & 63) + 31 + ((b0 + f) & 1);
    *out = __longlong_as_double(b0 + f + (up >> 6));
    return true;
}

constexpr int kBinadeMinN = 33;   // fine grids of fewer points a side: FP64, as the cycles' tail restricts them

// Coarse-grid outputs, any may be null: rc = I r (0 on the shell);
// wc = approximation restriction of uf (approx 0: injection everywhere;
// 1: the kind weighting inside, injection on the shell); uc = copy of wc.
// The block body takes its block index as an argument, so that a batched
// launch over the grids of several hierarchies runs the same code.
template <typename T>
__device__ __forceinline__ void restrict_block(const T* __restrict__ uf, const T* __restrict__ rf, int nf,
                                               T* __restrict__ wc, T* __restrict__ uc, T* __restrict__ rc, int nc,
                                               int kind, int approx, uint3 bid)
{
    const int I = bid.x * BX + threadIdx.x;
    const int J = bid.y * BY + threadIdx.y;
    const int K = bid.z;
    if (I >= nc || J >= nc) return;
    const long long pc = lin(I, J, K, nc);
    const long long pf = lin(2 * I, 2 * J, 2 * K, nf);
    const long long sy = nf, sz = (long long)nf * nf;
    const bool interior = I > 0 && J > 0 && K > 0 && I < nc - 1 && J < nc - 1 && K < nc - 1;
    if (rc) rc[pc] = interior ? weighted_restrict(rf, pf, sy, sz, kind) : T(0);
    if (uf) {
        T w;
        bool done = false;
        if constexpr (sizeof(T) == sizeof(double))
            done = interior && approx == 1 && kind == 1 && nf >= kBinadeMinN && restrict_binade(uf, pf, sy, sz, &w);
        if (!done) w = (interior && approx == 1) ? weighted_restrict(uf, pf, sy, sz, kind) : uf[pf];
        if (wc) wc[pc] = w;
        if (uc) uc[pc] = w;
    }
}

template <typename T>
__global__ void __launch_bounds__(BX * BY) k_restrict(const T* __restrict__ uf, const T* __restrict__ rf, int nf,
                                                      T* __restrict__ wc, T* __restrict__ uc, T* __restrict__ rc,
                                                      int nc, int kind, int approx)
{
    restrict_block<T>(uf, rf, nf, wc, uc, rc, nc, kind, approx, blockIdx);
}

// Trilinear interpolation at fine interior points: along each axis an even
// index sits on a coarse point, an odd one halfway between two.  With L(I) the
// coarse values d = uc - wc (add != 0) or d = uc (add == 0) summed over the
// one, two or four coarse rows around fine row (j, k) and scaled by their
// weight, fine point 2I gets L(I) and fine point 2I + 1 gets
// (L(I) + L(I + 1)) / 2.
// add != 0: uf += I(uc - wc) (coarse-grid correction); add == 0: uf = I(uc).
//
// Thread (I, J, K) owns the coarse cell between coarse points I..I+1,
// J..J+1, K..K+1: the four fine rows j in {2J, 2J + 1}, k in {2K, 2K + 1}
// (rows on the shell skipped) and two fine points of each.  It loads the four
// coarse rows' values at column I + 1 once for all four fine rows and takes
// those at column I from the lane before it (lane 0 loads them).  nf is odd,
// so in fine row (j, k) the point pair that starts at an even linear index is
// (2I, 2I + 1) when j + k is even and (2I + 1, 2I + 2) when it is odd: each
// lane moves that pair as one aligned 2-element access (scalar accesses
// where the pair would reach the shell, or where uf is not aligned to two
// elements).  With add != 0 the fine pairs are loaded first, so their HBM
// latency overlaps the coarse loads.  Every fine value is the same
// expression, summed in the same order (dk outer, dj inner), as one thread
// per fine point would form it.
// Grid: prolong_grid(nf), blocks of BX x BY.
template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
    using type = float2;
};
template <>
struct Vec2<double> {
    using type = double2;
};

template <typename T>
__device__ __forceinline__ void prolong_block(const T* __restrict__ uc, const T* __restrict__ wc, int nc,
                                              T* __restrict__ uf, int nf, int add, uint3 bid)
{
    using V = typename Vec2<T>::type;
    const int I = bid.x * BX + threadIdx.x;
    const int J = bid.y * BY + threadIdx.y;
    const int K = bid.z;
    const bool act = I <= nc - 2 && J <= nc - 2;   // J uniform over the warp (BX = 32)
    const bool vec = ((unsigned long long)uf & (2 * sizeof(T) - 1)) == 0;
    // the fine pair of row (j, k): its first point p0 and whether both points
    // are interior (else only the second, 2I + 1, for even rows at I = 0, or
    // only the first, 2I + 1, for odd rows at the far end)
    auto pair_at = [&](int j, int k, long long* p0, bool* full) {
        const bool even = ((j + k) & 1) == 0;
        *p0 = lin(even ? 2 * I : 2 * I + 1, j, k, nf);
        *full = even ? I >= 1 : 2 * I + 2 <= nf - 2;
        return even;
    };
    T f[2][2][2];
#pragma unroll
    for (int ok = 0; ok < 2; ++ok)
#pragma unroll
        for (int oj = 0; oj < 2; ++oj) {
            f[ok][oj][0] = f[ok][oj][1] = T(0);
            const int j = 2 * J + oj, k = 2 * K + ok;
            if (!add || !act || j < 1 || k < 1) continue;
            long long p0;
            bool full;
            const bool even = pair_at(j, k, &p0, &full);
            if (full && vec) {
                const V v = *reinterpret_cast<const V*>(uf + p0);
                f[ok][oj][0] = v.x;
                f[ok][oj][1] = v.y;
            } else {
                if (full || !even) f[ok][oj][0] = uf[p0];
                if (full || even) f[ok][oj][1] = uf[p0 + 1];
            }
        }
    // The four rows' sums of d at column I + 1, and those at column I from the
    // lane before (lane 0 forms them).  No sum starts from 0 and the weights,
    // powers of two, go into the final multiply-add: the same rounding as
    // scaling first, in 28 operations a cell in place of 48 (FP64, the bound of
    // that type: all the levels of a 257^3 solve 1480 -> 1030 us).
    auto sums = [&](int col, T s[2][2]) {
        T d[2][2];
#pragma unroll
        for (int dk = 0; dk < 2; ++dk)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj) {
                const long long q = lin(col, J + dj, K + dk, nc);
                d[dk][dj] = add ? uc[q] - wc[q] : uc[q];
            }
        s[0][0] = d[0][0];
        s[0][1] = d[0][0] + d[0][1];
        s[1][0] = d[0][0] + d[1][0];
        s[1][1] = (s[0][1] + d[1][0]) + d[1][1];
    };
    T sb[2][2] = {}, sa[2][2];   // [ok][oj]
    if (act) sums(I + 1, sb);
#pragma unroll
    for (int ok = 0; ok < 2; ++ok)
#pragma unroll
        for (int oj = 0; oj < 2; ++oj) sa[ok][oj] = __shfl_up_sync(0xffffffffu, sb[ok][oj], 1);
    if (!act) return;
    if (threadIdx.x == 0) sums(I, sa);
#pragma unroll
    for (int ok = 0; ok < 2; ++ok)
#pragma unroll
        for (int oj = 0; oj < 2; ++oj) {
            const int j = 2 * J + oj, k = 2 * K + ok;
            if (j < 1 || k < 1) continue;
            const T w = T(1) / T(1 << (oj + ok)), m = sa[ok][oj] + sb[ok][oj];
            long long p0;
            bool full;
            const bool even = pair_at(j, k, &p0, &full);
            // the values at p0, p0 + 1: column I and the midpoint, or the midpoint and column I + 1
            const T x0 = even ? sa[ok][oj] : m, x1 = even ? m : sb[ok][oj];
            const T w0 = even ? w : w * T(0.5), w1 = even ? w * T(0.5) : w;
            const T r0 = add ? fma_t(x0, w0, f[ok][oj][0]) : x0 * w0, r1 = add ? fma_t(x1, w1, f[ok][oj][1]) : x1 * w1;
            if (full && vec) {
                V v;
                v.x = r0;
                v.y = r1;
                *reinterpret_cast<V*>(uf + p0) = v;
            } else {
                if (full || !even) uf[p0] = r0;
                if (full || even) uf[p0 + 1] = r1;
            }
        }
}

template <typename T>
__global__ void __launch_bounds__(BX * BY) k_prolong(const T* __restrict__ uc, const T* __restrict__ wc, int nc,
                                                     T* __restrict__ uf, int nf, int add)
{
    prolong_block<T>(uc, wc, nc, uf, nf, add, blockIdx);
}

// One thread per coarse cell (I, J, K), I, J, K in [0, nc - 2].
inline dim3 prolong_grid(int nf)
{
    const int nc = (nf + 1) / 2;
    return dim3((nc - 1 + BX - 1) / BX, (nc - 1 + BY - 1) / BY, nc - 1);
}

// Cubic interpolation (Algorithm 2 step 4) as three 1-D passes, x then y
// then z.  Along an axis, fine index i on a coarse grid of nc points: even i
// is coarse point i/2; odd i, halfway between coarse I0 = (i-1)/2 and I0 + 1,
// takes the cubic through four coarse neighbours -- I0-1 .. I0+2 with weights
// (-1, 9, 9, -1)/16, or the four nearest ones next to either end ((5, 15, -5,
// 1)/16 from the left end, mirrored at the right) -- a 3-point grid the
// quadratic (3, 6, -1)/8 (mirrored for the second interval), a 2-point grid
// the midpoint.  Returns the first coarse index and fills up to 4 weights.
__device__ __forceinline__ int cubic_axis(int i, int nc, double w[4], int* cnt)
{
    if ((i & 1) == 0) {
        w[0] = 1.0;
        *cnt = 1;
        return i >> 1;
    }
    const int I0 = i >> 1;
    if (nc == 2) {
        w[0] = w[1] = 0.5;
        *cnt = 2;
        return 0;
    }
    if (nc == 3) {
        *cnt = 3;
        if (I0 == 0) { w[0] = 0.375; w[1] = 0.75; w[2] = -0.125; }
        else { w[0] = -0.125; w[1] = 0.75; w[2] = 0.375; }
        return 0;
    }
    *cnt = 4;
    if (I0 == 0) {
        w[0] = 0.3125; w[1] = 0.9375; w[2] = -0.3125; w[3] = 0.0625;
        return 0;
    }
    if (I0 == nc - 2) {
        w[0] = 0.0625; w[1] = -0.3125; w[2] = 0.9375; w[3] = 0.3125;
        return nc - 4;
    }
    w[0] = -0.0625; w[1] = 0.5625; w[2] = 0.5625; w[3] = -0.0625;
    return I0 - 1;
}

// One pass along axis AX (0 = x, 1 = y, 2 = z): out has dims ox x oy x oz
// ([z][y][x], x fastest), in has the same dims except nc along AX.  A thread
// per output point (threads run along x); interior_only writes only points
// with every index in 1 .. dim-2 (the last pass, which keeps the Dirichlet
// shell of the target).
template <int AX>
__device__ __forceinline__ void cubic_pass_block(const double* __restrict__ in, double* __restrict__ out, int nc,
                                                 int ox, int oy, int oz, int interior_only, uint3 bid)
{
    const int x = bid.x * BX + threadIdx.x;
    const int y = bid.y * BY + threadIdx.y;
    const int z = bid.z;
    if (x >= ox || y >= oy) return;
    if (interior_only && (x < 1 || x > ox - 2 || y < 1 || y > oy - 2 || z < 1 || z > oz - 2)) return;
    const int ix = AX == 0 ? nc : ox, iy = AX == 1 ? nc : oy;
    const int a = AX == 0 ? x : (AX == 1 ? y : z);
    double w[4];
    int cnt;
    const int I = cubic_axis(a, nc, w, &cnt);
    const long long step = AX == 0 ? 1 : (AX == 1 ? (long long)ix : (long long)ix * iy);
    const int xi = AX == 0 ? I : x, yi = AX == 1 ? I : y, zi = AX == 2 ? I : z;
    const double* src = in + ((long long)zi * iy + yi) * ix + xi;
    double s = w[0] * src[0];
    for (int q = 1; q < cnt; ++q) s = fma(w[q], src[q * step], s);
    out[((long long)z * oy + y) * ox + x] = s;
}

template <int AX>
__global__ void __launch_bounds__(BX * BY) k_cubic_pass(const double* __restrict__ in, double* __restrict__ out,
                                                        int nc, int ox, int oy, int oz, int interior_only)
{
    cubic_pass_block<AX>(in, out, nc, ox, oy, oz, interior_only, blockIdx);
}

template <typename T>
__device__ __forceinline__ void inject_block(const T* __restrict__ vf, int nf, T* __restrict__ vc, int nc, uint3 bid)
{
    const int I = bid.x * BX + threadIdx.x;
    const int J = bid.y * BY + threadIdx.y;
    const int K = bid.z;
    if (I >= nc || J >= nc) return;
    vc[lin(I, J, K, nc)] = vf[lin(2 * I, 2 * J, 2 * K, nf)];
}

template <typename T>
__global__ void k_inject(const T* __restrict__ vf, int nf, T* __restrict__ vc, int nc)
{
    inject_block<T>(vf, nf, vc, nc, blockIdx);
}

template <typename T>
__device__ __forceinline__ void zero_interior_block(T* u, int n, uint3 bid)
{
    const int i = bid.x * BX + threadIdx.x;
    const int j = bid.y * BY + threadIdx.y;
    const int k = bid.z;
    if (i < 1 || j < 1 || k < 1 || i > n - 2 || j > n - 2 || k > n - 2) return;
    u[lin(i, j, k, n)] = T(0);
}

template <typename T>
__global__ void k_zero_interior(T* u, int n)
{
    zero_interior_block<T>(u, n, blockIdx);
}

inline dim3 grid_of(int n) { return dim3((n + BX - 1) / BX, (n + BY - 1) / BY, n); }

}  // namespace xfer
}  // namespace ma
