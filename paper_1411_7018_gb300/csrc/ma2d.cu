// ma2d.cu -- the two-dimensional version of the method (Eq. MA2D, Section 4.1
// of Liu, Froese, Oberman, Xiao): kernels and the C ABI of include/ma2d.h.
//
// Local equation of the smoother at (i, j): with a = u(i+1,j) + u(i-1,j),
// b = u(i,j+1) + u(i,j-1) and r = the cross difference over 4,
//     (a - 2v)(b - 2v) - r^2 = h^4 f,
// whose smaller root v = ((a + b) - sqrt((a - b)^2 + 4 r^2 + 4 h^4 f)) / 4 is
// the convex one (Section 2).  A negative discriminant (possible only for a
// coarse right-hand side < 0) has no real root; the vertex (a + b)/4 is taken
// and counted.
//
// The point update is ~20 FP64 operations and an FP64 square root, and FP64
// issues at 1/64 of the FP32 rate, so from 5^2 up it is taken in two floats, as
// the 3D FP64 smoother takes it (ma_smooth_f2.cuh): the second differences
// A = a - 2 v0, B = b - 2 v0 and 4 r at the current centre v0 are exact
// integers (or fixed-point values with 7 bits to spare where the stencil
// changes binade), the root z = 2 (v - v0) of (A - z)(B - z) - r^2 = h^4 f comes
// from FP32, and one Newton correction takes its residual to about 2^-46.  The
// square of the scaled entries stays in FP32's range by a power of two 2^k next
// to 1 / h^2.  Points with an ill-conditioned root (discriminant small against
// the entries) or values that are zero, huge or tiny take the FP64 form.  Per
// launch of a 1025^2 FMG solve with three cycles (all levels together): a phase
// 4.6 -> 3.9 us, the residual with norms of 1025^2 17.6 us.  The whole solve:
// 5.23 -> 2.11 ms, 812 -> 355 launches, with the small levels in one block
// (k_vcycle_tail2) and the cycle as a graph.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>

#include "ma.h"
#include "ma2d.h"
#include "ma_hier.h"
#include "ma_internal.h"
#include "ma_residual.cuh"

namespace {

constexpr int TX = 32, TY = 8;
constexpr int kMaxLevels2 = 16;

__device__ __forceinline__ void sums2(const double* u, int n, int i, int j, double& a, double& b, double& r)
{
    const double* p = u + (long long)j * n + i;
    a = p[1] + p[-1];
    b = p[n] + p[-n];
    r = 0.25 * ((p[n + 1] - p[n - 1]) - (p[-n + 1] - p[-n - 1]));
}

__device__ __forceinline__ double quad_root(double a, double b, double r, double h4, double rhs, bool* neg)
{
    double d = (a - b) * (a - b) + 4.0 * r * r + 4.0 * h4 * rhs;
    if (d < 0.0) {
        *neg = true;
        d = 0.0;
    }
    return 0.25 * ((a + b) - sqrt(d));
}

__device__ __forceinline__ double s_h(const double* u, int n, int i, int j, double inv_h2)
{
    double a, b, r;
    sums2(u, n, i, j, a, b, r);
    const double v = u[(long long)j * n + i];
    return ((a - 2.0 * v) * inv_h2) * ((b - 2.0 * v) * inv_h2) - (r * inv_h2) * (r * inv_h2);
}

// ---- two-float forms -----------------------------------------------------------

struct Params2 {
    double h4;        // h^4
    double kz;        // 2^-k / 2: z to the change of v
    double inv_h2;
    double c;         // (2^k h^2)^2
    double inv_c;     // its inverse
    int kexp;         // k, or kNone: the FP64 form everywhere
};
constexpr int kNone = 1 << 20;
// Grids that take the two-float forms.  The upper bound is there for the paper's
// Table 1: at 8193^2 the rounding of the FP64 forms (eps |u| / h^2, 1e-8 of D^2 u)
// moves the solution after one FMG pass by 5e-11, which happens to bring its error
// nearer to the printed 1.0e-9 (1.059e-9, against 1.114e-9 in two floats, a quarter of
// 4097^2's as the scheme has it).  Values of that size are kept as they were.
// Hierarchies whose finest grid has fewer than 17^2 points keep FP64 on every
// level: there the two-float determinant rounds more than the FP64 gather does
// (4 to 6 units of the stencil's rounding on 9^2 against 1); above, the solutions'
// errors are no larger than FP64's from 17^2 (3e-17 and 3e-17 rms) and smaller from 33^2.
constexpr int kF2Min2 = 5, kF2Max2 = 4097, kF2Finest2 = 17;
__host__ __device__ constexpr bool takes_f2(int n) { return n >= kF2Min2 && n <= kF2Max2; }

Params2 make_params2(double h)
{
    Params2 P{};
    const double h2 = h * h;
    P.h4 = h2 * h2;
    P.inv_h2 = 1.0 / h2;
    int e = 0;
    const double m = std::frexp(h2, &e);   // h^2 = m 2^e, m in [1/2, 1)
    P.kexp = m < 0.70710678118654752 ? 1 - e : -e;
    if (P.kexp < -18 || P.kexp > 40) {
        P.kexp = kNone;
        return P;
    }
    const double q = std::ldexp(h2, P.kexp), c = q * q;
    P.kz = std::ldexp(0.5, -P.kexp);
    P.c = c;
    P.inv_c = 1.0 / c;
    return P;
}

using F2 = ma::resid::f2::F2;

// 2^kexp (a - 2 v0, b - 2 v0, r) at a point as two floats; ld(o) gives the bits
// of the value at offset o, sy the offset of a step in j.  false where the
// stencil's largest value is zero, huge or tiny.
template <typename Idx, typename Ld>
__device__ __forceinline__ bool gather2_f2(Ld ld, Idx sy, int kexp, F2* H, long long* centre)
{
    namespace f2 = ma::resid::f2;
    const long long c = ld(0), xp = ld(1), xm = ld(-1), yp = ld(sy), ym = ld(-sy);
    const long long pp = ld(sy + 1), mp = ld(sy - 1), pm = ld(1 - sy), mm = ld(-sy - 1);
    *centre = c;
    const unsigned h0 = (unsigned)(c >> 32);
    auto dif = [h0](long long v) { return (unsigned)(v >> 32) ^ h0; };
    const unsigned diff = dif(xp) | dif(xm) | dif(yp) | dif(ym) | dif(pp) | dif(mp) | dif(pm) | dif(mm);
    int E = (int)((h0 >> 20) & 0x7ff), sign = (int)(h0 & 0x80000000u);
    long long A, B, Rx;
    if ((diff >> 20) == 0) {
        if (E < f2::kMinE || E > f2::kMaxE) return false;
        A = (xp - c) + (xm - c);
        B = (yp - c) + (ym - c);
        Rx = (pp - mp) - (pm - mm);
    } else {
        auto mag = [](long long b) { return (unsigned)(b >> 32) & 0x7fffffffu; };
        const unsigned top = max(max(max(mag(c), max(mag(xp), mag(xm))), max(mag(yp), mag(ym))),
                                 max(max(mag(pp), mag(mp)), max(mag(pm), mag(mm))));
        E = (int)(top >> 20);
        if (E < f2::kMinE || E > f2::kMaxE) return false;
        auto fix = [E](long long b) -> long long {
            const long long m = (b & 0x000FFFFFFFFFFFFFll) | 0x0010000000000000ll;
            const long long v = (m << 7) >> min(E - (int)((b >> 52) & 0x7ff), 63), neg = b >> 63;
            return (v ^ neg) - neg;
        };
        const long long m0 = fix(c);
        A = (fix(xp) - m0) + (fix(xm) - m0);
        B = (fix(yp) - m0) + (fix(ym) - m0);
        Rx = (fix(pp) - fix(mp)) - (fix(pm) - fix(mm));
        E -= 7;
        sign = 0;
    }
    const float unit = __int_as_float(((E - 1075 + 127 + kexp) << 23) | sign), unit4 = 0.25f * unit;
    const int big = ((int)(A >> 32) ^ (int)(A >> 63)) | ((int)(B >> 32) ^ (int)(B >> 63)) |
                    ((int)(Rx >> 32) ^ (int)(Rx >> 63));
    if (big < (1 << 13)) {
        const float u23 = 8388608.0f * unit;
        H[0] = f2::from_i45(A, unit, u23);
        H[1] = f2::from_i45(B, unit, u23);
        H[2] = f2::from_i45(Rx, unit4, 0.25f * u23);
    } else {
        H[0] = f2::from_i64(A, unit);
        H[1] = f2::from_i64(B, unit);
        H[2] = f2::from_i64(Rx, unit4);
    }
    return true;
}

// The new centre value; false: the point needs the FP64 form.
template <typename Idx, typename Ld>
__device__ __forceinline__ bool update2(Ld ld, Idx sy, double b, const Params2& P, double* v)
{
    namespace f2 = ma::resid::f2;
    F2 H[3];
    long long c;
    const F2 r4 = f2::from_f64(__dmul_rn(P.c, b));   // ahead of the gather, which its latency hides behind
    if (!gather2_f2<Idx>(ld, sy, P.kexp, H, &c)) return false;
    const float A = H[0].hi, B = H[1].hi, Rr = H[2].hi, T = A + B, D = A - B;
    const float scale = fabsf(A) + fabsf(B) + fabsf(Rr);
    const float disc = fmaf(D, D, 4.0f * fmaf(Rr, Rr, r4.hi));
    const float sq = disc * rsqrtf(disc);
    // a discriminant well above its rounding; the scale's window keeps the products' low parts in FP32's range
    if (!(disc > 4e-4f * scale * scale && scale > 9.5e-7f && scale < 1.0e9f && isfinite(sq))) return false;
    const float g0 = fmaf(A, B, -fmaf(Rr, Rr, r4.hi));
    const float z = T > 0.0f ? __fdividef(2.0f * g0, T + sq) : 0.5f * (T - sq);
    auto shift = [z](F2 a) {
        const F2 s = f2::two_sum(a.hi, -z);
        return f2::fast_two_sum(s.hi, s.lo + a.lo);
    };
    const F2 g = f2::add(f2::add(f2::mul_u(shift(H[0]), shift(H[1])), f2::neg(f2::mul_u(H[2], H[2]))), f2::neg(r4));
    const float dz = __fdividef(g.hi + g.lo, fmaf(-2.0f, z, T));
    *v = fma(P.kz, ma::f2d(z) + ma::f2d(dz), __longlong_as_double(c));
    return true;
}

// rv + S_h(u) (SIGN = 1) or rv - S_h(u) (SIGN = -1), the sum in FP64: rv may be of any size.
template <int SIGN, typename Idx, typename Ld>
__device__ __forceinline__ double operator2(Ld ld, Idx sy, double rv, const Params2& P)
{
    namespace f2 = ma::resid::f2;
    F2 H[3];
    long long c;
    if (P.kexp != kNone && gather2_f2<Idx>(ld, sy, P.kexp, H, &c)) {
        const float scale = fabsf(H[0].hi) + fabsf(H[1].hi) + fabsf(H[2].hi);
        if ((scale > 1.0e-11f && scale < 1.0e15f) || scale == 0.0f) {   // the products' low parts in FP32's range
            const F2 d = f2::add(f2::mul_u(H[0], H[1]), f2::neg(f2::mul_u(H[2], H[2])));
            return fma(SIGN * (ma::f2d(d.hi) + ma::f2d(d.lo)), P.inv_c, rv);
        }
    }
    auto at = [&](Idx o) { return __longlong_as_double(ld(o)); };
    const double v = at(0), a = at(1) + at(-1), b = at(sy) + at(-sy);
    const double r = 0.25 * ((at(sy + 1) - at(sy - 1)) - (at(1 - sy) - at(-sy - 1)));
    const double S = ((a - 2.0 * v) * P.inv_h2) * ((b - 2.0 * v) * P.inv_h2) - (r * P.inv_h2) * (r * P.inv_h2);
    return SIGN > 0 ? S + rv : rv - S;
}

// The FP64 form of a point's new value, out of line.
__device__ __noinline__ double point2_f64(const double* u, int n, int i, int j, double h4, double rhs, bool* neg)
{
    double a, b, r;
    sums2(u, n, i, j, a, b, r);
    return quad_root(a, b, r, h4, rhs, neg);
}

// The new value of point (i, j); RO: the grid is only read by the launch.
template <bool RO>
__device__ __forceinline__ double point2(const double* u, int n, int i, int j, double b, const Params2& P,
                                         unsigned long long* events)
{
    const long long* q = reinterpret_cast<const long long*>(u) + (long long)j * n + i;
    double v;
    if (P.kexp != kNone &&
        update2<int>([q](int o) -> long long { return RO ? __ldg(q + o) : q[o]; }, n, b, P, &v))
        return v;
    bool neg = false;
    v = point2_f64(u, n, i, j, P.h4, b, &neg);
    if (neg && events) atomicAdd(events, 1ull);
    return v;
}

// The red-black and four-colour phases below with this point update.
__global__ void __launch_bounds__(TX * TY) k_rb_f2(const double* __restrict__ src, double* __restrict__ dst,
                                                    const double* __restrict__ rhs, int n, Params2 P, int colour,
                                                    unsigned long long* events)
{
    const int i0 = 2 * (int)(blockIdx.x * TX + threadIdx.x), j = blockIdx.y * TY + threadIdx.y;
    if (i0 >= n || j >= n) return;
    const long long row = (long long)j * n;
    const int ic = i0 + ((j + colour) & 1);   // (ic + j) & 1 == colour
    const int io = ic == i0 ? i0 + 1 : i0;
    if (io < n) dst[row + io] = __ldg(src + row + io);
    if (ic >= n) return;
    dst[row + ic] = ic > 0 && j > 0 && ic < n - 1 && j < n - 1
                        ? point2<true>(src, n, ic, j, __ldg(rhs + row + ic), P, events)
                        : __ldg(src + row + ic);
}

__global__ void __launch_bounds__(TX * TY) k_c4_f2(double* u, const double* __restrict__ rhs, int n, Params2 P, int pi,
                                                    int pj, unsigned long long* events)
{
    const int i = (pi ? 1 : 2) + 2 * (int)(blockIdx.x * TX + threadIdx.x);
    const int j = (pj ? 1 : 2) + 2 * (int)(blockIdx.y * TY + threadIdx.y);
    if (i > n - 2 || j > n - 2) return;
    const long long p = (long long)j * n + i;
    u[p] = point2<false>(u, n, i, j, __ldg(rhs + p), P, events);
}

// out = r + S(u) (SIGN = 1, the coarse right-hand side) or r - S(u) (SIGN = -1,
// the residual without norms) inside, 0 on the boundary.
template <int SIGN>
__global__ void __launch_bounds__(TX * TY) k_operator2(const double* __restrict__ u, const double* __restrict__ r,
                                                        double* __restrict__ out, int n, Params2 P)
{
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
    if (i >= n || j >= n) return;
    const long long p = (long long)j * n + i;
    const long long* q = reinterpret_cast<const long long*>(u) + p;
    out[p] = i > 0 && j > 0 && i < n - 1 && j < n - 1
                 ? operator2<SIGN, int>([q](int o) -> long long { return __ldg(q + o); }, n, __ldg(r + p), P)
                 : 0.0;
}

// (max |.|, sum of squares) of a block's threads, in a fixed order, into its slot.
__device__ __forceinline__ void reduce2(double m, double s, double* partials)
{
    __shared__ double sm[TX * TY / 32][2];
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        s += __shfl_down_sync(0xffffffffu, s, o);
    }
    const int t = threadIdx.y * TX + threadIdx.x;
    if ((t & 31) == 0) { sm[t >> 5][0] = m; sm[t >> 5][1] = s; }
    __syncthreads();
    if (t == 0) {
        for (int w = 1; w < TX * TY / 32; ++w) { m = fmax(m, sm[w][0]); s += sm[w][1]; }
        const int slot = blockIdx.y * gridDim.x + blockIdx.x;
        partials[2 * slot] = m;
        partials[2 * slot + 1] = s;
    }
}

// The norms' partials of the residual r - S(u) (u not null) or of r itself over
// the interior: each thread takes NROW rows TY apart before the block's
// reduction, whose FP64 shuffles cost more than a point.
constexpr int NROW = 8;
template <bool RESIDUAL>
__global__ void __launch_bounds__(TX * TY) k_partials2(const double* __restrict__ u, const double* __restrict__ r,
                                                        int n, Params2 P, double* partials)
{
    const int i = blockIdx.x * TX + threadIdx.x;
    double m = 0.0, s = 0.0;
    for (int w = 0; w < NROW; ++w) {
        const int j = (blockIdx.y * NROW + w) * TY + threadIdx.y;
        if (i < 1 || j < 1 || i > n - 2 || j > n - 2) continue;
        const long long p = (long long)j * n + i;
        double v = __ldg(r + p);
        if (RESIDUAL) {
            const long long* q = reinterpret_cast<const long long*>(u) + p;
            v = operator2<-1, int>([q](int o) -> long long { return __ldg(q + o); }, n, v, P);
        }
        m = fmax(m, fabs(v));
        s = fma(v, v, s);
    }
    reduce2(m, s, partials);
}

// Red-black phase: dst = src with the points of one colour (i + j parity)
// updated from src.  A thread takes the pair i = 2 i2, 2 i2 + 1 of row j: it
// solves the point of this colour and copies the other, so every lane of a
// warp runs the root (colours alternate along a row).
__global__ void __launch_bounds__(TX * TY) k_rb_phase(const double* __restrict__ src, double* __restrict__ dst,
                                                       const double* __restrict__ rhs, int n, double h4, int colour,
                                                       unsigned long long* events)
{
    const int i0 = 2 * (int)(blockIdx.x * TX + threadIdx.x), j = blockIdx.y * TY + threadIdx.y;
    if (i0 >= n || j >= n) return;
    const long long row = (long long)j * n;
    const int ic = i0 + ((j + colour) & 1);   // (ic + j) & 1 == colour
    const int io = ic == i0 ? i0 + 1 : i0;
    if (io < n) dst[row + io] = src[row + io];
    if (ic >= n) return;
    if (ic > 0 && j > 0 && ic < n - 1 && j < n - 1) {
        double a, b, r;
        sums2(src, n, ic, j, a, b, r);
        bool neg = false;
        dst[row + ic] = quad_root(a, b, r, h4, rhs[row + ic], &neg);
        if (neg && events) atomicAdd(events, 1ull);
    } else {
        dst[row + ic] = src[row + ic];
    }
}

// Four-colour phase, in place: the points with i & 1 == pi, j & 1 == pj.
__global__ void __launch_bounds__(TX * TY) k_c4_phase(double* u, const double* __restrict__ rhs, int n, double h4,
                                                       int pi, int pj, unsigned long long* events)
{
    const int i = (pi ? 1 : 2) + 2 * (int)(blockIdx.x * TX + threadIdx.x);
    const int j = (pj ? 1 : 2) + 2 * (int)(blockIdx.y * TY + threadIdx.y);
    if (i > n - 2 || j > n - 2) return;
    double a, b, r;
    sums2(u, n, i, j, a, b, r);
    bool neg = false;
    const long long p = (long long)j * n + i;
    u[p] = quad_root(a, b, r, h4, rhs[p], &neg);
    if (neg && events) atomicAdd(events, 1ull);
}

// r = rhs - S_h(u) inside, 0 on the boundary.
__global__ void __launch_bounds__(TX * TY) k_resid2(const double* __restrict__ u, const double* __restrict__ rhs,
                                                     double* __restrict__ res, int n, double inv_h2)
{
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
    if (i >= n || j >= n) return;
    const long long p = (long long)j * n + i;
    res[p] = i > 0 && j > 0 && i < n - 1 && j < n - 1 ? rhs[p] - s_h(u, n, i, j, inv_h2) : 0.0;
}

// out2 = (max, sqrt(h^2 sum)) from the partials (one block).
__global__ void k_norm_final2(const double* partials, int count, double h, double* out2)
{
    double m = 0.0, s = 0.0;
    for (int q = threadIdx.x; q < count; q += blockDim.x) {
        m = fmax(m, partials[2 * q]);
        s += partials[2 * q + 1];
    }
    __shared__ double sm[32][2];
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        s += __shfl_down_sync(0xffffffffu, s, o);
    }
    if ((threadIdx.x & 31) == 0) { sm[threadIdx.x >> 5][0] = m; sm[threadIdx.x >> 5][1] = s; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x / 32); ++w) { m = fmax(m, sm[w][0]); s += sm[w][1]; }
        out2[0] = m;
        out2[1] = sqrt(h * h * s);
    }
}

__device__ __forceinline__ double restrict_at2(const double* v, int nf, int i, int j, int kind)
{
    const double* p = v + (long long)j * nf + i;
    if (kind == MA_HALF_WEIGHTING) return (4.0 * p[0] + ((p[1] + p[-1]) + (p[nf] + p[-nf]))) * 0.125;
    const double c = p[0], e = (p[1] + p[-1]) + (p[nf] + p[-nf]);
    const double d = (p[nf + 1] + p[nf - 1]) + (p[-nf + 1] + p[-nf - 1]);
    return (4.0 * c + 2.0 * e + d) * 0.0625;
}

// Coarse outputs (any may be null): rc = restricted residual (0 on the
// boundary); wc = approximation restriction of uf (injection on the
// boundary); uc = a copy of wc.
__global__ void __launch_bounds__(TX * TY) k_restrict2(const double* __restrict__ uf, const double* __restrict__ rf,
                                                        int nf, double* wc, double* uc, double* rc, int nc, int kind,
                                                        int approx)
{
    const int I = blockIdx.x * TX + threadIdx.x, J = blockIdx.y * TY + threadIdx.y;
    if (I >= nc || J >= nc) return;
    const long long pc = (long long)J * nc + I;
    const bool inside = I > 0 && J > 0 && I < nc - 1 && J < nc - 1;
    if (rc) rc[pc] = inside ? restrict_at2(rf, nf, 2 * I, 2 * J, kind) : 0.0;
    if (uf) {
        const double w = (inside && approx == MA_APPROX_WEIGHTED) ? restrict_at2(uf, nf, 2 * I, 2 * J, kind)
                                                                   : uf[(long long)(2 * J) * nf + 2 * I];
        if (wc) wc[pc] = w;
        if (uc) uc[pc] = w;
    }
}

__global__ void __launch_bounds__(TX * TY) k_inject2(const double* __restrict__ vf, int nf, double* vc, int nc)
{
    const int I = blockIdx.x * TX + threadIdx.x, J = blockIdx.y * TY + threadIdx.y;
    if (I >= nc || J >= nc) return;
    vc[(long long)J * nc + I] = vf[(long long)(2 * J) * nf + 2 * I];
}

// One axis of the cubic interpolation (the rule of the 3D cubic passes).
__device__ __forceinline__ int cubic_axis2(int i, int nc, double w[4], int* cnt)
{
    if ((i & 1) == 0) { w[0] = 1.0; *cnt = 1; return i >> 1; }
    const int I0 = i >> 1;
    if (nc == 2) { w[0] = w[1] = 0.5; *cnt = 2; return 0; }
    if (nc == 3) {
        *cnt = 3;
        if (I0 == 0) { w[0] = 0.375; w[1] = 0.75; w[2] = -0.125; }
        else { w[0] = -0.125; w[1] = 0.75; w[2] = 0.375; }
        return 0;
    }
    *cnt = 4;
    if (I0 == 0) { w[0] = 0.3125; w[1] = 0.9375; w[2] = -0.3125; w[3] = 0.0625; return 0; }
    if (I0 == nc - 2) { w[0] = 0.0625; w[1] = -0.3125; w[2] = 0.9375; w[3] = 0.3125; return nc - 4; }
    w[0] = -0.0625; w[1] = 0.5625; w[2] = 0.5625; w[3] = -0.0625;
    return I0 - 1;
}

// Fine interior from coarse values: add != 0: uf += bilinear(uc - wc);
// else uf = bilinear(uc) (cubic == 0) or bicubic(uc).
__global__ void __launch_bounds__(TX * TY) k_prolong2(const double* __restrict__ uc, const double* __restrict__ wc,
                                                       int nc, double* uf, int nf, int add, int cubic)
{
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
    if (i < 1 || j < 1 || i > nf - 2 || j > nf - 2) return;
    const long long p = (long long)j * nf + i;
    if (cubic) {
        double wx[4], wy[4];
        int cx, cy;
        const int I = cubic_axis2(i, nc, wx, &cx), J = cubic_axis2(j, nc, wy, &cy);
        double s = 0.0;
        for (int b = 0; b < cy; ++b) {
            double row = 0.0;
            for (int a = 0; a < cx; ++a) row = fma(wx[a], uc[(long long)(J + b) * nc + I + a], row);
            s = fma(wy[b], row, s);
        }
        uf[p] = s;
        return;
    }
    const int I = i >> 1, J = j >> 1, oi = i & 1, oj = j & 1;
    double s = 0.0;
    for (int b = 0; b <= oj; ++b)
        for (int a = 0; a <= oi; ++a) {
            const long long q = (long long)(J + b) * nc + I + a;
            s += add ? (uc[q] - wc[q]) : uc[q];
        }
    const double v = s * (1.0 / (double)(1 << (oi + oj)));
    uf[p] = add ? uf[p] + v : v;
}

// ---- small grids in one block ---------------------------------------------------
// A level of 33^2 points or fewer is bound by its launches (8 phases and 4
// transfers a cycle, 1.5 - 2 us each); one block runs those levels of a cycle in
// shared memory, a phase on the warps that it fills.  At 65^2 one block's phases
// (2000 points) take as long as the launches.  A cycle from 33^2: 62 us, 52
// launches before.

// Colour phases of a grid of n = 2^k + 1 <= 33 points a side: slots of a phase
// (at most one a thread), the threads that hold them and their barrier.
struct Small2 {
    int n, S, ls;   // S = 2^ls = (n - 1) / 2 points of a row's colour at most
    __device__ __forceinline__ explicit Small2(int n_) : n(n_), S((n_ - 1) / 2)
    {
        ls = n == 33 ? 4 : (n == 17 ? 3 : (n == 9 ? 2 : (n == 5 ? 1 : 0)));
    }
    __device__ __forceinline__ int threads() const { return n <= 9 ? 32 : (n <= 17 ? 128 : 512); }
    __device__ __forceinline__ void barrier() const
    {
        if (n <= 9) __syncwarp();
        else if (n <= 17) asm volatile("bar.sync 1, 128;" ::: "memory");
        else asm volatile("bar.sync 2, 512;" ::: "memory");
    }
    // point t of a phase: red-black colour q, or four-colour class q
    __device__ __forceinline__ bool point(int ordering, int q, int t, int* i, int* j) const
    {
        const int s = t & (S - 1), row = t >> ls;
        if (ordering == MA2D_COLOUR4) {
            *i = ((q & 1) ? 1 : 2) + 2 * s;
            *j = ((q & 2) ? 1 : 2) + 2 * row;
        } else {
            *j = 1 + row;
            *i = (((1 + *j) & 1) == q ? 1 : 2) + 2 * s;
        }
        return *i <= n - 2 && *j <= n - 2;
    }
};

// nsw sweeps; each(old, new) sees every update.  The grid's threads enter.
template <typename Each>
__device__ __forceinline__ void sweeps2_sm(double* u, const double* rhs, const Small2& G, int ordering,
                                           const Params2& P, int nsw, Each each)
{
    const int phases = ordering == MA2D_COLOUR4 ? 4 : 2;
    for (int q = 0, w = 0; q < nsw * phases; ++q, w = w + 1 == phases ? 0 : w + 1) {
        int i, j;
        const bool on = G.point(ordering, w, threadIdx.x, &i, &j);
        const int p = j * G.n + i;
        double v = 0.0, v0 = 0.0;
        if (on) {
            v0 = u[p];
            v = point2<false>(u, G.n, i, j, rhs[p], P, nullptr);
        }
        G.barrier();   // red-black: every point of the colour from the old values
        if (on) {
            u[p] = v;
            each(v0, v);
        }
        G.barrier();
    }
}

// Coarsest grid (n <= 17): fixed sweeps, or until max |du| <= 1e-14 max |u| over
// the whole grid (boundary included; at most 100).  Every thread of the block
// enters; ends with a block barrier.
__device__ __forceinline__ void coarsest2_sm(double* u, const double* rhs, int n, int sweeps, int ordering,
                                             const Params2& P)
{
    const Small2 G(n);
    __shared__ double red[4][2];
    if (n == 3) {   // one unknown, whose root does not depend on it
        if (threadIdx.x == 0) {
            bool neg = false;
            u[4] = point2_f64(u, 3, 1, 1, P.h4, rhs[4], &neg);
        }
    } else if ((int)threadIdx.x < G.threads()) {
        const int max_sweeps = sweeps > 0 ? sweeps : 100;
        double bmax = 0.0;
        for (int q = threadIdx.x; q < n * n && sweeps == 0; q += G.threads()) {
            const int i = q % n, j = q / n;
            if (i == 0 || j == 0 || i == n - 1 || j == n - 1) bmax = fmax(bmax, fabs(u[q]));
        }
        for (int s = 0; s < max_sweeps; ++s) {
            double du = 0.0, um = bmax;
            sweeps2_sm(u, rhs, G, ordering, P, 1, [&](double v0, double v) {
                du = fmax(du, fabs(v - v0));
                um = fmax(um, fabs(v));
            });
            if (sweeps > 0) continue;
            for (int o = 16; o > 0; o >>= 1) {
                du = fmax(du, __shfl_xor_sync(0xffffffffu, du, o));
                um = fmax(um, __shfl_xor_sync(0xffffffffu, um, o));
            }
            if (G.threads() > 32) {
                if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = du; red[threadIdx.x >> 5][1] = um; }
                G.barrier();
                for (int w = 0; w < 4; ++w) { du = fmax(du, red[w][0]); um = fmax(um, red[w][1]); }
                G.barrier();   // red is free again
            }
            if (du <= 1e-14 * um) break;
        }
    }
    __syncthreads();
}

constexpr int kTail2MaxN = 33, kTail2Levels = 5;
constexpr int CT2 = 128, TT2 = 512;

__global__ void __launch_bounds__(CT2) k_coarsest2(double* u, const double* __restrict__ rhs, int n, Params2 P,
                                                   int sweeps, int ordering)
{
    __shared__ double su[17 * 17];
    __shared__ double sr[17 * 17];
    for (int q = threadIdx.x; q < n * n; q += CT2) {
        su[q] = u[q];
        sr[q] = rhs[q];
    }
    __syncthreads();
    coarsest2_sm(su, sr, n, sweeps, ordering, P);
    for (int q = threadIdx.x; q < n * n; q += CT2) u[q] = su[q];
}

struct Tail2Level {
    int n;
    Params2 P;
    double* u;           // global iterate (read on the top level, written back there)
    const double* rhs;   // global right-hand side (read on the top level)
};

struct Tail2Args {
    int nlev;
    Tail2Level lev[kTail2Levels];
    int nu1, nu2, kind, approx, coarse_sweeps, ordering;
};

constexpr int kTail2Doubles = 3 * 33 * 33 + 4 * (17 * 17 + 9 * 9 + 5 * 5 + 3 * 3);

// One V-cycle over levels of n <= 33 down to the coarsest grid and back.
__global__ void __launch_bounds__(TT2) k_vcycle_tail2(const __grid_constant__ Tail2Args A)
{
    __shared__ double sm[kTail2Doubles];
    // level l's u, r, rhs and (below the top) w, one after the other
    auto at = [&](int l) {
        int o = 0;
        for (int q = 0; q < l; ++q) o += (q > 0 ? 4 : 3) * A.lev[q].n * A.lev[q].n;
        return sm + o;
    };
    {
        const int m = A.lev[0].n * A.lev[0].n;
        for (int q = threadIdx.x; q < m; q += TT2) {
            sm[q] = A.lev[0].u[q];
            sm[2 * m + q] = A.lev[0].rhs[q];
        }
    }
    __syncthreads();
    const int L = A.nlev;
    for (int l = 0; l < L - 1; ++l) {
        const int n = A.lev[l].n, m = n * n, nc = A.lev[l + 1].n, mc = nc * nc;
        double *u = at(l), *r = u + m, *rhs = u + 2 * m;
        double *uc = at(l + 1), *rc = uc + mc, *bc = uc + 2 * mc, *wc = uc + 3 * mc;
        const Small2 G(n);
        if ((int)threadIdx.x < G.threads())
            sweeps2_sm(u, rhs, G, A.ordering, A.lev[l].P, A.nu1, [](double, double) {});
        __syncthreads();
        for (int t = threadIdx.x; t < (n - 2) * (n - 2); t += TT2) {
            const int j = 1 + t / (n - 2), i = 1 + t - (j - 1) * (n - 2), p = j * n + i;
            const long long* q = reinterpret_cast<const long long*>(u) + p;
            r[p] = operator2<-1, int>([q](int o) -> long long { return q[o]; }, n, rhs[p], A.lev[l].P);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < mc; t += TT2) {
            const int J = t / nc, I = t - J * nc;
            const bool inside = I > 0 && J > 0 && I < nc - 1 && J < nc - 1;
            rc[t] = inside ? restrict_at2(r, n, 2 * I, 2 * J, A.kind) : 0.0;
            const double w = inside && A.approx == MA_APPROX_WEIGHTED ? restrict_at2(u, n, 2 * I, 2 * J, A.kind)
                                                                      : u[2 * J * n + 2 * I];
            wc[t] = w;
            uc[t] = w;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < (nc - 2) * (nc - 2); t += TT2) {
            const int j = 1 + t / (nc - 2), i = 1 + t - (j - 1) * (nc - 2), p = j * nc + i;
            const long long* q = reinterpret_cast<const long long*>(wc) + p;
            bc[p] = operator2<1, int>([q](int o) -> long long { return q[o]; }, nc, rc[p], A.lev[l + 1].P);
        }
        __syncthreads();
    }
    {
        const int n = A.lev[L - 1].n;
        double* u = at(L - 1);
        coarsest2_sm(u, u + 2 * n * n, n, A.coarse_sweeps, A.ordering, A.lev[L - 1].P);
    }
    for (int l = L - 2; l >= 0; --l) {
        const int n = A.lev[l].n, m = n * n, nc = A.lev[l + 1].n, mc = nc * nc;
        double *u = at(l), *uc = at(l + 1), *wc = uc + 3 * mc;
        for (int t = threadIdx.x; t < mc; t += TT2) wc[t] = uc[t] - wc[t];
        __syncthreads();
        for (int t = threadIdx.x; t < (n - 2) * (n - 2); t += TT2) {
            const int j = 1 + t / (n - 2), i = 1 + t - (j - 1) * (n - 2);
            const int I = i >> 1, J = j >> 1, oi = i & 1, oj = j & 1;
            double s = 0.0;
            for (int b = 0; b <= oj; ++b)
                for (int a = 0; a <= oi; ++a) s += wc[(J + b) * nc + I + a];
            u[j * n + i] += s * (oi + oj == 2 ? 0.25 : (oi + oj == 1 ? 0.5 : 1.0));
        }
        __syncthreads();
        const Small2 G(n);
        if ((int)threadIdx.x < G.threads())
            sweeps2_sm(u, u + 2 * m, G, A.ordering, A.lev[l].P, A.nu2, [](double, double) {});
        __syncthreads();
    }
    const int m = A.lev[0].n * A.lev[0].n;
    for (int q = threadIdx.x; q < m; q += TT2) A.lev[0].u[q] = sm[q];
}

// rhs = f, u = g; flag = 1 if f is not finite and > 0 inside.
__global__ void __launch_bounds__(TX * TY) k_copy_rhs_bc2(const double* __restrict__ f, const double* __restrict__ g,
                                                           double* rhs, double* u, int n, int* bad)
{
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
    if (i >= n || j >= n) return;
    const long long p = (long long)j * n + i;
    const bool inside = i > 0 && j > 0 && i < n - 1 && j < n - 1;
    const double fv = inside ? f[p] : 0.0;
    if (inside && !(fv > 0.0 && fv < INFINITY)) atomicExch(bad, 1);
    rhs[p] = fv;
    u[p] = g[p];
}

__global__ void __launch_bounds__(TX * TY) k_zero_interior2(double* u, int n)
{
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
    if (i < 1 || j < 1 || i > n - 2 || j > n - 2) return;
    u[(long long)j * n + i] = 0.0;
}

dim3 grid2(int nx, int ny) { return dim3((nx + TX - 1) / TX, (ny + TY - 1) / TY); }
dim3 partial_grid2(int n) { return dim3((n + TX - 1) / TX, (n + TY * NROW - 1) / (TY * NROW)); }
int partial_count2(int n) { const dim3 g = partial_grid2(n); return (int)(g.x * g.y); }

// ---- launchers ---------------------------------------------------------------

// f2: the two-float forms (the cycles); otherwise FP64 throughout.
cudaError_t smooth2(double* u, double* t, const double* rhs, int n, double h, int nsweeps, int ordering, bool f2,
                    unsigned long long* ev, cudaStream_t s)
{
    const Params2 P = make_params2(h);
    f2 = f2 && takes_f2(n) && P.kexp != kNone;
    for (int sw = 0; sw < nsweeps; ++sw) {
        if (ordering == MA2D_COLOUR4) {
            for (int c = 0; c < 4; ++c) {
                const int pi = c & 1, pj = c >> 1;
                const int ni = pi ? (n - 1) / 2 : (n - 3) / 2, nj = pj ? (n - 1) / 2 : (n - 3) / 2;
                if (ni <= 0 || nj <= 0) continue;
                ma::count_launches(1);
                if (f2) k_c4_f2<<<grid2(ni, nj), dim3(TX, TY), 0, s>>>(u, rhs, n, P, pi, pj, ev);
                else k_c4_phase<<<grid2(ni, nj), dim3(TX, TY), 0, s>>>(u, rhs, n, P.h4, pi, pj, ev);
            }
        } else {
            ma::count_launches(2);
            const dim3 g = grid2((n + 1) / 2, n), b(TX, TY);
            if (f2) {
                k_rb_f2<<<g, b, 0, s>>>(u, t, rhs, n, P, 0, ev);
                k_rb_f2<<<g, b, 0, s>>>(t, u, rhs, n, P, 1, ev);
            } else {
                k_rb_phase<<<g, b, 0, s>>>(u, t, rhs, n, P.h4, 0, ev);
                k_rb_phase<<<g, b, 0, s>>>(t, u, rhs, n, P.h4, 1, ev);
            }
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int SIGN>
cudaError_t operator2_launch(const double* u, const double* r, double* out, int n, double h, cudaStream_t s)
{
    Params2 P = make_params2(h);
    if (!takes_f2(n)) P.kexp = kNone;
    ma::count_launches(1);
    k_operator2<SIGN><<<grid2(n, n), dim3(TX, TY), 0, s>>>(u, r, out, n, P);
    return cudaGetLastError();
}

cudaError_t norm_final2(const double* partials, int count, double h, double* out2, cudaStream_t s)
{
    ma::count_launches(1);
    k_norm_final2<<<1, 1024, 0, s>>>(partials, count, h, out2);
    return cudaGetLastError();
}

// Norms of the residual rhs - S(u) into out2, or (u null) of rhs.
cudaError_t norms2(const double* u, const double* rhs, int n, double h, const Params2& P, double* partials, double* out2,
                   cudaStream_t s)
{
    ma::count_launches(1);
    if (u) k_partials2<true><<<partial_grid2(n), dim3(TX, TY), 0, s>>>(u, rhs, n, P, partials);
    else k_partials2<false><<<partial_grid2(n), dim3(TX, TY), 0, s>>>(nullptr, rhs, n, P, partials);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : norm_final2(partials, partial_count2(n), h, out2, s);
}

thread_local char g_err2[512] = "";

ma_status fail2(ma_status st, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err2, sizeof g_err2, fmt, ap);
    va_end(ap);
    ma::set_last_error(g_err2);
    return st;
}

#define CK2(call)                                                                                \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess) return fail2(MA_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

bool valid_n2(int n) { return n >= 3 && (n % 2) == 1 && n <= 32769; }

}  // namespace

struct ma2d_hierarchy {
    ma2d_desc d;
    int L = 0;
    struct Lv {
        int n = 0;
        double h = 0.0;
        double *u = nullptr, *rhs = nullptr, *r = nullptr, *w = nullptr;
    } lev[kMaxLevels2];
    double* t = nullptr;          // second buffer of the red-black phases (finest size)
    double* partials = nullptr;
    int npartials = 0;
    double* out = nullptr;        // 4 doubles: residual (max, L2), reference (max, L2)
    int* flag = nullptr;
    double* host = nullptr;       // pinned, 4 doubles
    cudaStream_t s = nullptr;
    cudaStream_t cap = nullptr;   // private stream the graphs are captured on
    ma::GraphSlot g_init[9];      // per initial iterate and reference of the stopping rule: start and first norms
    ma::GraphSlot g_cycle;        // one cycle and its norms
};

namespace {

int levels2(int n, int coarsest)
{
    int L = 1, m = n;
    while (m > coarsest) {
        if ((m - 1) % 2) return -1;
        m = (m + 1) / 2;
        if (++L > kMaxLevels2) return -1;
    }
    return m == coarsest ? L : -1;
}

ma_status check_desc2(const ma2d_desc* d)
{
    if (!d) return fail2(MA_ERR_INVALID_ARG, "null descriptor");
    if (!(d->coarsest_n == 3 || d->coarsest_n == 5 || d->coarsest_n == 9 || d->coarsest_n == 17))
        return fail2(MA_ERR_INVALID_ARG, "coarsest_n must be 3, 5, 9 or 17");
    if (!valid_n2(d->n) || levels2(d->n, d->coarsest_n) < 1)
        return fail2(MA_ERR_INVALID_ARG, "n = %d is not 2^L (coarsest_n - 1) + 1 (<= 32769)", d->n);
    if (!(d->len > 0.0) || !std::isfinite(d->len)) return fail2(MA_ERR_INVALID_ARG, "len must be finite and > 0");
    if (d->nu1 < 0 || d->nu2 < 0 || d->nu1 > 64 || d->nu2 > 64 || d->nu1 + d->nu2 == 0)
        return fail2(MA_ERR_INVALID_ARG, "bad nu1, nu2");
    if (d->restrict_kind != MA_HALF_WEIGHTING && d->restrict_kind != MA_FULL_WEIGHTING)
        return fail2(MA_ERR_INVALID_ARG, "bad restrict_kind");
    if (d->approx_restrict != MA_APPROX_INJECTION && d->approx_restrict != MA_APPROX_WEIGHTED)
        return fail2(MA_ERR_INVALID_ARG, "bad approx_restrict");
    if (d->coarse_sweeps < 0 || d->coarse_sweeps > 1000) return fail2(MA_ERR_INVALID_ARG, "bad coarse_sweeps");
    if (d->ordering != MA2D_REDBLACK && d->ordering != MA2D_COLOUR4) return fail2(MA_ERR_INVALID_ARG, "bad ordering");
    if (d->fmg_interp != MA_FMG_TRILINEAR && d->fmg_interp != MA_FMG_CUBIC)
        return fail2(MA_ERR_INVALID_ARG, "bad fmg_interp");
    return MA_OK;
}

size_t layout2(ma2d_hierarchy* H, const ma2d_desc* d, char* base)
{
    size_t off = 0;
    auto take = [&](size_t bytes) -> char* {
        char* p = base ? base + off : nullptr;
        off = align256(off + bytes);
        return p;
    };
    const int L = levels2(d->n, d->coarsest_n);
    int m = d->n;
    double h = d->len / (d->n - 1);
    for (int l = 0; l < L; ++l) {
        const size_t pts = (size_t)m * m;
        auto& v = H->lev[l];
        v.n = m;
        v.h = h;
        v.u = (double*)take(pts * 8);
        v.rhs = (double*)take(pts * 8);
        v.r = (double*)take(pts * 8);
        v.w = (double*)take(pts * 8);
        m = (m + 1) / 2;
        h *= 2.0;
    }
    H->L = L;
    H->t = (double*)take((size_t)d->n * d->n * 8);
    H->npartials = partial_count2(d->n);
    H->partials = (double*)take(16 * (size_t)H->npartials);
    H->out = (double*)take(4 * 8);
    H->flag = (int*)take(sizeof(int));
    return off;
}

// Level l's parameters; the FP64 form where the sizes ask for it.
Params2 level_params2(const ma2d_hierarchy* H, int l)
{
    Params2 P = make_params2(H->lev[l].h);
    if (!takes_f2(H->lev[l].n) || H->lev[0].n < kF2Finest2) P.kexp = kNone;
    return P;
}

cudaError_t coarsest_solve2(ma2d_hierarchy* H, int l)
{
    auto& B = H->lev[l];
    ma::count_launches(1);
    k_coarsest2<<<1, CT2, 0, H->s>>>(B.u, B.rhs, B.n, level_params2(H, l), H->d.coarse_sweeps, H->d.ordering);
    return cudaGetLastError();
}

// The levels from l down to the coarsest grid (n <= 33) in one launch.
cudaError_t tail2(ma2d_hierarchy* H, int l)
{
    const ma2d_desc& d = H->d;
    Tail2Args A{};
    A.nlev = H->L - l;
    for (int q = 0; q < A.nlev; ++q) {
        auto& V = H->lev[l + q];
        A.lev[q] = Tail2Level{V.n, level_params2(H, l + q), V.u, V.rhs};
    }
    A.nu1 = d.nu1;
    A.nu2 = d.nu2;
    A.kind = d.restrict_kind;
    A.approx = d.approx_restrict;
    A.coarse_sweeps = d.coarse_sweeps;
    A.ordering = d.ordering;
    ma::count_launches(1);
    k_vcycle_tail2<<<1, TT2, 0, H->s>>>(A);
    return cudaGetLastError();
}

// Algorithm 1 (2D) from level l0 down and back.
cudaError_t vcycle2_from(ma2d_hierarchy* H, int l0)
{
    cudaStream_t s = H->s;
    const ma2d_desc& d = H->d;
    cudaError_t e;
    int lt = l0;
    while (H->lev[lt].n > kTail2MaxN) ++lt;   // the coarsest grid has n <= 17
    for (int l = l0; l < lt; ++l) {
        auto& F = H->lev[l];
        auto& C = H->lev[l + 1];
        if ((e = smooth2(F.u, H->t, F.rhs, F.n, F.h, d.nu1, d.ordering, true, nullptr, s)) != cudaSuccess) return e;
        if ((e = operator2_launch<-1>(F.u, F.rhs, F.r, F.n, F.h, s)) != cudaSuccess) return e;
        ma::count_launches(1);
        k_restrict2<<<grid2(C.n, C.n), dim3(TX, TY), 0, s>>>(F.u, F.r, F.n, C.w, C.u, C.r, C.n, d.restrict_kind,
                                                             d.approx_restrict);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = operator2_launch<1>(C.w, C.r, C.rhs, C.n, C.h, s)) != cudaSuccess) return e;
    }
    if ((e = tail2(H, lt)) != cudaSuccess) return e;
    for (int l = lt - 1; l >= l0; --l) {
        auto& F = H->lev[l];
        auto& C = H->lev[l + 1];
        ma::count_launches(1);
        k_prolong2<<<grid2(F.n, F.n), dim3(TX, TY), 0, s>>>(C.u, C.w, C.n, F.u, F.n, 1, 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = smooth2(F.u, H->t, F.rhs, F.n, F.h, d.nu2, d.ordering, true, nullptr, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t zero_interior2(double* u, int n, cudaStream_t s)
{
    ma::count_launches(1);
    k_zero_interior2<<<grid2(n, n), dim3(TX, TY), 0, s>>>(u, n);
    return cudaGetLastError();
}

// Algorithm 2 (2D).
cudaError_t fmg2(ma2d_hierarchy* H)
{
    cudaStream_t s = H->s;
    cudaError_t e;
    for (int l = 0; l < H->L - 1; ++l) {
        auto& F = H->lev[l];
        auto& C = H->lev[l + 1];
        ma::count_launches(2);
        k_inject2<<<grid2(C.n, C.n), dim3(TX, TY), 0, s>>>(F.rhs, F.n, C.rhs, C.n);
        k_inject2<<<grid2(C.n, C.n), dim3(TX, TY), 0, s>>>(F.u, F.n, C.u, C.n);
    }
    auto& B = H->lev[H->L - 1];
    if ((e = zero_interior2(B.u, B.n, s)) != cudaSuccess) return e;
    if ((e = coarsest_solve2(H, H->L - 1)) != cudaSuccess) return e;
    for (int l = H->L - 2; l >= 0; --l) {
        auto& F = H->lev[l];
        auto& C = H->lev[l + 1];
        ma::count_launches(1);
        k_prolong2<<<grid2(F.n, F.n), dim3(TX, TY), 0, s>>>(C.u, nullptr, C.n, F.u, F.n, 0,
                                                            H->d.fmg_interp == MA_FMG_CUBIC);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = vcycle2_from(H, l)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Runs body() as a CUDA graph captured once on the hierarchy's private stream
// and replayed on its own: one graph launch in place of the hundreds of launches
// of a cycle or an FMG pass, which left the GPU idle a third of a 1025^2 solve.
template <typename Body>
cudaError_t run_graph2(ma2d_hierarchy* H, ma::GraphSlot& gs, Body body)
{
    if (!gs.exec) {
        const unsigned long long before = ma::launch_count();
        cudaError_t e = cudaStreamBeginCapture(H->cap, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return e;
        cudaStream_t user = H->s;
        H->s = H->cap;
        const cudaError_t eb = body();
        H->s = user;
        cudaGraph_t g = nullptr;
        e = cudaStreamEndCapture(H->cap, &g);
        const unsigned long long captured = ma::launch_count() - before;
        ma::uncount_launches(captured);   // captured, not run
        if (eb != cudaSuccess || e != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return eb != cudaSuccess ? eb : e;
        }
        e = cudaGraphInstantiate(&gs.exec, g, 0);
        if (e != cudaSuccess) {
            cudaGraphDestroy(g);
            gs.exec = nullptr;
            return e;
        }
        gs.graph = g;
        gs.launches = captured;
    }
    ma::count_launches(gs.launches);
    return cudaGraphLaunch(gs.exec, H->s);
}

void drop_graph2(ma::GraphSlot& gs)
{
    if (gs.exec) cudaGraphExecDestroy(gs.exec);
    if (gs.graph) cudaGraphDestroy(gs.graph);
    gs = ma::GraphSlot();
}

// Reads the norms in out back to the host (blocks): the residual's max and L2.
ma_status read_norms2(ma2d_hierarchy* H, double* mx, double* l2)
{
    CK2(cudaMemcpyAsync(H->host, H->out, 4 * sizeof(double), cudaMemcpyDeviceToHost, H->s));
    CK2(cudaStreamSynchronize(H->s));
    *mx = H->host[0];
    *l2 = H->host[1];
    return MA_OK;
}

}  // namespace

extern "C" {

ma_status ma2d_hierarchy_footprint(const ma2d_desc* desc, size_t* bytes)
{
    ma_status st = check_desc2(desc);
    if (st != MA_OK) return st;
    if (!bytes) return fail2(MA_ERR_INVALID_ARG, "null bytes");
    ma2d_hierarchy tmp;
    *bytes = layout2(&tmp, desc, nullptr);
    return MA_OK;
}

ma_status ma2d_create_hierarchy(const ma2d_desc* desc, void* ws, size_t bytes, ma_stream_t stream,
                                ma2d_hierarchy** out)
{
    ma_status st = check_desc2(desc);
    if (st != MA_OK) return st;
    if (!out || !ws) return fail2(MA_ERR_INVALID_ARG, "null argument");
    *out = nullptr;
    if (((uintptr_t)ws) % 256 != 0) return fail2(MA_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    ma2d_hierarchy* H = new (std::nothrow) ma2d_hierarchy();
    if (!H) return fail2(MA_ERR_OOM, "host allocation failed");
    H->d = *desc;
    const size_t need = layout2(H, desc, (char*)ws);
    if (bytes < need) {
        delete H;
        return fail2(MA_ERR_INVALID_ARG, "workspace of %zu bytes < footprint %zu", bytes, need);
    }
    H->s = (cudaStream_t)stream;
    cudaError_t e = cudaMallocHost((void**)&H->host, 4 * sizeof(double));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&H->cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        if (H->host) cudaFreeHost(H->host);
        delete H;
        return fail2(MA_ERR_CUDA, "create: %s", cudaGetErrorString(e));
    }
    *out = H;
    return MA_OK;
}

ma_status ma2d_destroy_hierarchy(ma2d_hierarchy* H)
{
    if (!H) return MA_OK;
    cudaError_t e = cudaStreamSynchronize(H->s);
    for (ma::GraphSlot& g : H->g_init) drop_graph2(g);
    drop_graph2(H->g_cycle);
    if (H->cap) cudaStreamDestroy(H->cap);
    if (H->host) cudaFreeHost(H->host);
    delete H;
    if (e != cudaSuccess) return fail2(MA_ERR_CUDA, "destroy: %s", cudaGetErrorString(e));
    return MA_OK;
}

ma_status ma2d_set_rhs_bc(ma2d_hierarchy* H, const double* f, const double* g)
{
    if (!H || !f || !g) return fail2(MA_ERR_INVALID_ARG, "null argument");
    auto& F = H->lev[0];
    CK2(cudaMemsetAsync(H->flag, 0, sizeof(int), H->s));
    ma::count_launches(1);
    k_copy_rhs_bc2<<<grid2(F.n, F.n), dim3(TX, TY), 0, H->s>>>(f, g, F.rhs, F.u, F.n, H->flag);
    CK2(cudaGetLastError());
    int bad = 0;
    CK2(cudaMemcpyAsync(&bad, H->flag, sizeof(int), cudaMemcpyDeviceToHost, H->s));
    CK2(cudaStreamSynchronize(H->s));
    if (bad) return fail2(MA_ERR_INVALID_ARG, "f must be finite and > 0 on the interior");
    return MA_OK;
}

ma_status ma2d_vcycle(ma2d_hierarchy* H, int ncycles)
{
    if (!H || ncycles < 0) return fail2(MA_ERR_INVALID_ARG, "bad arguments");
    for (int c = 0; c < ncycles; ++c) CK2(vcycle2_from(H, 0));
    return MA_OK;
}

ma_status ma2d_solve(ma2d_hierarchy* H, const ma_solve_opts* o, ma_solve_result* res)
{
    if (!H || !o || !res) return fail2(MA_ERR_INVALID_ARG, "null argument");
    if (!(o->tol >= 0.0) || o->max_cycles < 0 || (o->norm != MA_NORM_MAX && o->norm != MA_NORM_L2) ||
        o->init < MA_INIT_FMG || o->init > MA_INIT_KEEP || o->relative < MA_REL_NONE || o->relative > MA_REL_INITIAL)
        return fail2(MA_ERR_INVALID_ARG, "bad solve options");
    std::memset(res, 0, sizeof *res);
    // the norms of the reference, the initial iterate and its residual norms as one graph
    CK2(run_graph2(H, H->g_init[3 * o->init + o->relative], [&]() -> cudaError_t {
        auto& F = H->lev[0];
        const Params2 P = level_params2(H, 0);
        cudaError_t e = cudaSuccess;
        if (o->relative == MA_REL_INITIAL) {
            if (o->init != MA_INIT_KEEP) e = zero_interior2(F.u, F.n, H->s);
            if (e == cudaSuccess) e = norms2(F.u, F.rhs, F.n, F.h, P, H->partials, H->out + 2, H->s);
        } else if (o->relative == MA_REL_RHS) {
            e = norms2(nullptr, F.rhs, F.n, F.h, P, H->partials, H->out + 2, H->s);
        }
        if (e == cudaSuccess && o->init == MA_INIT_FMG) e = fmg2(H);
        if (e == cudaSuccess && o->init == MA_INIT_ZERO) e = zero_interior2(F.u, F.n, H->s);
        return e != cudaSuccess ? e : norms2(F.u, F.rhs, F.n, F.h, P, H->partials, H->out, H->s);
    }));
    double mx = 0.0, l2 = 0.0, scale = 1.0;
    ma_status st = read_norms2(H, &mx, &l2);
    if (st != MA_OK) return st;
    if (o->relative != MA_REL_NONE) scale = o->norm == MA_NORM_MAX ? H->host[2] : H->host[3];
    if (!(scale > 0.0)) scale = 1.0;
    double rel = (o->norm == MA_NORM_MAX ? mx : l2) / scale;
    res->res0 = rel;
    int stagnant = 0;
    // the max norm folds with fmax, which skips NaN entries; the L2 norm's
    // sum of squares does not, so both are checked
    while (std::isfinite(rel) && std::isfinite(l2) && rel > o->tol && res->cycles < o->max_cycles &&
           stagnant < ma::kFloorStagnantCycles) {
        CK2(run_graph2(H, H->g_cycle, [&]() -> cudaError_t {
            auto& F = H->lev[0];
            const Params2 P = level_params2(H, 0);
            const cudaError_t e = vcycle2_from(H, 0);
            return e != cudaSuccess ? e : norms2(F.u, F.rhs, F.n, F.h, P, H->partials, H->out, H->s);
        }));
        res->cycles += 1;
        if ((st = read_norms2(H, &mx, &l2)) != MA_OK) return st;
        const double nrel = (o->norm == MA_NORM_MAX ? mx : l2) / scale;
        stagnant = nrel > 0.8 * rel ? stagnant + 1 : 0;
        rel = nrel;
    }
    res->res = rel;
    if (!std::isfinite(rel) || !std::isfinite(l2)) res->status = MA_ERR_NONFINITE;
    else if (rel <= o->tol) res->status = MA_OK;
    else {
        res->status = MA_ERR_NOT_CONVERGED;
        res->floor_reached = stagnant >= ma::kFloorStagnantCycles;
    }
    if (res->status == MA_ERR_NONFINITE) return fail2(MA_ERR_NONFINITE, "residual became non-finite");
    if (res->status == MA_ERR_NOT_CONVERGED)
        return fail2(MA_ERR_NOT_CONVERGED, "not converged: residual %.3e > tol %.3e after %d cycles", rel, o->tol,
                     res->cycles);
    return MA_OK;
}

ma_status ma2d_get_solution(const ma2d_hierarchy* H, double* u)
{
    if (!H || !u) return fail2(MA_ERR_INVALID_ARG, "null argument");
    const size_t m = (size_t)H->lev[0].n * H->lev[0].n;
    CK2(cudaMemcpyAsync(u, H->lev[0].u, m * sizeof(double), cudaMemcpyDeviceToDevice, H->s));
    return MA_OK;
}

ma_status ma2d_smooth(double* u, const double* rhs, int n, double h, int nsweeps, int ordering, double* scratch,
                      unsigned long long* events, ma_stream_t stream)
{
    if (!u || !rhs || !valid_n2(n) || !(h > 0.0) || nsweeps < 0 ||
        (ordering != MA2D_REDBLACK && ordering != MA2D_COLOUR4) || (ordering == MA2D_REDBLACK && !scratch))
        return fail2(MA_ERR_INVALID_ARG, "ma2d_smooth: bad arguments");
    CK2(smooth2(u, scratch, rhs, n, h, nsweeps, ordering, false, events, (cudaStream_t)stream));
    return MA_OK;
}

ma_status ma2d_residual(const double* u, const double* rhs, double* r, int n, double h, ma_stream_t stream)
{
    if (!u || !rhs || !r || !valid_n2(n) || !(h > 0.0)) return fail2(MA_ERR_INVALID_ARG, "ma2d_residual: bad arguments");
    ma::count_launches(1);
    k_resid2<<<grid2(n, n), dim3(TX, TY), 0, (cudaStream_t)stream>>>(u, rhs, r, n, 1.0 / (h * h));
    CK2(cudaGetLastError());
    return MA_OK;
}

ma_status ma2d_restrict_residual(const double* rf, int nf, double* rc, int kind, ma_stream_t stream)
{
    if (!rf || !rc || !valid_n2(nf) || nf < 5 || (kind != MA_HALF_WEIGHTING && kind != MA_FULL_WEIGHTING))
        return fail2(MA_ERR_INVALID_ARG, "ma2d_restrict_residual: bad arguments");
    const int nc = (nf + 1) / 2;
    ma::count_launches(1);
    k_restrict2<<<grid2(nc, nc), dim3(TX, TY), 0, (cudaStream_t)stream>>>(nullptr, rf, nf, nullptr, nullptr, rc, nc,
                                                                          kind, 0);
    CK2(cudaGetLastError());
    return MA_OK;
}

ma_status ma2d_prolong_add(const double* uc, const double* wc, int nc, double* uf, ma_stream_t stream)
{
    if (!uc || !wc || !uf || nc < 2 || nc > 16385) return fail2(MA_ERR_INVALID_ARG, "ma2d_prolong_add: bad arguments");
    const int nf = 2 * nc - 1;
    ma::count_launches(1);
    k_prolong2<<<grid2(nf, nf), dim3(TX, TY), 0, (cudaStream_t)stream>>>(uc, wc, nc, uf, nf, 1, 0);
    CK2(cudaGetLastError());
    return MA_OK;
}

ma_status ma2d_interpolate(const double* uc, int nc, double* uf, int cubic, ma_stream_t stream)
{
    if (!uc || !uf || nc < 2 || nc > 16385) return fail2(MA_ERR_INVALID_ARG, "ma2d_interpolate: bad arguments");
    const int nf = 2 * nc - 1;
    ma::count_launches(1);
    k_prolong2<<<grid2(nf, nf), dim3(TX, TY), 0, (cudaStream_t)stream>>>(uc, nullptr, nc, uf, nf, 0, cubic ? 1 : 0);
    CK2(cudaGetLastError());
    return MA_OK;
}

}  // extern "C"
