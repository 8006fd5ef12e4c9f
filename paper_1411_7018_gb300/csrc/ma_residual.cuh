// ma_residual.cuh -- the FP64 fine-grid residual r = rhs - det(D^2_h u)
// (Algorithm 1 step 3; the operator of Eq. MA_discrete) with the partials of
// its max and discrete-L2 norms (stopping rule of Section 4).
//
// FP64 throughput bounds this kernel on GB300, so each thread walks one (i, j)
// column through a contiguous run of k and reuses the x- and y-differences
// Dx = u(i+1) - u(i-1), Dy = u(j+1) - u(j-1) of the planes above and below:
// the xz and yz cross sums are Dx(k+1) - Dx(k-1) and Dy(k+1) - Dy(k-1), two
// FP64 operations per point instead of six.  The norm partials are taken on
// the FP32 value of r (the stopping rule needs ~7 digits of a norm, not 16),
// which keeps them off the FP64 pipe.  Grid: (ceil(n/32), ceil(n/4), kz)
// blocks of 32 x 4 threads, k runs of ceil(n/kz) planes; one partial pair per
// block.
#pragma once

#include "ma_point.cuh"

namespace ma {
namespace resid {

constexpr int RX = 32, RY = 4;

// Writes the residual value of interior point (i, j, k), linear index p
// (H4 = 4 h^2 D^2_h u at the point, for outputs that also store it).
struct NaturalF64Out {
    double* r;
    __device__ __forceinline__ void put(long long p, int, int, int, int, double v, float, const HessS&) const
    {
        r[p] = v;
    }
    __device__ __forceinline__ void zero(long long p) const { r[p] = 0.0; }
};

// Block body with the block index and the grid's dimensions as arguments (a
// batched launch over several grids runs the same code).
template <typename Out>
__device__ __forceinline__ void residual_col_block(const double* __restrict__ u, const double* __restrict__ rhs,
                                                   const Out& out, int n, double inv_h6, double* partials, int kchunk,
                                                   uint3 bid, uint3 gdim)
{
    const int i = bid.x * RX + threadIdx.x;
    const int j = bid.y * RY + threadIdx.y;
    const int k0 = bid.z * kchunk;
    const int k1 = min(n, k0 + kchunk);
    const long long sy = n, sz = (long long)n * n;
    float mx = 0.0f, ss = 0.0f;
    if (i < n && j < n && k0 < k1) {
        const bool col_interior = i > 0 && j > 0 && i < n - 1 && j < n - 1;
        if (!col_interior) {
            for (int k = k0; k < k1; ++k) out.zero(((long long)k * n + j) * n + i);
        } else {
            auto DX = [&](int k) -> double {
                const double* q = u + ((long long)k * n + j) * n + i;
                return __ldg(q + 1) - __ldg(q - 1);
            };
            auto DY = [&](int k) -> double {
                const double* q = u + ((long long)k * n + j) * n + i;
                return __ldg(q + sy) - __ldg(q - sy);
            };
            double dxa = k0 >= 1 ? DX(k0 - 1) : 0.0, dya = k0 >= 1 ? DY(k0 - 1) : 0.0;
            double dxb = DX(k0), dyb = DY(k0);
            for (int k = k0; k < k1; ++k) {
                const long long p = ((long long)k * n + j) * n + i;
                if (k == 0 || k == n - 1) {
                    out.zero(p);
                } else {
                    const double dxc = DX(k + 1), dyc = DY(k + 1);
                    const double* q = u + p;
                    const double v0 = q[0];
                    const double a = __ldg(q + 1) + __ldg(q - 1);
                    const double b = __ldg(q + sy) + __ldg(q - sy);
                    const double c = __ldg(q + sz) + __ldg(q - sz);
                    const double r4 = (__ldg(q + sy + 1) - __ldg(q + sy - 1)) - (__ldg(q - sy + 1) - __ldg(q - sy - 1));
                    HessS H;
                    const double m8v = -8.0 * v0;
                    H.A = fma(4.0, a, m8v);
                    H.B = fma(4.0, b, m8v);
                    H.C = fma(4.0, c, m8v);
                    H.R = r4;
                    H.S = dxc - dxa;
                    H.T = dyc - dya;
                    const double val = fma(-det0(H), inv_h6, rhs[p]);   // inv_h6 = 1 / (64 h^6)
                    const float v32 = d2f_trunc(val);
                    mx = fmaxf(mx, fabsf(v32));
                    ss = fmaf(v32, v32, ss);
                    out.put(p, i, j, k, n, val, v32, H);
                    dxa = dxb; dya = dyb;
                    dxb = dxc; dyb = dyc;
                    continue;
                }
                // boundary plane: advance the difference window
                if (k + 1 <= n - 1) {
                    const double dxc = DX(k + 1), dyc = DY(k + 1);
                    dxa = dxb; dya = dyb;
                    dxb = dxc; dyb = dyc;
                }
            }
        }
    }
    if (partials) {
        __shared__ float smx[RX * RY / 32], sss[RX * RY / 32];
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
            ss += __shfl_down_sync(0xffffffffu, ss, o);
        }
        const int t = threadIdx.y * RX + threadIdx.x;
        if ((t & 31) == 0) { smx[t >> 5] = mx; sss[t >> 5] = ss; }
        __syncthreads();
        if (t == 0) {
            double m = f2d(smx[0]), q = f2d(sss[0]);
            for (int w = 1; w < RX * RY / 32; ++w) { m = fmax(m, f2d(smx[w])); q += f2d(sss[w]); }
            const int slot = (bid.z * gdim.y + bid.y) * gdim.x + bid.x;
            partials[2 * slot] = m;
            partials[2 * slot + 1] = q;
        }
    }
}

template <typename Out>
__global__ void __launch_bounds__(RX * RY) k_residual_col(const double* __restrict__ u, const double* __restrict__ rhs,
                                                          Out out, int n, double inv_h6, double* partials, int kchunk)
{
    residual_col_block<Out>(u, rhs, out, n, inv_h6, partials, kchunk, blockIdx, gridDim);
}

// The larger of a magnitude m and |x| as their bit patterns, which order like
// the values; a NaN is passed over, as fmax does.  (An FP64 maximum holds the
// FP64 pipe as long as an addition.)
__device__ __forceinline__ unsigned long long max_bits(unsigned long long m, double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return b > m && b <= 0x7ff0000000000000ull ? b : m;
}

// One block of NF = 256 threads folds the (max, sum of squares) partials in
// a fixed order: out2 = (max, sqrt(h^3 sum)), the max and discrete L2 norms
// of the stopping rule (Section 4).
constexpr int NF = 256;

__device__ __forceinline__ void norm_final_block(const double* __restrict__ partials, int count, double h3,
                                                 double* out2)
{
    __shared__ unsigned long long smx[NF];
    __shared__ double sss[NF];
    unsigned long long mx = 0;
    double ss = 0.0;
    for (int q = threadIdx.x; q < count; q += NF) {
        mx = max_bits(mx, partials[2 * q]);
        ss += partials[2 * q + 1];
    }
    smx[threadIdx.x] = mx;
    sss[threadIdx.x] = ss;
    __syncthreads();
    for (int w = NF / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            smx[threadIdx.x] = max(smx[threadIdx.x], smx[threadIdx.x + w]);
            sss[threadIdx.x] += sss[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out2[0] = __longlong_as_double((long long)smx[0]);
        out2[1] = sqrt(h3 * sss[0]);
    }
}

inline dim3 grid_for(int n, int kz) { return dim3((n + RX - 1) / RX, (n + RY - 1) / RY, kz); }

// ---------------------------------------------------------------------------
// The residual without FP64 arithmetic (the fine-grid residual of the mixed
// solve).  GB300 issues FP64 at 1/64 of its FP32 rate, which made the FP64
// residual the second most expensive kernel of a mixed solve.  Two facts
// take it off the FP64 pipe:
//  * Doubles of one sign and one binade (one exponent) differ by exact
//    integer multiples of their ulp: x - y = (bits(x) - bits(y)) 2^(E-1075)
//    for the 64-bit patterns, negated for negative values.  When the 19
//    stencil values of a point share the centre's binade, the six second
//    differences of 4 h^2 D^2_h u (the sums of Eq. MA_discrete's stencil,
//    Section 2) are formed exactly in int64 -- more accurately than the FP64
//    gather, which rounds the sums u(x+h) + u(x-h).
//  * The determinant is then evaluated in two-float arithmetic (value = hi +
//    lo, two FP32 numbers, about 48 significant bits), with Knuth's two-sum and
//    the FMA form of Dekker's exact product: |error| of a few 2^-46 relative to
//    the sum of the magnitudes of the determinant's terms, 3e-15 rms and without
//    a bias.  rhs - det is taken in FP64 where the output is FP64, in two floats
//    where it is FP32.
// A stencil that changes binade or sign is handled the same way, each value
// as a fixed-point number of the largest one's scale with 7 bits to spare.
//
// FP32 has the digits but not FP64's range, so the differences are held as
// 2^k 4 h^2 D^2_h u with 2^k next to 1 / (4 h^2) (struct Scaling): they have
// the size of D^2 u whatever the step, and the factor that takes the
// determinant back lies near 1.  A point takes the FP64 evaluation where k would
// leave [-20, 40] (h below 4e-7 or above 600), the stencil's largest value is
// zero or outside [2^-40, 2^20), the determinant overflows FP32, or it and the
// right-hand side are both below 2^-64 (usable()).
// ---------------------------------------------------------------------------
namespace f2 {

struct F2 {
    float hi, lo;
};

// a + b = s + e exactly (Knuth).
__device__ __forceinline__ F2 two_sum(float a, float b)
{
    const float s = a + b;
    const float v = s - a;
    return {s, (a - (s - v)) + (b - v)};
}

// a + b = s + e exactly when |a| >= |b| or a = 0 (Dekker).
__device__ __forceinline__ F2 fast_two_sum(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ F2 mul(F2 x, F2 y)
{
    const float p = x.hi * y.hi;
    float e = fmaf(x.hi, y.hi, -p);   // a * b = p + e exactly
    e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e));
    return fast_two_sum(p, e);
}

// The product left unnormalised (|lo| may exceed half an ulp of hi by the
// few roundings of the cross terms); for operands of add, which renormalises.
__device__ __forceinline__ F2 mul_u(F2 x, F2 y)
{
    const float p = x.hi * y.hi;
    const float e = fmaf(x.hi, y.hi, -p);
    return {p, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e))};
}

__device__ __forceinline__ F2 add(F2 x, F2 y)
{
    const F2 s = two_sum(x.hi, y.hi);
    return fast_two_sum(s.hi, s.lo + (x.lo + y.lo));
}

// The sum left unnormalised (|lo| may reach a few half ulps of hi): saves the
// three dependent operations of the last step where the result only enters a
// product, whose cross terms then drop |lo|^2, or an add.
__device__ __forceinline__ F2 add_u(F2 x, F2 y)
{
    const F2 s = two_sum(x.hi, y.hi);
    return {s.hi, s.lo + (x.lo + y.lo)};
}

__device__ __forceinline__ F2 neg(F2 x) { return {-x.hi, -x.lo}; }

// Exact FP32 value of an integer y in [0, 2^23) or, for the signed form, in
// (-2^22, 2^22): placed in the significand of 2^23 (or 1.5 * 2^23) by an
// integer add, the constant then subtracted exactly.  Integer and FP32
// instructions only (GB300 runs 64-bit integer conversions at its FP64 rate).
__device__ __forceinline__ float u23_to_f(unsigned y) { return __int_as_float(0x4B000000 | (int)y) - 8388608.0f; }
__device__ __forceinline__ float s22_to_f(int y) { return __int_as_float(0x4B400000 + y) - 12582912.0f; }

// x * U as hi + lo, exact, for |x| < 2^45 and U a power of two: x = a 2^23 + c
// with c in [0, 2^23) and |a| < 2^22.  Each piece is placed in the significand
// of 1.5 2^23 (or 2^23) and one FMA scales it and takes the constant off, all
// of it exact.  U23 = 2^23 U.
__device__ __forceinline__ F2 from_i45(long long x, float U, float U23)
{
    const float a = fmaf(__int_as_float(0x4B400000 + (int)(x >> 23)), U23, -12582912.0f * U23);
    const float c = fmaf(__int_as_float(0x4B000000 | ((int)x & 0x7fffff)), U, -8388608.0f * U);
    return fast_two_sum(a, c);
}

// x * scale as hi + lo, |x| < 2^68 (exact to ~2^-48 relative), scale a
// power of two: x = a 2^46 + b 2^23 + c with b, c in [0, 2^23).
__device__ __forceinline__ F2 from_i64(long long x, float scale)
{
    const unsigned c = (unsigned)x & 0x7fffffu;
    const unsigned b = (unsigned)(x >> 23) & 0x7fffffu;
    const int a = (int)(x >> 46);
    const F2 ab = fast_two_sum(s22_to_f(a) * 70368744177664.0f, u23_to_f(b) * 8388608.0f);   // 2^46, 2^23
    const F2 t = two_sum(ab.hi, u23_to_f(c));
    const F2 r = fast_two_sum(t.hi, t.lo + ab.lo);
    return {r.hi * scale, r.lo * scale};
}

// A double as hi + lo, each rounded to nearest (hi: 24 bits, lo: 24 of the 29
// below, signed), with integer and FP32 operations only: within 2^-49 of x, and
// without a bias, for 2^-104 <= |x| < 2^127.  (lo cut off instead of rounded
// is 5e-15 of x too small on average, which a solve carries into u.)  Below 2^-104 hi
// alone, within 2^-129; below 2^-126 zero.
__device__ __forceinline__ F2 from_f64(double x)
{
    const long long b = __double_as_longlong(x);
    const int hw = (int)(b >> 32), ex = (hw >> 20) & 0x7ff;
    const int low = (int)((unsigned)b << 3) >> 3;   // the low 29 bits, signed: x = hi + low ulps, away from 0
    const float hi = d2f_trunc(__longlong_as_double(b + (1ll << 28)));
    if ((unsigned)(ex - 919) > 253u) return {hi, 0.0f};
    const float unit = __int_as_float(((ex - 1045 + 127) << 23) | (hw & 0x80000000));   // +-2^(ex-1045), 2^30 ulps
    return {hi, __int2float_rn(low) * 9.31322574615478515625e-10f * unit};              // 2^-30
}

// det(H) for the symmetric 3x3 H = [[A, R, S], [R, B, T], [S, T, C]]: the
// cofactor expansion along the first row.  UNORM leaves the sums inside
// unnormalised: about 15 of 91 operations fewer, and up to twice the error
// (1.7e-15 against 1.4e-15 of max f on the rational-arithmetic test's 129^3
// points, where FP64's rounded neighbour sums leave 4e-12).
template <bool UNORM = false>
__device__ __forceinline__ F2 det3(const F2& A, const F2& B, const F2& C, const F2& R, const F2& S, const F2& T)
{
    auto sum = [](F2 x, F2 y) { return UNORM ? add_u(x, y) : add(x, y); };
    const F2 c1 = sum(mul_u(B, C), neg(mul_u(T, T)));
    const F2 c2 = sum(mul_u(R, C), neg(mul_u(S, T)));
    const F2 c3 = sum(mul_u(R, T), neg(mul_u(B, S)));
    return sum(sum(mul_u(A, c1), neg(mul_u(R, c2))), mul_u(S, c3));
}

// The exact paths accept binades E with 2^(E-1075), and a scaling 2^k of it
// for -20 <= k <= 40, inside FP32's normal range: 2^-40 <= |u| < 2^20.
constexpr int kMinE = 1023 - 40, kMaxE = 1023 + 20;

}  // namespace f2

// A level's scaling and constants, from its step h.
struct Scaling {
    double h6, inv_h6;   // 64 h^6, the right-hand side's factor of the FP64 forms, and its inverse
    double c, inv_c;     // (2^k 4 h^2)^3 and its inverse
    double kz;           // 2^-k / 8: a root z of the scaled matrix to the change of u
    double kh;           // 2^k: 4 h^2 D^2_h u to the scaled differences
    float kb;            // scaled differences to D^2_h u
    int kexp;            // k, or kNone: every point takes the FP64 form
};
constexpr int kNone = 1 << 20;

inline Scaling make_scaling(double h)
{
    Scaling P{};
    const double h2 = h * h;
    P.h6 = 64.0 * h2 * h2 * h2;
    P.inv_h6 = 1.0 / P.h6;
    int e = 0;
    const double m = frexp(4.0 * h2, &e);   // 4 h^2 = m 2^e, m in [1/2, 1)
    P.kexp = m < 0.70710678118654752 ? 1 - e : -e;
    if (P.kexp < -20 || P.kexp > 40) {
        P.kexp = kNone;
        P.kh = 1.0 / (4.0 * h2);   // the FP64 form's differences as D^2_h u
        P.kb = 1.0f;
        return P;
    }
    const double q = ldexp(4.0 * h2, P.kexp);   // in [0.7, 1.42)
    P.c = q * q * q;
    P.inv_c = 1.0 / P.c;
    P.kz = ldexp(0.125, -P.kexp);
    P.kh = ldexp(1.0, P.kexp);
    P.kb = (float)(1.0 / q);
    return P;
}

// Whether the two-float determinant d of scaled differences serves rhs - det and
// rhs + det: none of its products overflowed (an infinity or NaN stays one to the
// end), and what they lost below FP32's range, some 2^-126, lies below the
// rounding of the larger of d and rhs.
__device__ __forceinline__ bool usable(f2::F2 d, double rhs)
{
    return fabsf(d.hi) < 3.0e38f &&
           (fabsf(d.hi) >= 5.421010862427522e-20f || (__double2hiint(rhs) & 0x7ff00000) >= (1023 - 64) << 20);   // 2^-64
}

// Residual rhs - det(D^2_h u) at an interior point and the scaled differences
// for outputs that store them.
struct ResF2 {
    double v;      // FP64 outputs
    float v32;     // its FP32 rounding
    float H[6];    // 2^k 4 h^2 D^2_h u: xx, yy, zz, xy, xz, yz
};

// H = 2^kexp 4 h^2 D^2_h u at a point, formed exactly in int64 and held as
// two-float values; ld(o) gives the bits of the value at offset o from the
// point, sy and sz are the offsets of a step in j and k.  false (H unset) where
// the stencil's largest value is zero, huge or tiny.  -20 <= kexp <= 40 keeps
// every scaled unit inside FP32's range.
// FORM, how a warp that meets a change of binade is served: kDirect, for grids
// that fill the GPU: stencils of one binade first, the general form for the
// rest; kSmall, for grids where most warps meet one and a phase is one point's
// chain: all by a left shift where it serves the warp.
enum Form { kDirect, kSmall };

template <int FORM = kDirect, typename Idx, typename Ld>
__device__ __forceinline__ bool gather_f2_of(Ld ld, Idx sy, Idx sz, int kexp, f2::F2* H, long long* centre)
{
    const long long b0 = ld(0);
    const long long bxp = ld(1), bxm = ld(-1), byp = ld(sy), bym = ld(-sy), bzp = ld(sz), bzm = ld(-sz);
    const long long rpp = ld(sy + 1), rmm = ld(-sy - 1), rpm = ld(sy - 1), rmp = ld(1 - sy);
    const long long spp = ld(sz + 1), smm = ld(-sz - 1), spm = ld(sz - 1), smp = ld(1 - sz);
    const long long tpp = ld(sz + sy), tmm = ld(-sz - sy), tpm = ld(sz - sy), tmp = ld(sy - sz);
    *centre = b0;
    // one sign and one exponent: the top 12 bits of every pattern equal b0's
    const unsigned h0 = (unsigned)(b0 >> 32);
    unsigned diff = 0;
#define MA_F2_CK(v) diff |= (unsigned)((v) >> 32) ^ h0
    MA_F2_CK(bxp); MA_F2_CK(bxm); MA_F2_CK(byp); MA_F2_CK(bym); MA_F2_CK(bzp); MA_F2_CK(bzm);
    MA_F2_CK(rpp); MA_F2_CK(rmm); MA_F2_CK(rpm); MA_F2_CK(rmp);
    MA_F2_CK(spp); MA_F2_CK(smm); MA_F2_CK(spm); MA_F2_CK(smp);
    MA_F2_CK(tpp); MA_F2_CK(tmm); MA_F2_CK(tpm); MA_F2_CK(tmp);
#undef MA_F2_CK
    int E = (int)((h0 >> 20) & 0x7ff);
    int sign = (int)(h0 & 0x80000000u);   // the ulp of the binade, negated for negative values
    // a quarter of the diagonal entries, and the off-diagonal ones, in ulps
    long long A, B, C, R, S, T;
    if (FORM == kDirect && (diff >> 20) == 0) {
        if (E < f2::kMinE || E > f2::kMaxE) return false;
        A = (bxp - b0) + (bxm - b0);
        B = (byp - b0) + (bym - b0);
        C = (bzp - b0) + (bzm - b0);
        R = (rpp - rmp) - (rpm - rmm);
        S = (spp - smp) - (spm - smm);
        T = (tpp - tmp) - (tpm - tmm);
    } else {
        // The stencil changes binade or sign: each value as its signed
        // significand in units of 2^-7 of the largest one's ulp.  Exact down
        // to 2^-7 of the largest value, truncated by less than 2^-7 of its
        // ulp below (a sum in FP64 rounds by half of one); four of them fit
        // int64.
        auto mag = [](long long b) { return (unsigned)(b >> 32) & 0x7fffffffu; };
        auto max4 = [&](long long a, long long b, long long c, long long d) {
            return max(max(mag(a), mag(b)), max(mag(c), mag(d)));
        };
        const unsigned top = max(max(max(max4(bxp, bxm, byp, bym), max4(bzp, bzm, b0, b0)),
                                     max(max4(rpp, rmm, rpm, rmp), max4(spp, smm, spm, smp))),
                                 max4(tpp, tmm, tpm, tmp));
        E = (int)(top >> 20);
        if (E < f2::kMinE || E > f2::kMaxE) return false;
        auto sums = [&](auto g) {
            const long long m0 = g(b0);
            A = (g(bxp) - m0) + (g(bxm) - m0);
            B = (g(byp) - m0) + (g(bym) - m0);
            C = (g(bzp) - m0) + (g(bzm) - m0);
            R = (g(rpp) - g(rmp)) - (g(rpm) - g(rmm));
            S = (g(spp) - g(smp)) - (g(spm) - g(smm));
            T = (g(tpp) - g(tmp)) - (g(tpm) - g(tmm));
        };
        // (zeros and denormals shift out with the rest: E exceeds 63 by far)
        auto fix = [E](long long b) -> long long {
            const long long m = (b & 0x000FFFFFFFFFFFFFll) | 0x0010000000000000ll;
            return (m << 7) >> min(E - (int)((b >> 52) & 0x7ff), 63);
        };
        // all of one sign (the unit carries it) and within seven binades: a left
        // shift, a third fewer instructions, but 16 registers more (129^3: 48 us
        // the right-hand side with it, 36 without)
        const int low = E - 7 + (int)((h0 >> 20) & 0x800);
        auto left = [low](long long b) { return (int)((unsigned)(b >> 32) >> 20) - low; };
        bool near = false;
        if (FORM == kSmall) {
            const int far = (left(bxp) | left(bxm) | left(byp)) | (left(bym) | left(bzp) | left(bzm)) |
                            (left(rpp) | left(rmm) | left(rpm)) | (left(rmp) | left(spp) | left(smm)) |
                            (left(spm) | left(smp) | left(tpp)) | (left(tmm) | left(tpm) | left(tmp)) | left(b0);
            near = !__any_sync(__activemask(), (unsigned)far > 7u);
        }
        if (near) {
            sums([&](long long b) { return ((b & 0x000FFFFFFFFFFFFFll) | 0x0010000000000000ll) << left(b); });
        } else if (FORM == kDirect && !__any_sync(__activemask(), (int)diff < 0)) {
            sums(fix);
        } else {
            // a stencil of one sign keeps its unit's sign whatever its warp's others hold: the conversion of a
            // sum beyond 2^48 rounds a value and its negative differently, so the bits would depend on them
            const long long mixed = (int)diff >> 31;
            sums([&](long long b) {
                const long long v = fix(b), neg = (b >> 63) & mixed;
                return (v ^ neg) - neg;
            });
            sign &= (int)~mixed;
        }
        E -= 7;
    }
    const float unit = __int_as_float(((E - 1075 + 127 + kexp) << 23) | sign);
    const float unit4 = 4.0f * unit;
    // |x| < 2^45 for all six (the common case on fine grids): the two-piece
    // conversion; otherwise the three-piece one
    int big = 0;
#define MA_F2_HW(x) big |= (int)((x) >> 32) ^ (int)((x) >> 63)
    MA_F2_HW(A); MA_F2_HW(B); MA_F2_HW(C); MA_F2_HW(R); MA_F2_HW(S); MA_F2_HW(T);
#undef MA_F2_HW
    if (FORM == kDirect && big < (1 << 13)) {
        const float u23 = 8388608.0f * unit, u423 = 8388608.0f * unit4;
        H[0] = f2::from_i45(A, unit4, u423);
        H[1] = f2::from_i45(B, unit4, u423);
        H[2] = f2::from_i45(C, unit4, u423);
        H[3] = f2::from_i45(R, unit, u23);
        H[4] = f2::from_i45(S, unit, u23);
        H[5] = f2::from_i45(T, unit, u23);
    } else {
        H[0] = f2::from_i64(A, unit4);
        H[1] = f2::from_i64(B, unit4);
        H[2] = f2::from_i64(C, unit4);
        H[3] = f2::from_i64(R, unit);
        H[4] = f2::from_i64(S, unit);
        H[5] = f2::from_i64(T, unit);
    }
    return true;
}

// The same at interior point p of a grid in global memory, through the
// read-only path (no launch writes a point and reads it as a neighbour).
template <typename Idx>
__device__ __forceinline__ bool gather_f2(const double* __restrict__ u, Idx p, Idx sy, Idx sz, int kexp, f2::F2* H,
                                          long long* centre)
{
    const long long* q = reinterpret_cast<const long long*>(u) + p;
    return gather_f2_of<kDirect, Idx>([q](Idx o) -> long long { return __ldg(q + o); }, sy, sz, kexp, H, centre);
}

// F64: the value in FP64, the right-hand side with all its digits (two FP64
// operations); otherwise its FP32 rounding, from two floats.  ic: P.inv_c as two
// floats.  false: the point needs the FP64 form.
template <bool F64, bool UNORM>
__device__ __forceinline__ bool residual_point_f2(const double* __restrict__ u, long long p, long long sy,
                                                  long long sz, double rhs, const Scaling& P, f2::F2 ic, ResF2* out)
{
    f2::F2 H[6];
    long long b0;
    if (P.kexp == kNone || !gather_f2<long long>(u, p, sy, sz, P.kexp, H, &b0)) return false;
    const f2::F2 d = f2::det3<UNORM>(H[0], H[1], H[2], H[3], H[4], H[5]);
    if (!usable(d, rhs)) return false;
    if constexpr (F64) {
        out->v = fma(-(f2d(d.hi) + f2d(d.lo)), P.inv_c, rhs);
        out->v32 = d2f_trunc(out->v);
    } else {
        out->v32 = f2::add(f2::from_f64(rhs), f2::neg(f2::mul(d, ic))).hi;
    }
    for (int c = 0; c < 6; ++c) out->H[c] = H[c].hi;
    return true;
}

// r + sign det(D^2_h u) in FP64, for the points the two-float forms leave (out of
// line: inline it cost those forms 8 registers); q points at the centre.
static __device__ __noinline__ double operator_f64(const double* q, long long sy, long long sz, double r, double inv_h6,
                                                   int sign)
{
    auto at = [&](long long o) { return q[o]; };
    const HessS G = gather_hess_of(at, sy, sz, at(0));
    return fma(sign * det0(G), inv_h6, r);
}

// Block body: one (i, j) column per thread over a run of k (as
// residual_col_block), each point evaluated by residual_point_f2; Out::put2
// receives (its Column, p, k, ResF2).  Out::put64 evaluates the points left in
// FP64, in a second walk of a run that has any (a call within the first took the
// 513^3 residual of a mixed solve from 2055 to 2260 us; this one takes 2094).
// Norm partials from the FP32 rounding of the value.
template <typename Out, int NN = 0>
__device__ __forceinline__ void residual_f2_block(const double* __restrict__ u, const double* __restrict__ rhs,
                                                  const Out& out, int n_rt, const Scaling& P, double* partials,
                                                  int kchunk, uint3 bid, uint3 gdim)
{
    // NN > 0: the grid size at compile time, so the stencil offsets are
    // immediates of the loads (the same values and arithmetic either way)
    const int n = NN > 0 ? NN : n_rt;
    const int i = bid.x * RX + threadIdx.x;
    const int j = bid.y * RY + threadIdx.y;
    const int k0 = bid.z * kchunk;
    const int k1 = min(n, k0 + kchunk);
    const long long sy = n, sz = (long long)n * n;
    const float ih = (float)P.inv_c;
    const f2::F2 ic = {ih, (float)(P.inv_c - (double)ih)};
    float mx = 0.0f, ss = 0.0f;
    if (i < n && j < n && k0 < k1) {
        const bool col_interior = i > 0 && j > 0 && i < n - 1 && j < n - 1;
        const typename Out::Column col(i, j, n);
        bool left = false;   // a point for FP64
        for (int k = k0; k < k1; ++k) {
            const long long p = ((long long)k * n + j) * n + i;
            if (!col_interior || k == 0 || k == n - 1) {
                out.zero(p);
                continue;
            }
            ResF2 r;
            const double b = rhs[p];
            if (!residual_point_f2<Out::kF64, Out::kUnorm>(u, p, sy, sz, b, P, ic, &r)) {
                left = true;
                continue;
            }
            out.put2(col, p, k, r);
            mx = fmaxf(mx, fabsf(r.v32));
            ss = fmaf(r.v32, r.v32, ss);
        }
        for (int k = max(k0, 1); left && k < min(k1, n - 1); ++k) {
            const long long p = ((long long)k * n + j) * n + i;
            ResF2 r;
            const double b = rhs[p];
            if (residual_point_f2<Out::kF64, Out::kUnorm>(u, p, sy, sz, b, P, ic, &r)) continue;
            const float v32 = out.put64(col, p, k, u + p, sy, sz, b, P);
            mx = fmaxf(mx, fabsf(v32));
            ss = fmaf(v32, v32, ss);
        }
    }
    if (partials) {
        __shared__ float smx[RX * RY / 32], sss[RX * RY / 32];
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
            ss += __shfl_down_sync(0xffffffffu, ss, o);
        }
        const int t = threadIdx.y * RX + threadIdx.x;
        if ((t & 31) == 0) { smx[t >> 5] = mx; sss[t >> 5] = ss; }
        __syncthreads();
        if (t == 0) {
            double m = f2d(smx[0]), q = f2d(sss[0]);
            for (int w = 1; w < RX * RY / 32; ++w) { m = fmax(m, f2d(smx[w])); q += f2d(sss[w]); }
            const int slot = (bid.z * gdim.y + bid.y) * gdim.x + bid.x;
            partials[2 * slot] = m;
            partials[2 * slot + 1] = q;
        }
    }
}

// 8 resident blocks at 64 registers (5 at 96 with the size at run time): left to
// itself the compiler takes 72 for the calls of the second walk.  None spill.
template <typename Out, int NN = 0>
__global__ void __launch_bounds__(RX * RY, NN > 0 ? 8 : 5)
    k_residual_f2(const double* __restrict__ u, const double* __restrict__ rhs, Out out, int n, Scaling P,
                  double* partials, int kchunk)
{
    residual_f2_block<Out, NN>(u, rhs, out, n, P, partials, kchunk, blockIdx, gridDim);
}

// Launch with the grid size fixed at compile time for the sizes of a
// hierarchy's larger levels (the runtime form takes up to 115 registers for
// its 64-bit offsets).
template <typename Out>
void launch_k_residual_f2(dim3 grid, cudaStream_t s, const double* u, const double* rhs, Out out, int n,
                          const Scaling& P, double* partials, int kchunk)
{
    const dim3 blk(RX, RY);
    switch (n) {
    case 33: k_residual_f2<Out, 33><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    case 65: k_residual_f2<Out, 65><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    case 129: k_residual_f2<Out, 129><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    case 257: k_residual_f2<Out, 257><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    case 513: k_residual_f2<Out, 513><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    default: k_residual_f2<Out, 0><<<grid, blk, 0, s>>>(u, rhs, out, n, P, partials, kchunk); break;
    }
}

// FP64 output of the two-float residual.  UNORM: the determinant with
// unnormalised sums (f2::det3).
template <bool UNORM>
struct NaturalF2Out {
    static constexpr bool kF64 = true, kUnorm = UNORM;
    double* r;
    struct Column {
        __device__ __forceinline__ Column(int, int, int) {}
    };
    __device__ __forceinline__ void put2(const Column&, long long p, int, const ResF2& v) const
    {
        r[p] = v.v;
    }
    __device__ __forceinline__ float put64(const Column&, long long p, int, const double* q, long long sy, long long sz,
                                           double rhs, const Scaling& P) const
    {
        const double v = operator_f64(q, sy, sz, rhs, P.inv_h6, -1);
        r[p] = v;
        return d2f_trunc(v);
    }
    __device__ __forceinline__ void zero(long long p) const { r[p] = 0.0; }
};

}  // namespace resid
}  // namespace ma
