// ma_smooth_f2.cuh -- the FP64 smoother's point update (Section 2) with its
// arithmetic off the FP64 pipe.  GB300 issues FP64 at 1/64 of its FP32 rate,
// and the FP64 form of this update (35 FP64 operations a point) held that pipe
// at 85 % of its peak: 137 us per colour at 257^3, against 20 us for the
// bytes.  Here the six second differences are exact integers
// (resid::gather_f2), the determinant at the shifted Hessian is taken in
// two-float arithmetic, and three FP64 operations are left: the scaling of the
// right-hand side and the addition of the change to the centre value.
//
// Measured per sweep under graph replay (Example 4 / random cosine, us), FP64
// form -> this one: 257^3 1075 / 1076 -> 329 / 380, 129^3 152 / 152 -> 64 / 74,
// 65^3 34 / 34 -> 24 / 24, 33^3 26 / 26 -> 15 / 15 (two sweeps in one cluster
// launch).  Bound at 257^3 by issue (about 450 integer and FP32 instructions a
// point); at 65^3 and below by the length of one point's dependent chain.  The random cosine's values
// cross more binades, so more warps take gather_f2's fixed-point branch.
//
// Scaling (resid::Scaling): H = 2^k 4 h^2 D^2_h u with 2^k next to 1 / (4 h^2);
// the local equation det(H - z I) = (2^k 4 h^2)^3 rhs has the root of Eq.
// (realroots) at v = v0 + z / (8 2^k).
//
// The root is found as smallest_root finds it: in FP32 on the rounded entries
// (by the iteration of corr_root_fast where it is small, else by Newton from 0,
// or from left of it where the matrix is not positive definite), then one Newton
// correction whose residual is evaluated to about 2^-45 of the entries' cube (in
// FP64 there), with the FP32 derivative.  The second
// differences it starts from are exact, where the FP64 gather rounds the
// neighbour sums to 2^-53 |u|, so from 17^3 up the result lies closer to the
// exact update.  A point that smallest_root would not solve by that path
// (rhs <= 0, degenerate, no convergence), or whose stencil gather_f2 refuses,
// takes the FP64 form.
#pragma once

#include "ma_point.cuh"
#include "ma_residual.cuh"

namespace ma {
namespace smoothf2 {

using Params = resid::Scaling;
using resid::kNone;
inline Params make_params(double h) { return resid::make_scaling(h); }

// The new centre value by the FP64 form, for the points the fast path leaves;
// q points at the centre.
static __device__ __noinline__ double point_f64(const double* q, long long sy, long long sz, double rhs6,
                                                bool* nonconvex)
{
    auto at = [&](long long o) { return q[o]; };
    const double v0 = at(0);
    const HessS H = gather_hess_of(at, sy, sz, v0);
    return fma(0.125, smallest_root(H, rhs6, nonconvex), v0);
}

// a - z as two floats, z one float
__device__ __forceinline__ resid::f2::F2 shift(resid::f2::F2 a, float z)
{
    const resid::f2::F2 s = resid::f2::two_sum(a.hi, -z);
    return resid::f2::fast_two_sum(s.hi, s.lo + a.lo);
}

// The new centre value; ld as gather_f2_of takes it, b the right-hand side.
// false: the point needs the FP64 form.  UNORM: det3's sums unnormalised, which
// saves 15 operations and leaves the root's residual to about 2^-45 of the
// entries' cube in place of 2^-46; that is below an ulp of u from 33^3 up.
template <bool UNORM, int FORM, typename Idx, typename Ld>
__device__ __forceinline__ bool update(Ld ld, Idx sy, Idx sz, double b, const Params& P, double* v)
{
    using namespace resid;
    f2::F2 H[6];
    long long b0;
    // on a small grid ahead of the gather, which hides its latency (33^3 solve: 2 % of it); on one that fills the
    // GPU after it, in fewer registers (257^3 solve: 1 %)
    f2::F2 r6;
    if (FORM == kSmall) r6 = f2::from_f64(__dmul_rn(P.c, b));
    // rhs > 0 by its bits (NaN passes and fails to converge below)
    if (!gather_f2_of<FORM, Idx>(ld, sy, sz, P.kexp, H, &b0) || __double_as_longlong(b) <= 0) return false;
    if (FORM == kDirect) r6 = f2::from_f64(__dmul_rn(P.c, b));
    HessSf F;
    F.A = H[0].hi; F.B = H[1].hi; F.C = H[2].hi;
    F.R = H[3].hi; F.S = H[4].hi; F.T = H[5].hi;
    const float scale = fabsf(F.A) + fabsf(F.B) + fabsf(F.C) + fabsf(F.R) + fabsf(F.S) + fabsf(F.T);
    // the FP32 root of c - M z + T z^2 - z^3 = det(F - z I) - r6
    const float d0 = det_shift_f(F, 0.0f), c = d0 - r6.hi, T = F.A + F.B + F.C, M = minors_shift_f(F, 0.0f);
    const bool pd = is_pd<HessSf, float>(F, d0);
    const float tol = 2e-6f * scale;
    // a root that is small against the entries: two steps of z <- (c + z^2 (T - z)) / M, one reciprocal
    const float iM = __fdividef(1.0f, M), z0 = __fmul_rn(c, iM);
    const float z1 = __fmul_rn(fmaf(__fmul_rn(z0, z0), T - z0, c), iM);
    float z = __fmul_rn(fmaf(__fmul_rn(z1, z1), T - z1, c), iM);
    bool conv = pd && M > 0.05f * scale * scale && fabsf(T * z0) <= 0.05f * M && fabsf(z - z1) <= tol;
    if (!conv) {
        z = pd ? 0.0f : gershgorin_low<HessSf, float>(F) - cbrtf(r6.hi);
        for (int it = 0; it < 60; ++it) {
            const float dz = __fdividef(fmaf(-z, fmaf(-z, T - z, M), c), fmaf(-z, fmaf(-3.0f, z, 2.0f * T), M));
            z += dz;
            if (!isfinite(z)) break;
            if (fabsf(dz) <= tol) { conv = true; break; }
        }
    }
    const float m = fmaf(-z, fmaf(-3.0f, z, 2.0f * T), M);
    // the scale's window keeps the cube's low parts inside FP32's range
    if (!(conv && m > 0.05f * scale * scale && r6.hi > 0.0f && scale > 9.5e-7f && scale < 1.0e9f)) return false;
    const f2::F2 d = f2::det3<UNORM>(shift(H[0], z), shift(H[1], z), shift(H[2], z), H[3], H[4], H[5]);
    const f2::F2 g = UNORM ? f2::add_u(d, f2::neg(r6)) : f2::add(d, f2::neg(r6));
    const float dz = __fdividef(g.hi + g.lo, m);
    *v = fma(P.kz, f2d(z) + f2d(dz), __longlong_as_double(b0));
    return true;
}

// A point of a grid in global memory, in place.
template <bool UNORM, int FORM, typename Idx>
__device__ __forceinline__ void point(double* u, const double* __restrict__ rhs, Idx p, Idx sy, Idx sz,
                                      const Params& P, unsigned long long* events)
{
    const long long* q = reinterpret_cast<const long long*>(u) + p;
    const double b = __ldg(rhs + p);
    double v;
    if (update<UNORM, FORM, Idx>([q](Idx o) -> long long { return __ldg(q + o); }, sy, sz, b, P, &v)) {
        u[p] = v;   // (one store after both forms: 10 % slower at 257^3)
        return;
    }
    bool nonconvex = false;
    u[p] = point_f64(u + p, sy, sz, __dmul_rn(P.h6, b), &nonconvex);
    if (nonconvex && events) atomicAdd(events, 1ull);
}

// A point of a grid in shared memory: its new value.
__device__ __forceinline__ double point_sm(const double* q, int sy, int sz, double b, const Params& P, bool* nonconvex)
{
    double v;
    if (P.kexp != kNone &&
        update<false, resid::kSmall, int>([q](int o) -> long long { return __double_as_longlong(q[o]); }, sy, sz, b, P, &v))
        return v;
    return point_f64(q, sy, sz, __dmul_rn(P.h6, b), nonconvex);
}

}  // namespace smoothf2
}  // namespace ma
