// device_math.cuh -- time-integrated heat kernels and Chebyshev helpers for the GPU kernels.
//
// Section 2, Eq. heat_kernel: G(r, s) = (4 pi alpha s)^(-3/2) exp(-r^2 / (4 alpha s)) for s > 0.
// The Galerkin entries of V_h integrate G over a target step and a source step; with uniform
// steps h and offset d = k - j they are second differences of the second time antiderivative
//   G2(r, s) = [(s + r^2/(2 alpha)) erfc(u) - r sqrt(s/(pi alpha)) e^{-u^2}] / (4 pi alpha r),
//   u = r / (2 sqrt(alpha s)),
// V_d(r) = G2((d+1)h) - 2 G2(d h) + G2((d-1)h)   (G2 = 0 for s <= 0).
// For d >= 1 the part of G2 linear in s cancels; when u is small we evaluate the bounded form
//   G2t = G2 - s/(4 pi alpha r)
//       = r erfc(u)/(8 pi alpha^2) - sqrt(s) (erf(u)/u)/(8 pi alpha^1.5) - sqrt(s) e^{-u^2}/(4 pi^1.5 alpha^1.5),
// and for large u the plain form (whose terms then carry no common linear part).
// The double layer alpha dG/dn_y = (x - y).n_y G / (2 s) integrates to (x - y).n_y * DL2 with
//   DL2 = [(s/r^2 - 1/(2 alpha)) erfc(u) + sqrt(s/(pi alpha)) e^{-u^2} / r] / (4 pi r),
//   DL2t = DL2 - s/(4 pi r^3) = -[u phi2(u)/2 + erfc(u)] / (8 pi alpha r),
//   phi2(u) = (erf(u) - 2u e^{-u^2}/sqrt(pi)) / u^3.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace pfmm {
namespace dev {

constexpr double kPi = 3.14159265358979323846;
constexpr double kSqrtPi = 1.77245385090551602730;

__device__ __forceinline__ double d_erf(double x) { return erf(x); }
__device__ __forceinline__ float d_erf(float x) { return erff(x); }
__device__ __forceinline__ double d_erfc(double x) { return erfc(x); }
__device__ __forceinline__ float d_erfc(float x) { return erfcf(x); }
__device__ __forceinline__ double d_exp(double x) { return exp(x); }
__device__ __forceinline__ float d_exp(float x) { return expf(x); }
__device__ __forceinline__ double d_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float d_sqrt(float x) { return sqrtf(x); }

// erf(u) and erfc(u), each from the function that is accurate for it
template <typename R>
__device__ __forceinline__ void erf_pair(R u, R &ef, R &efc)
{
    if (u < R(0.5)) {
        ef = d_erf(u);
        efc = R(1) - ef;
    } else {
        efc = d_erfc(u);
        ef = R(1) - efc;
    }
}

// A constant of the formulas below: FP64, or in FP32 the rounded value and what that leaves.  One FP32
// rounding of it would be the same for every entry, and the second differences in time amplify what
// the step ends' constants differ by (768 triangles x 256 steps, alpha 0.5: the nearfield came out 7.5e-7 from FP64
// instead of 3.4e-7)
template <typename R>
struct Num {
    R hi;
    __host__ __device__ constexpr void set(double v) { hi = v; }
};
template <>
struct Num<float> {
    float hi, lo;
    __host__ __device__ constexpr void set(double v)
    {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    }
};
__device__ __forceinline__ double mulc(double x, Num<double> c) { return x * c.hi; }
__device__ __forceinline__ float mulc(float x, Num<float> c) { return fmaf(x, c.hi, x * c.lo); }
__device__ __forceinline__ double addc(double x, Num<double> c) { return c.hi + x; }
__device__ __forceinline__ float addc(float x, Num<float> c) { return c.hi + (x + c.lo); }
__device__ __forceinline__ double subc(double x, Num<double> c) { return x - c.hi; }
__device__ __forceinline__ float subc(float x, Num<float> c) { return (x - c.hi) - c.lo; }
template <typename R>
__device__ constexpr Num<R> num(double v)
{
    Num<R> c{};
    c.set(v);
    return c;
}

// erf(u)/u (Maclaurin series below 0.05), iu = 1/u
template <typename R>
__device__ __forceinline__ R erf_over_u(R u, R ef, R iu)
{
    if (u < R(0.05)) {
        R u2 = u * u;
        R s = R(1) + u2 * (R(-1.0 / 3.0) + u2 * (R(1.0 / 10.0) + u2 * (R(-1.0 / 42.0) + u2 * R(1.0 / 216.0))));
        return mulc(s, num<R>(2.0 / kSqrtPi));
    }
    return ef * iu;
}

// phi2(u) = (erf(u) - 2u e^{-u^2}/sqrt(pi)) / u^3; series (2/sqrt(pi)) sum_{n>=1} (-1)^{n+1} 2n u^{2n-2} / (n! (2n+1))
// iu = 1/u
template <typename R>
__device__ __forceinline__ R phi2(R u, R ef, R ex, R iu)
{
    if (u < R(0.5)) {
        R u2 = u * u, acc = R(0);
        // Horner from n = 12 down to n = 1
        double fact[13] = {1, 1, 2, 6, 24, 120, 720, 5040, 40320, 362880, 3628800, 39916800, 479001600};
#pragma unroll
        for (int n = 12; n >= 1; --n) {
            double c = (2.0 * n) / (fact[n] * (2.0 * n + 1.0));
            acc = acc * u2 + R((n % 2) ? c : -c);
        }
        return mulc(acc, num<R>(2.0 / kSqrtPi));
    }
    return (ef - mulc(u, num<R>(2.0 / kSqrtPi)) * ex) * (iu * iu * iu);
}

// Constants of the step ends s = k h, k = 1 .. nd, and of the formulas above, from the host in FP64
template <typename R>
struct TimeConst {
    Num<R> cu[8], icu[8];       // u = r cu, 1/u = icu / r:  cu = 1 / (2 sqrt(alpha s))
    Num<R> s[8], b1[8], b2[8];  // s, sqrt(s) / (8 pi alpha^1.5), sqrt(s) / (4 pi^1.5 alpha^1.5)
    Num<R> b3[8];               // sqrt(s / (pi alpha))
    Num<R> a1, a2, clin, k8;    // 1 / (8 pi alpha^2), 1 / (2 alpha), 1 / (4 pi alpha), 1 / (8 pi alpha)
    void set(double h, double alpha, int nd)
    {
        const double a32 = alpha * sqrt(alpha);
        for (int k = 0; k < nd; ++k) {
            const double sk = (k + 1) * h, ss = sqrt(sk);
            cu[k].set(1.0 / (2.0 * sqrt(alpha) * ss));
            icu[k].set(2.0 * sqrt(alpha) * ss);
            s[k].set(sk);
            b1[k].set(ss / (8.0 * kPi * a32));
            b2[k].set(ss / (4.0 * kPi * sqrt(kPi) * a32));
            b3[k].set(ss / sqrt(kPi * alpha));
        }
        a1.set(1.0 / (8.0 * kPi * alpha * alpha));
        a2.set(1.0 / (2.0 * alpha));
        clin.set(1.0 / (4.0 * kPi * alpha));
        k8.set(1.0 / (8.0 * kPi * alpha));
    }
};

// Time integrals for d = 0 .. ND-1 at distance r: V[d] of the single layer and K[d] of the double
// layer (to be multiplied by (x - y).n_y; 0 at r = 0).  r must be > 0 when d = 0 of V is used.  Both
// layers share erf, erfc and exp of a step end; the divisions are one reciprocal of r (a step end
// costs some 130 FP64 operations for both instead of some 700).
template <typename R, bool DOV, bool DOK, int ND>
__device__ __forceinline__ void time_integrals(R r, const TimeConst<R> &c, R *V, R *K)
{
    const R ir = r > R(0) ? R(1) / r : R(0), r2 = r * r;
    R g1 = R(0), g2 = R(0), t1 = R(0), t2 = R(0);  // G2, bounded form at k - 1 and k - 2
    R d1 = R(0), d2 = R(0), e1 = R(0), e2 = R(0);  // the same of the double layer
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        const R u = mulc(r, c.cu[k]), iu = mulc(ir, c.icu[k]);
        R ef, efc;
        erf_pair(u, ef, efc);
        const R ex = d_exp(-u * u);
        const bool small = u < R(1);
        if (DOV) {
            const R t = mulc(r * efc, c.a1) - mulc(erf_over_u(u, ef, iu), c.b1[k]) - mulc(ex, c.b2[k]);
            const R g = (addc(mulc(r2, c.a2), c.s[k]) * efc - mulc(r, c.b3[k]) * ex) * mulc(ir, c.clin);
            V[k] = k == 0 ? g : (small ? t - t1 - t1 + t2 : g - g1 - g1 + g2);
            g2 = g1;
            g1 = g;
            t2 = t1;
            t1 = t;
        }
        if (DOK) {
            const R g = (subc(mulc(ir, c.s[k]) * ir, c.a2) * efc + mulc(ex, c.b3[k]) * ir) * mulc(ir, num<R>(1.0 / (4 * kPi)));
            const R t = -(R(0.5) * u * phi2(u, ef, ex, iu) + efc) * mulc(ir, c.k8);
            K[k] = k == 0 ? g : (small ? t - e1 - e1 + e2 : g - d1 - d1 + d2);
            d2 = d1;
            d1 = g;
            e2 = e1;
            e1 = t;
        }
    }
}

// G2 and its bounded form G2t (above) at one time difference s (both 0 for s <= 0)
__device__ __forceinline__ void g2_and_g2t(double r, double s, double alpha, double &g2, double &g2t)
{
    if (!(s > 0.0)) {
        g2 = g2t = 0.0;
        return;
    }
    const double ss = sqrt(s), a32 = alpha * sqrt(alpha), u = r / (2.0 * sqrt(alpha) * ss);
    double ef, efc;
    erf_pair(u, ef, efc);
    const double ex = exp(-u * u);
    g2t = r * efc / (8.0 * kPi * alpha * alpha) - ss * erf_over_u(u, ef, 1.0 / u) / (8.0 * kPi * a32) -
          ss * ex / (4.0 * kPi * kSqrtPi * a32);
    g2 = r > 0.0 ? ((s + r * r / (2.0 * alpha)) * efc - r * ss / sqrt(kPi * alpha) * ex) / (4.0 * kPi * alpha * r) : 0.0;
}

// Single-layer entry factor for a target step (tk0, tk1] and a source step (tj0, tj1] of any
// lengths (general time steps): the second difference of G2 over the four time differences;
// 0 for a later source step, G2(tk1 - tk0) alone for the same step (r > 0 then).  As for uniform
// steps the bounded form is taken when u at the largest difference is below 1 (the linear parts
// cancel when the source step precedes the target step).
__device__ __forceinline__ double time_V_steps(double r, double tk0, double tk1, double tj0, double tj1,
                                               double alpha)
{
    if (tj0 >= tk1) return 0.0;
    double g[4], gt[4];
    if (tj0 == tk0 && tj1 == tk1) {
        g2_and_g2t(r, tk1 - tk0, alpha, g[0], gt[0]);
        return g[0];
    }
    const double s[4] = {tk1 - tj0, tk1 - tj1, tk0 - tj0, tk0 - tj1};
    for (int i = 0; i < 4; ++i) g2_and_g2t(r, s[i], alpha, g[i], gt[i]);
    const double u = r / (2.0 * sqrt(alpha * s[0]));
    return u < 1.0 ? (gt[0] - gt[1]) - (gt[2] - gt[3]) : (g[0] - g[1]) - (g[2] - g[3]);
}

// Chebyshev polynomials T_0..T_m at x (three-term recurrence)
template <typename R>
__device__ __forceinline__ void cheb_all(R x, int m, R *T)
{
    T[0] = R(1);
    if (m >= 1) T[1] = x;
    for (int k = 2; k <= m; ++k) T[k] = R(2) * x * T[k - 1] - T[k - 2];
}

// derivatives T_k'(x) = k U_{k-1}(x)
template <typename R>
__device__ __forceinline__ void cheb_deriv_all(R x, int m, R *dT)
{
    R u0 = R(1), u1 = R(2) * x;
    dT[0] = R(0);
    if (m >= 1) dT[1] = R(1);
    for (int k = 2; k <= m; ++k) {
        dT[k] = R(k) * u1;
        R u2 = R(2) * x * u1 - u0;
        u0 = u1;
        u1 = u2;
    }
}

}  // namespace dev
}  // namespace pfmm
