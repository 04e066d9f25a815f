// sincos64.cuh -- double-precision sines and cosines of link and plaquette
// phases.
//
// GB300 issues two FP64 lanes per clock and SM, so the count of FP64
// instructions is the time of an FP64 step; integer tests and votes are free
// beside them.  sin r = r + r^3 S(r^2) and cos r = 1 - r^2/2 + r^4 C(r^2) with
// polynomials S, C that interpolate the exact functions at the Chebyshev nodes of
// r^2 in [0, R^2] (computed in 60 digits and rounded), for three ranges picked by
// a warp vote on the high words of the phases.  Number of coefficients and
// largest error of the rounded polynomials in units of 2^-53 (sine relative,
// cosine absolute):
//   R = 2^-4     3 + 3   0.18, 7e-5
//   R = 0.4      5 + 5   0.05, 6e-4
//   R = 0.7855   6 + 6   0.18, 8e-3
// Beyond pi/4 (0.78 is tested) an additive range reduction in the manner of
// Cody & Waite: k = nearest integer to t 2/pi, r = t - k pi/2 with pi/2 split
// into P1 + P2 + P3, P1 = fl(pi/2), P2 = fl(pi/2 - P1), P3 = fl(pi/2 - P1 - P2),
// by fused multiply-adds.  Arguments with |t| >= 2^20 go to the library's sincos.
#pragma once

namespace ah {

// S and C of range R (0: 2^-4, 1: 0.4, 2: 0.7855) at u = r^2
template <int R>
__device__ __forceinline__ double sin_series(double u)
{
    if constexpr (R == 0)
        return __fma_rn(u, __fma_rn(u, -0x1.a01156816e25bp-13, 0x1.11111104106ccp-7), -0x1.555555555549cp-3);
    double p;
    if constexpr (R == 1) {
        p = __fma_rn(u, -0x1.ad4a2c774fcaep-26, 0x1.71ddeb5be025cp-19);
        p = __fma_rn(u, p, -0x1.a01a018e0dab9p-13);
        p = __fma_rn(u, p, 0x1.111111110f9f8p-7);
        return __fma_rn(u, p, -0x1.5555555555554p-3);
    }
    p = __fma_rn(u, 0x1.5e0ae5873e651p-33, -0x1.ae600a711c40ep-26);
    p = __fma_rn(u, p, 0x1.71de3795fe529p-19);
    p = __fma_rn(u, p, -0x1.a01a019e833f2p-13);
    p = __fma_rn(u, p, 0x1.1111111110bb1p-7);
    return __fma_rn(u, p, -0x1.5555555555555p-3);
}
template <int R>
__device__ __forceinline__ double cos_series(double u)
{
    if constexpr (R == 0)
        return __fma_rn(u, __fma_rn(u, 0x1.a013125156a5cp-16, -0x1.6c16c161afd1cp-10), 0x1.555555555550bp-5);
    double p;
    if constexpr (R == 1) {
        p = __fma_rn(u, 0x1.1e4c4c059fc62p-29, -0x1.27e4ce544be23p-22);
        p = __fma_rn(u, p, 0x1.a01a0195c9378p-16);
        p = __fma_rn(u, p, -0x1.6c16c16c15ee3p-10);
        return __fma_rn(u, p, 0x1.5555555555555p-5);
    }
    p = __fma_rn(u, -0x1.907d6ee97cd28p-37, 0x1.1eeb68a05cf19p-29);
    p = __fma_rn(u, p, -0x1.27e4fa17941a8p-22);
    p = __fma_rn(u, p, 0x1.a01a019f4e7a2p-16);
    p = __fma_rn(u, p, -0x1.6c16c16c16966p-10);
    return __fma_rn(u, p, 0x1.5555555555555p-5);
}
template <int R>
__device__ __forceinline__ double sin_range(double r)
{
    const double u = __dmul_rn(r, r);
    return __fma_rn(__dmul_rn(r, u), sin_series<R>(u), r);
}
template <int R>
__device__ __forceinline__ void sincos_range(double r, double *s, double *c)
{
    const double u = __dmul_rn(r, r);
    *s = __fma_rn(__dmul_rn(r, u), sin_series<R>(u), r);
    *c = __fma_rn(u, __fma_rn(u, cos_series<R>(u), -0.5), 1.0);
}
// 1 - cos r, without cancellation
template <int R>
__device__ __forceinline__ double vers_range(double r)
{
    const double u = __dmul_rn(r, r);
    return __dmul_rn(u, __fma_rn(u, -cos_series<R>(u), 0.5));
}
static __device__ __noinline__ double2 sincos_far64(double t)
{
    double2 r;
    sincos(t, &r.x, &r.y);
    return r;
}
// sin, cos of t + lo, |lo| small beside |t| (the rounding error of a sum that
// gave t; 0 for a phase taken as it is).  Without FAR |t| < 2^20 is the caller's to see to.
template <bool FAR = true>
__device__ __forceinline__ void sincos_reduced(double t, double lo, double *s, double *c)
{
    if (FAR && !(fabs(t) < 1048576.0)) {
        const double2 r = sincos_far64(t);
        *s = r.x;
        *c = r.y;
        return;
    }
    const double kf = rint(__dmul_rn(t, 0.63661977236758134308));                    // 2/pi
    double r = __fma_rn(-kf, 0x1.921fb54442d18p+0, t);                                // P1
    r = __fma_rn(-kf, 0x1.1a62633145c07p-54, r);                                      // P2
    r = __fma_rn(-kf, -0x1.f1976b7ed8fbcp-110, r);                                    // P3
    r = __dadd_rn(r, lo);
    double sr, cr;
    sincos_range<2>(r, &sr, &cr);
    const int q = (int)kf;
    const double a = (q & 1) ? cr : sr, b = (q & 1) ? sr : cr;
    *s = (q & 2) ? -a : a;
    *c = ((q + 1) & 2) ? -b : b;
}

// |t| by its high word, which orders as |t| does to 2^-20, and the ranges' bounds
__device__ __forceinline__ int abs_hi(double t) { return __double2hiint(t) & 0x7fffffff; }
__device__ __forceinline__ int abs_hi3(const double t[3]) { return max(abs_hi(t[0]), max(abs_hi(t[1]), abs_hi(t[2]))); }
constexpr int kHi2m4 = 0x3faffffe;       // just below 2^-4
constexpr int kHi04 = 0x3fd99998;        // just below 0.4
constexpr int kHi078 = 0x3fe8f5c1;       // just below 0.78
constexpr int kHi2p18 = 0x41100000;      // 2^18

}  // namespace ah
