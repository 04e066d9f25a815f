// site_math.cuh -- per-site arithmetic of the leapfrog (Eqs. up_pi, up_E of
// arXiv:1809.00995) of the FP64 step, with every multiply-add written out
// (__fma_rn), since the count of FP64 instructions is the time of the step.
//
// The plaquette sines come from the link phases themselves,
//   Xi_ij = (theta_i^x - theta_i^{x+j}) + (theta_j^{x+i} - theta_j^x),
// instead of from products of four link exponentials: 3 subtractions and an odd
// polynomial instead of ten multiply-adds on eight values, neighbours exchange
// one phase instead of a complex exponential, and the halo of a tile needs no
// sincos of its own except for the one link per site that points into the tile.
#pragma once
#include "ah_internal.cuh"
#include "sincos64.cuh"

namespace ah {
namespace {

__device__ __forceinline__ double fm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double ml(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sb(double a, double b) { return __dsub_rn(a, b); }

template <typename real> struct alignas(2 * sizeof(real)) V2 { real r, i; };
template <typename real> struct alignas(16) V4 { real a, b, c, d; };

// rounding error of s = fl(a + b) (Knuth)
__device__ __forceinline__ double two_sum_err(double a, double b, double s)
{
    const double bb = sb(s, a);
    return ad(sb(a, sb(s, bb)), sb(b, bb));
}

// U phi
template <typename real>
__device__ __forceinline__ V2<real> fwd(V2<real> u, V2<real> f)
{
    return { fm(-u.i, f.i, ml(u.r, f.r)), fm(u.i, f.r, ml(u.r, f.i)) };
}

// U = e^{i theta} of NL links of a site (sincos64.cuh; one warp vote picks the
// range of the polynomials)
template <int NL>
__device__ __forceinline__ void link_exps(const double *t, V2<double> *u)
{
    int m = abs_hi(t[0]);
#pragma unroll
    for (int d = 1; d < NL; ++d) m = max(m, abs_hi(t[d]));
    const unsigned mm = __reduce_max_sync(__activemask(), (unsigned)m);
    if (mm <= kHi2m4) {
#pragma unroll
        for (int d = 0; d < NL; ++d) sincos_range<0>(t[d], &u[d].i, &u[d].r);
    } else if (mm <= kHi04) {
#pragma unroll
        for (int d = 0; d < NL; ++d) sincos_range<1>(t[d], &u[d].i, &u[d].r);
    } else if (mm <= kHi078) {
#pragma unroll
        for (int d = 0; d < NL; ++d) sincos_range<2>(t[d], &u[d].i, &u[d].r);
    } else {
#pragma unroll
        for (int d = 0; d < NL; ++d) sincos_reduced(t[d], 0.0, &u[d].i, &u[d].r);
    }
}

// sin Xi from the link exponentials, whose accuracy does not depend on the phases' size
static __device__ __noinline__ double plaq_far(double ti, double tij, double tj, double tji)
{
    const double2 a = sincos_far64(ti), b = sincos_far64(tji), c = sincos_far64(tij), d = sincos_far64(tj);
    const double abr = a.y * b.y - a.x * b.x, abi = a.y * b.x + a.x * b.y;
    const double cdr = c.y * d.y - c.x * d.x, cdi = c.y * d.x + c.x * d.y;
    return abi * cdr - abr * cdi;
}
// Sines of NX plaquettes from their phases: Xi = (ti - tij) + (tji - tj), the
// phases of U_i^x, U_i^{x+j}, U_j^{x+i}, U_j^x.  Where |Xi| and |ti - tij| are at most
// 0.78 for the whole warp the sum is good to 1.2 x 2^-53, as good as the links it is
// made of, and the odd polynomial applies.  Beyond, the sum's rounding errors
// (Knuth's TwoSum) are added after the range reduction: a Xi near a multiple of
// 2 pi (compact phases on the two sides of the cut) and a small Xi between large phases
// lose nothing.  Differences past 2^18, whose errors are no longer small, go through
// the link exponentials (by a vote too, as calls among the reduced forms take
// registers that the step has none of).
template <int NX>
__device__ __forceinline__ void plaq_sines(const double *ti, const double *tij, const double *tj, const double *tji,
                                           double *p)
{
    double x[NX];
    int m = 0, ma = 0;
#pragma unroll
    for (int k = 0; k < NX; ++k) {
        const double a = sb(ti[k], tij[k]);
        x[k] = ad(a, sb(tji[k], tj[k]));
        m = max(m, abs_hi(x[k]));
        ma = max(ma, abs_hi(a));
    }
    const unsigned mm = __reduce_max_sync(__activemask(), (unsigned)(ma <= kHi078 ? m : max(m, ma)));
    if (mm <= kHi2m4) {
#pragma unroll
        for (int k = 0; k < NX; ++k) p[k] = sin_range<0>(x[k]);
    } else if (mm <= kHi04) {
#pragma unroll
        for (int k = 0; k < NX; ++k) p[k] = sin_range<1>(x[k]);
    } else if (mm <= kHi078) {
#pragma unroll
        for (int k = 0; k < NX; ++k) p[k] = sin_range<2>(x[k]);
    } else if (mm >= kHi2p18) {
#pragma unroll
        for (int k = 0; k < NX; ++k) p[k] = plaq_far(ti[k], tij[k], tj[k], tji[k]);
    } else {
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const double a = sb(ti[k], tij[k]), b = sb(tji[k], tj[k]);
            const double ea = two_sum_err(ti[k], -tij[k], a), eb = two_sum_err(tji[k], -tj[k], b);
            double c;
            sincos_reduced<false>(x[k], ad(two_sum_err(a, b, x[k]), ad(ea, eb)), &p[k], &c);
        }
    }
}

// One kick of Pi (Eq. up_pi) and the scalar currents Im[conj(U_d phi^{x+d}) phi^x]
// of a site: f0 = phi^x, w_d = U_d phi^{x+d}; ub_d, fb_d the link and the field of
// x - d, whose backward product conj(U) phi goes into the Laplacian by
// multiply-adds.
template <typename real>
struct PiKick { real pr, pi, c1, c2, c3; };
template <typename real>
__device__ __forceinline__ PiKick<real> pi_kick(const KickCoef<real> &c, V2<real> f0, V2<real> w1, V2<real> w2,
                                                V2<real> w3, V2<real> ub1, V2<real> fb1, V2<real> ub2, V2<real> fb2,
                                                V2<real> ub3, V2<real> fb3, real pr, real pi)
{
    real lr = fm(real(-6), f0.r, ad(ad(w1.r, w2.r), w3.r));
    real li = fm(real(-6), f0.i, ad(ad(w1.i, w2.i), w3.i));
    lr = fm(ub1.i, fb1.i, fm(ub1.r, fb1.r, lr));
    li = fm(-ub1.i, fb1.r, fm(ub1.r, fb1.i, li));
    lr = fm(ub2.i, fb2.i, fm(ub2.r, fb2.r, lr));
    li = fm(-ub2.i, fb2.r, fm(ub2.r, fb2.i, li));
    lr = fm(ub3.i, fb3.i, fm(ub3.r, fb3.r, lr));
    li = fm(-ub3.i, fb3.r, fm(ub3.r, fb3.i, li));
    const real pot = ml(c.c_pot, sb(fm(f0.r, f0.r, ml(f0.i, f0.i)), c.sigma2));
    PiKick<real> k;
    k.pr = fm(c.c_lap, lr, fm(-pot, f0.r, ml(c.c_damp, pr)));
    k.pi = fm(c.c_lap, li, fm(-pot, f0.i, ml(c.c_damp, pi)));
    k.c1 = fm(w1.r, f0.i, -ml(w1.i, f0.r));
    k.c2 = fm(w2.r, f0.i, -ml(w2.i, f0.r));
    k.c3 = fm(w3.r, f0.i, -ml(w3.i, f0.r));
    return k;
}

// Kick of one E component (Eq. up_E) in two parts: everything but the curl,
// then the curl sum_{j != i} [sin Xi_ij^x - sin Xi_ij^{x-j}], whose terms at the
// neighbours x - j arrive one barrier later.
template <typename real>
__device__ __forceinline__ real e_local(const KickCoef<real> &c, real e, real cur)
{
    return fm(c.c_cur, cur, ml(c.c_edamp, e));
}
template <typename real>
__device__ __forceinline__ real e_kick(const KickCoef<real> &c, real local, real curl)
{
    return fm(-c.c_curl, curl, local);
}

// Drift of a link phase, compact if the run asks for it
template <typename real>
__device__ __forceinline__ real th_drift(const KickCoef<real> &c, real t, real e)
{
    real n = fm(c.dt, e, t);
    if (c.wrap) n = wrap_phase(n);
    return n;
}

}  // namespace
}  // namespace ah
