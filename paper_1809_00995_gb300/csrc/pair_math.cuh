// pair_math.cuh -- packed two-wide FP32 arithmetic (sm_100 FFMA2 / FMUL2 / FADD2)
// on two sites of neighbouring rows, and the link and plaquette phases in that
// form.
//
// One instruction works on both sites, so a kernel bound by instruction issue
// handles nearly twice the sites per issue slot.  Packed operands take no sign
// modifier: differences are a + (-1) b by one multiply-add (the same rounding as
// a - b), and the sign of a sine is applied once per link.  Every operation is
// written with its rounding, so the compiler neither fuses nor splits any: an
// element gets the same bits as in any other kernel that uses these forms.
#pragma once
#include "ah_internal.cuh"

namespace ah {
namespace {

// the library's sine and cosine, out of line: its stack and registers are not the
// callers'
static __device__ __noinline__ float2 sincos_far(float t)
{
    float2 r;
    sincosf(t, &r.x, &r.y);
    return r;
}
__device__ __forceinline__ float2 pk(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fm(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 ml(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 ad(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sb(float2 a, float2 b) { return __ffma2_rn(b, pk(-1.f), a); }
__device__ __forceinline__ float2 ng(float2 a) { return __fmul2_rn(a, pk(-1.f)); }

// phi-like complex pair and a link exponential with the negated sine beside it
struct C22 { float2 r, i; };
struct U22 { float2 r, i, n; };
__device__ __forceinline__ C22 fwd(const U22 &u, const C22 &f)
{
    return { fm(u.n, f.i, ml(u.r, f.r)), fm(u.i, f.r, ml(u.r, f.i)) };
}
__device__ __forceinline__ C22 bwd(const U22 &u, const C22 &f)
{
    return { fm(u.i, f.i, ml(u.r, f.r)), fm(u.n, f.r, ml(u.r, f.i)) };
}

// Coefficients of a step as pairs, with the signs in which they are used.
struct KickCoef2 {
    float2 c_damp, n_pot, c_lap, c_edamp, c_cur, n_curl, dt, n_sigma2;
    int wrap;
};
__host__ __device__ inline KickCoef2 pair_coef(const KickCoef<float> &c)
{
    auto p = [](float a) { return make_float2(a, a); };
    return { p(c.c_damp), p(-c.c_pot), p(c.c_lap), p(c.c_edamp), p(c.c_cur), p(-c.c_curl), p(c.dt), p(-c.sigma2),
             c.wrap };
}

struct PiKick2 { float2 pr, pi, c1, c2, c3; };
__device__ __forceinline__ PiKick2 pi_kick(const KickCoef2 &c, const C22 &f0, const C22 &w1, const C22 &w2,
                                           const C22 &w3, const C22 &b1, const C22 &b2, const C22 &b3, float2 pr,
                                           float2 pi)
{
    const float2 lr = fm(pk(-6.f), f0.r, ad(ad(ad(w1.r, b1.r), ad(w2.r, b2.r)), ad(w3.r, b3.r)));
    const float2 li = fm(pk(-6.f), f0.i, ad(ad(ad(w1.i, b1.i), ad(w2.i, b2.i)), ad(w3.i, b3.i)));
    const float2 npot = ml(c.n_pot, ad(fm(f0.r, f0.r, ml(f0.i, f0.i)), c.n_sigma2));
    const float2 nr = ng(f0.r);
    PiKick2 k;
    k.pr = fm(c.c_lap, lr, fm(npot, f0.r, ml(c.c_damp, pr)));
    k.pi = fm(c.c_lap, li, fm(npot, f0.i, ml(c.c_damp, pi)));
    k.c1 = fm(w1.r, f0.i, ml(w1.i, nr));
    k.c2 = fm(w2.r, f0.i, ml(w2.i, nr));
    k.c3 = fm(w3.r, f0.i, ml(w3.i, nr));
    return k;
}
__device__ __forceinline__ float2 e_local(const KickCoef2 &c, float2 e, float2 cur)
{
    return fm(c.c_cur, cur, ml(c.c_edamp, e));
}
__device__ __forceinline__ float2 e_kick(const KickCoef2 &c, float2 local, float2 curl)
{
    return fm(c.n_curl, curl, local);
}
__device__ __forceinline__ float2 th_drift(const KickCoef2 &c, float2 t, float2 e)
{
    float2 n = fm(c.dt, e, t);
    if (c.wrap) {
        n.x = wrap_phase(n.x);
        n.y = wrap_phase(n.y);
    }
    return n;
}

__device__ __forceinline__ float2 sin_poly2(float2 r)
{
    const float2 r2 = ml(r, r);
    float2 ps = fm(r2, pk(2.755731884e-06f), pk(-1.984127011e-04f));
    ps = fm(r2, ps, pk(8.333333768e-03f));
    ps = fm(r2, ps, pk(-1.666666716e-01f));
    return fm(ml(r, r2), ps, r);
}
__device__ __forceinline__ float2 cos_poly2(float2 r)
{
    const float2 r2 = ml(r, r);
    float2 pc = fm(r2, pk(-2.755731998e-07f), pk(2.480158764e-05f));
    pc = fm(r2, pc, pk(-1.388888923e-03f));
    pc = fm(r2, pc, pk(4.166666791e-02f));
    pc = fm(r2, pc, pk(-0.5f));
    return fm(r2, pc, pk(1.f));
}
__device__ __forceinline__ float amax2(float2 a) { return fmaxf(fabsf(a.x), fabsf(a.y)); }

// t + lo reduced to r in [-pi/4, pi/4] (sincos32.cuh); the low bits of *qx, *qy
// are the quadrants.  Valid for |t| < 2^17.
__device__ __forceinline__ float2 reduce2(float2 t, float2 lo, int *qx, int *qy)
{
    const float2 magic = pk(12582912.0f);                  // 1.5 * 2^23
    const float2 kb = fm(t, pk(0x1.45f306p-1f), magic);    // t 2/pi + magic
    *qx = __float_as_int(kb.x);
    *qy = __float_as_int(kb.y);
    const float2 kf = ad(kb, pk(-12582912.0f));
    float2 r = fm(kf, pk(-0x1.921fb6p+0f), t);
    r = fm(kf, pk(0x1.777a5cp-25f), r);
    r = fm(kf, pk(0x1.ee59dap-50f), r);
    return ad(r, lo);
}
__device__ __forceinline__ float flip(float a, int bit1)   // -a if bit 1 of the argument is set
{
    return __int_as_float(__float_as_int(a) ^ ((bit1 & 2) << 30));
}

// U = e^{i theta} of NL links of both sites; one warp vote on the largest phase
// picks the polynomials alone (|theta| <= 0.78) or the reduced forms.
template <int NL>
__device__ __forceinline__ void link_exps2(const float2 *t, U22 *u)
{
    float m = amax2(t[0]);
#pragma unroll
    for (int d = 1; d < NL; ++d) m = fmaxf(m, amax2(t[d]));
    if (__all_sync(__activemask(), m <= 0.78f)) {
#pragma unroll
        for (int d = 0; d < NL; ++d) {
            u[d].i = sin_poly2(t[d]);
            u[d].r = cos_poly2(t[d]);
        }
    } else {
#pragma unroll
        for (int d = 0; d < NL; ++d) {
            int qx, qy;
            const float2 r = reduce2(t[d], pk(0.f), &qx, &qy);
            const float2 s = sin_poly2(r), c = cos_poly2(r);
            u[d].i.x = flip((qx & 1) ? c.x : s.x, qx);
            u[d].r.x = flip((qx & 1) ? s.x : c.x, qx + 1);
            u[d].i.y = flip((qy & 1) ? c.y : s.y, qy);
            u[d].r.y = flip((qy & 1) ? s.y : c.y, qy + 1);
            if (!(amax2(t[d]) < 131072.0f)) {
                const float2 a = sincos_far(t[d].x), b = sincos_far(t[d].y);
                u[d].i = make_float2(a.x, b.x);
                u[d].r = make_float2(a.y, b.y);
            }
        }
    }
#pragma unroll
    for (int d = 0; d < NL; ++d) u[d].n = ng(u[d].i);
}

// sin Xi from the link exponentials, whose accuracy does not depend on the phases' size
static __device__ __noinline__ float plaq_far(float ti, float tij, float tj, float tji)
{
    const float2 a = sincos_far(ti), b = sincos_far(tji), c = sincos_far(tij), d = sincos_far(tj);
    const float abr = a.y * b.y - a.x * b.x, abi = a.y * b.x + a.x * b.y;
    const float cdr = c.y * d.y - c.x * d.x, cdi = c.y * d.x + c.x * d.y;
    return abi * cdr - abr * cdi;
}
// Sines of NX plaquettes of both sites from their link phases, Xi = (ti - tij) +
// (tji - tj).  Where |Xi| and |ti - tij| are at most 0.78 for the whole warp the sum is
// good to 1.2 x 2^-24, as good as the links it is made of, and the odd polynomial
// applies.  Beyond, the sum's rounding errors (Knuth's TwoSum) are added after the
// range reduction: a Xi near a multiple of 2 pi and a small Xi between large phases
// lose nothing.  Differences past 2^15, whose errors are no longer small, go through
// the link exponentials (by a vote, too).  What asking for |ti - tij| costs: 256^3 230.2 ->
// 231.0 us per step on a string network, 286 -> 293 us on random phases of 0.7.
template <int NX>
__device__ __forceinline__ void plaq_sines2(const float2 *ti, const float2 *tij, const float2 *tj, const float2 *tji,
                                            float2 *p)
{
    float2 x[NX];
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < NX; ++k) {
        const float2 a = sb(ti[k], tij[k]);
        x[k] = ad(a, sb(tji[k], tj[k]));
        m = fmaxf(fmaxf(m, amax2(a)), amax2(x[k]));
    }
    if (__all_sync(__activemask(), m <= 0.78f)) {
#pragma unroll
        for (int k = 0; k < NX; ++k) p[k] = sin_poly2(x[k]);
    } else if (__any_sync(__activemask(), m >= 32768.0f)) {
#pragma unroll
        for (int k = 0; k < NX; ++k)
            p[k] = make_float2(plaq_far(ti[k].x, tij[k].x, tj[k].x, tji[k].x),
                               plaq_far(ti[k].y, tij[k].y, tj[k].y, tji[k].y));
    } else {
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            // rounding errors of the three additions (Knuth)
            auto err = [](float2 a, float2 b, float2 s) {
                const float2 bb = sb(s, a);
                return ad(sb(a, sb(s, bb)), sb(b, bb));
            };
            const float2 a = sb(ti[k], tij[k]), b = sb(tji[k], tj[k]);
            const float2 lo = ad(err(a, b, x[k]), ad(err(ti[k], ng(tij[k]), a), err(tji[k], ng(tj[k]), b)));
            int qx, qy;
            const float2 r = reduce2(x[k], lo, &qx, &qy);
            const float2 s = sin_poly2(r), c = cos_poly2(r);
            p[k].x = flip((qx & 1) ? c.x : s.x, qx);
            p[k].y = flip((qy & 1) ? c.y : s.y, qy);
        }
    }
}

}  // namespace
}  // namespace ah
