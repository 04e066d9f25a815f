// diag_tile.cuh -- the whole-lattice diagnostics of one state (Sec. 2 of
// arXiv:1809.00995) on a tile, marched in z: energy sums, Gauss residual and
// plaquette windings, nothing written back.
//
// A CTA of 256 threads takes 32 x 8 columns of sites, a chunk of z planes at a
// time, and keeps its sums in registers over all the columns it takes; each site
// is one thread's.  Per plane and site: the three forward products U_d phi^{x+d}
// (the gradient energy), the three plaquette phases from the link phases
// (1 - cos Xi by its own series, without cancellation or division), and the
// Gauss residual (double-float for FP32 states, or FP64: G64).
//
// Windings without arctangents per edge.  With alpha = arg phi of each site, the
// bracket of Eq. 9 on link e from a to b is [alpha_b - alpha_a + theta_e] =
// alpha_b - alpha_a + theta_e - 2 pi n_e, n_e the nearest integer of that over
// 2 pi; around a plaquette the alphas cancel, so
//   W = (sum of the four brackets - [Xi]) / 2 pi = N - (n_1 + n_2 - n_3 - n_4),
// N the nearest integer of Xi / 2 pi: one arctangent per site and small integers.
// alpha is good to 1e-6 in FP32; where a bracket or [Xi] comes within 2^-15 of
// +-pi (kCutMargin), phi is too small or too large for alpha, or a phase makes
// thousands of turns (kMaxTurns), the plaquette goes to the list that the FP64 path
// decides, so the counts are those of the FP64 formula on the same state.  A site needs n_2, n_3 of x + 1 and n_1, n_3 of x + y
// (one packed word each) and its own n_1, n_2 of the next plane, so the windings
// of plane z - 1 are summed while plane z is worked on, and a plane costs one
// barrier (two copies of the shared arrays).
//
// FP32 is bound by instruction issue, FP64 by its pipe.  Against a walk with the
// step's link exponentials and chained edge products: FP32 512^3 5.48 -> 3.95 ms
// (this walk serves N that are no multiple of 4 or below 40, diag_pair.cuh the
// others; 381^3 1.60 ms), FP64 256^3 14.9 -> 5.7 ms.
#pragma once
#include <cmath>

#include "diag_common.cuh"
#include "fused_common.cuh"
#include "sincos32.cuh"
#include "site_math.cuh"

namespace ah {
namespace {

constexpr float kCutMargin = 1.0f / 32768.0f;
constexpr float kPi32 = 3.14159265f, kTwoPi32 = 6.28318531f, kInvTwoPi32 = 0.159154943f;

// atan(a) / a on [0, 1] as a polynomial in a^2 (interpolated at the Chebyshev
// nodes; largest error of atan 4.3e-7)
__device__ __forceinline__ float atan_unit(float a)
{
    const float u = a * a;
    float p = fmaf(u, 7.648353930562735e-03f, -3.636043146252632e-02f);
    p = fmaf(u, p, 8.312645554542542e-02f);
    p = fmaf(u, p, -1.344786435365677e-01f);
    p = fmaf(u, p, 1.9872039556503296e-01f);
    p = fmaf(u, p, -3.332567811012268e-01f);
    p = fmaf(u, p, 9.999992251396179e-01f);
    return a * p;
}
// arg phi to about 1e-6, or NaN where phi is too small, too large or not a number
// (maximum and minimum pass over one NaN component, the sum does not)
__device__ __forceinline__ float site_phase(float r, float i)
{
    const float x = fabsf(r), y = fabsf(i), hi = fmaxf(x, y), lo = fminf(x, y);
    float a = atan_unit(__fdividef(lo, hi));
    a = y > x ? 0.5f * kPi32 - a : a;
    a = r < 0.f ? kPi32 - a : a;
    a = i < 0.f ? -a : a;
    return hi > 1e-30f && x + y < 1e30f ? a : __int_as_float(0x7fc00000);
}
// FP64 phi past the range above: its phase is that of phi over a power of two
static __device__ __noinline__ float site_phase_scaled(double r, double i)
{
    const double m = fmax(fabs(r), fabs(i));
    if (!(m > 0.0 && m <= 0x1.fffffffffffffp+1023)) return __int_as_float(0x7fc00000);
    const int e = ilogb(m);
    return site_phase((float)scalbn(r, -e), (float)scalbn(i, -e));
}
__device__ __forceinline__ float site_phase(double r, double i)
{
    const float a = site_phase((float)r, (float)i);
    return a == a ? a : site_phase_scaled(r, i);
}

// n of a link whose bracket is a - 2 pi n, and whether the bracket is too near
// the cut: adding 1.5 x 2^23 rounds to the nearest integer, which the low bits then
// hold.
constexpr float kRound = 12582912.0f;
constexpr int kRoundBits = 0x4b400000;
__device__ __forceinline__ int turns(float a, bool *cut)
{
    const float kb = __fmaf_rn(a, kInvTwoPi32, kRound), k = __fsub_rn(kb, kRound);
    *cut = !(fabsf(fmaf(-k, kTwoPi32, a)) <= kPi32 - kCutMargin);
    return __float_as_int(kb) - kRoundBits;
}
// k modulo 16, in [-8, 7].  Turns are counted modulo 16: a winding is at most 2, and
// what the fields below add up, four links' turns (at most 8 each) and N, stays
// within a field's 8 bits whatever the phases, so that a plaquette left to the FP64
// list, whose sum lacks terms, borrows nothing from the next field.
__device__ __forceinline__ int turns16(int k) { return (int)((unsigned)k << 28) >> 28; }
// t - 2 pi k, k the nearest integer of t / 2 pi (or its neighbour, where t / 2 pi rounds
// across a half).  FP32 with 2 pi in two parts: up to 4 kMaxTurns turns the first
// difference is exact and the second good to an ulp of pi.
__device__ __forceinline__ float less_turns(float t, float *k)
{
    *k = rintf(t * kInvTwoPi32);
    return fmaf(*k, 1.74845553e-7f, fmaf(-*k, 6.28318548f, t));
}
__device__ __forceinline__ float less_turns(double t, float *k)
{
    const double kd = rint(t * 0.15915494309189535);
    *k = (float)kd;
    return (float)fma(-kd, 6.283185307179586, t);
}
// n_1, n_2, n_3 of a site's links to neighbours of phase b[], and a bit for each
// that is too near the cut.  Phases past 8 give up their whole turns first.  Links
// with more than kMaxTurns turns count as near the cut (and plaquettes with more than
// four times as many), which sends all their plaquettes to the FP64 list: at 128^3,
// random phases of up to 32 turns, a pass takes 0.13 ms, and 6.7 ms where the limit
// lets the list overflow and every plaquette is counted again.
constexpr float kMaxTurns = 4096.f;
template <typename real>
__device__ __forceinline__ int link_turns(float a, const float b[3], const real t[3], int n[3])
{
    const float f[3] = { (float)t[0], (float)t[1], (float)t[2] };
    const float m = fmaxf(fabsf(f[0]), fmaxf(fabsf(f[1]), fabsf(f[2])));
    bool c[3];
    if (__all_sync(__activemask(), m <= 8.f)) {
#pragma unroll
        for (int d = 0; d < 3; ++d) n[d] = turns(b[d] - a + f[d], &c[d]);
    } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float k;
            const float r = less_turns(t[d], &k);
            n[d] = turns(b[d] - a + r, &c[d]);
            c[d] = c[d] || !(fabsf(k) <= kMaxTurns);
            n[d] = c[d] ? 0 : turns16(n[d] + (int)k);
        }
    }
    if (!__any_sync(__activemask(), c[0] | c[1] | c[2])) return 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) n[d] = c[d] ? 0 : n[d];
    return (int)c[0] | (int)c[1] << 1 | (int)c[2] << 2;
}
// The terms that a link's n adds to n_1 + n_2 - n_3 - n_4 of the plaquettes (12),
// (13), (23), as three 8-bit fields (modulo 2^24) under three cut bits: of a site's
// own links, of its links seen from x - 1 and from x - y, and from z - 1.  Words are
// added, cut bits or-ed; windings takes the sum apart.
__device__ __forceinline__ unsigned field_word(int v, int cut) { return ((unsigned)v & 0xffffffu) | (unsigned)cut << 24; }
__device__ __forceinline__ unsigned own_word(const int n[3], int c)
{
    const int v = n[0] * 257 + n[1] * 65535 - n[2] * 65792;
    return field_word(v, c ? ((c | c >> 1) & 1) | ((c | c >> 2) & 1) << 1 | ((c >> 1 | c >> 2) & 1) << 2 : 0);
}
__device__ __forceinline__ unsigned x_word(int n2, int n3, int c)
{
    return field_word(n2 + n3 * 256, c ? (c >> 1 & 1) | (c >> 2 & 1) << 1 : 0);
}
__device__ __forceinline__ unsigned y_word(int n1, int n3, int c)
{
    return field_word(n3 * 65536 - n1, c ? (c & 1) | (c >> 2 & 1) << 2 : 0);
}
__device__ __forceinline__ unsigned z_word(const int n[3], int c)
{
    return field_word(-n[0] * 256 - n[1] * 65536, c ? (c & 1) << 1 | (c >> 1 & 1) << 2 : 0);
}
// The three windings of a sum of words, N - (n_1 + n_2 - n_3 - n_4): fields are at most
// 4 x 8 + 8 in size, so each is its low 8 bits with their sign.
__device__ __forceinline__ void windings(unsigned t, int w[3])
{
    const int w12 = (int)(t << 24) >> 24, r1 = (((int)(t << 8) >> 8) - w12) >> 8;
    const int w13 = (int)((unsigned)r1 << 24) >> 24;
    w[0] = turns16(w12);
    w[1] = turns16(w13);
    w[2] = turns16((r1 - w13) >> 8);
}

// 1 - cos Xi summed over the three plaquettes of a site, from the four phases of
// each (as in Eq. 3: ti, tj at x, tij = theta_i^{x+j}, tji = theta_j^{x+i}); *word
// the whole turns -N of each and the plaquettes whose [Xi] is too near the cut.  As in
// the steps' plaq_sines the sum's rounding errors are kept unless |Xi| and |ti - tij|
// are small for the whole warp, and the energies (the turns come with cut links) of
// differences past 2^15 (FP64: 2^18) are those of the link exponentials.
static __device__ __noinline__ float vers_far(float ti, float tij, float tj, float tji)
{
    C2<float> a, b, c, d;
    sincosf(ti, &a.i, &a.r);
    sincosf(tji, &b.i, &b.r);
    sincosf(tij, &c.i, &c.r);
    sincosf(tj, &d.i, &d.r);
    const C2<float> z = cmul(cmul(a, b), conj(cmul(c, d)));
    return one_minus_cos(z.r, z.i);
}
static __device__ __noinline__ double vers_far(double ti, double tij, double tj, double tji)
{
    C2<double> a, b, c, d;
    sincos(ti, &a.i, &a.r);
    sincos(tji, &b.i, &b.r);
    sincos(tij, &c.i, &c.r);
    sincos(tj, &d.i, &d.r);
    const C2<double> z = cmul(cmul(a, b), conj(cmul(c, d)));
    return one_minus_cos(z.r, z.i);
}
__device__ __forceinline__ float xi_terms(const float *ti, const float *tij, const float *tj, const float *tji,
                                          unsigned *word)
{
    float x[3], m = 0.f, sum = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = ti[k] - tij[k];
        x[k] = a + (tji[k] - tj[k]);
        m = fmaxf(m, fmaxf(fabsf(a), fabsf(x[k])));
    }
    *word = 0;
    if (__all_sync(__activemask(), m <= 0.78f)) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            // through x^8 / 8!: the next term is below 1e-8 of the sum
            const float u = x[k] * x[k];
            float p = fmaf(u, -2.480158764e-05f, 1.388888923e-03f);
            p = fmaf(u, p, -4.166666791e-02f);
            sum = fmaf(u, fmaf(u, p, 0.5f), sum);
        }
        return sum;
    }
    int n = 0, cuts = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const DF d1 = two_sum(ti[k], -tij[k]), d2 = two_sum(tji[k], -tj[k]), d3 = two_sum(d1.h, d2.h);
        const float lo = d3.l + (d1.l + d2.l);
        float kf;
        const float r = less_turns(d3.h, &kf) + lo;      // [Xi]
        const bool cut = !(fabsf(r) <= kPi32 - kCutMargin) || !(fabsf(kf) <= 4.f * kMaxTurns);
        cuts |= cut << k;
        n -= cut ? 0 : turns16((int)kf) << 8 * k;
        float s, c;
        sincos_link(0.5f * r, &s, &c);
        sum = fmaf(2.f * s, s, sum);
    }
    if (__any_sync(__activemask(), m >= 32768.f)) {
        sum = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) sum += vers_far(ti[k], tij[k], tj[k], tji[k]);
    }
    *word = field_word(n, cuts);
    return sum;
}
__device__ __forceinline__ double xi_terms(const double *ti, const double *tij, const double *tj, const double *tji,
                                           unsigned *word)
{
    double x[3], sum = 0.0;
    int m = 0, ma = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double a = sb(ti[k], tij[k]);
        x[k] = ad(a, sb(tji[k], tj[k]));
        m = max(m, abs_hi(x[k]));
        ma = max(ma, abs_hi(a));
    }
    *word = 0;
    const unsigned mm = __reduce_max_sync(__activemask(), (unsigned)(ma <= kHi078 ? m : max(m, ma)));
    if (mm <= kHi04) {
#pragma unroll
        for (int k = 0; k < 3; ++k) sum += mm <= kHi2m4 ? vers_range<0>(x[k]) : vers_range<1>(x[k]);
        return sum;
    }
    int n = 0, cuts = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float kf;
        const float r = less_turns(x[k], &kf);           // [Xi]
        const bool cut = !(fabsf(r) <= kPi32 - kCutMargin) || !(fabsf(kf) <= 4.f * kMaxTurns);
        cuts |= cut << k;
        n -= cut ? 0 : turns16((int)kf) << 8 * k;
        const double a = sb(ti[k], tij[k]), b = sb(tji[k], tj[k]);
        const double ea = two_sum_err(ti[k], -tij[k], a), eb = two_sum_err(tji[k], -tj[k], b);
        double s, c;
        sincos_reduced(0.5 * x[k], 0.5 * ad(two_sum_err(a, b, x[k]), ad(ea, eb)), &s, &c);
        sum += 2.0 * s * s;
    }
    if (mm >= kHi2p18) {
        sum = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) sum += vers_far(ti[k], tij[k], tj[k], tji[k]);
    }
    *word = field_word(n, cuts);
    return sum;
}

__device__ __forceinline__ void diag_links(const float t[3], float s[3], float c[3]) { sincos_link3(t, s, c); }
__device__ __forceinline__ void diag_links(const double t[3], double s[3], double c[3])
{
    const unsigned m = __reduce_max_sync(__activemask(), (unsigned)abs_hi3(t));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (m <= kHi04) sincos_range<1>(t[d], &s[d], &c[d]);
        else if (m <= kHi078) sincos_range<2>(t[d], &s[d], &c[d]);
        else sincos_reduced(t[d], 0.0, &s[d], &c[d]);
    }
}

template <typename real> struct alignas(16) D4 { real a, b, c, d; };
template <typename real> struct alignas(2 * sizeof(real)) D2 { real a, b; };

// DiagCoef in the state precision (the Gauss coefficients of an FP32 state as
// double-float pairs), converted once on the host: conversions from FP64 in the
// kernel took a third of the FP64 pipe.
template <typename real> struct SiteCoef;
template <> struct SiteCoef<float> { float inv_dx2, v_coef, eel_coef, b_coef, sigma2; DF g_div, g_phi; };
struct SiteCoef64 : SiteCoef<float> {
    double g_div64, g_phi64, g_div_tiny, g_phi_tiny;       // FP64, and times 2^896
    bool tiny_ok;                                          // the latter two are finite
};
template <typename real, bool G64> struct PassCoef { using type = SiteCoef<real>; };
template <> struct PassCoef<float, true> { using type = SiteCoef64; };
struct D1 { double h; };
template <> struct SiteCoef<double> { double inv_dx2, v_coef, eel_coef, b_coef, sigma2; D1 g_div, g_phi; };
inline SiteCoef<float> site_coef(const DiagCoef &d, float)
{
    return { (float)d.inv_dx2, (float)d.v_coef, (float)d.eel_coef, (float)d.b_coef, (float)d.sigma2, df_from(d.g_div),
             df_from(d.g_phi) };
}
inline SiteCoef64 site_coef64(const DiagCoef &d)
{
    const double a = d.g_div * 0x1p896, b = d.g_phi * 0x1p896;
    return { site_coef(d, 0.f), d.g_div, d.g_phi, a, b, std::isfinite(a) && std::isfinite(b) };
}
inline SiteCoef<double> site_coef(const DiagCoef &d, double)
{
    return { d.inv_dx2, d.v_coef, d.eel_coef, d.b_coef, d.sigma2, { d.g_div }, { d.g_phi } };
}

struct DiagGeo {
    static constexpr int TX = 32, TY = 8, NT = 256, EX = TX + 2, NE = EX * (TY + 2);
    // two copies of: { phi.re, phi.im, theta_3, theta_2 }, { E_1, E_2 }, theta_1,
    // alpha, turns as seen from x - 1 and from x - y
    template <typename real> static constexpr int bytes = NE * (7 * (int)sizeof(real) + 12);
    template <typename real> static constexpr size_t smem = 2 * (size_t)((bytes<real> + 15) / 16 * 16);
};

// Gauss residual G and scale = |g_div div E| + |g_phi Im(conj(phi) Pi)| of FP32 fields in
// FP64.
struct GaussTerms64 {
    double g, scale;
    long long size;                      // the bits of |g|, 0 for NaN
};
__device__ __forceinline__ GaussTerms64 gauss_terms64(double g_div, double g_phi, double fr, double fi, double pr, double pi,
                                                      double e1, double e1b, double e2, double e2b, double e3, double e3b)
{
    const double div = (e1 - e1b) + (e2 - e2b) + (e3 - e3b);
    const double p = g_div * div, q = g_phi * (fr * pi - fi * pr), g = p + q;
    return { g, fabs(p) + fabs(q), isnan(g) ? 0 : __double_as_longlong(fabs(g)) };
}
// The same of finite fields (a, b: the products fr pi and fi pr, exact from 2^-100 on).
// An FP64 instruction costs as much as 30 others here, and so does a conversion from
// FP32; with 24 of them per site the 200^3 pass took 548 us, against 248 without.  So
// the bits of a float are moved to where a double has them, which gives its value
// times 2^-896 (zero and subnormal ones too) in three integer instructions, and the
// coefficients bring the factor back; |p| + |q| is the larger of |p + q| and |p - q|; and
// the largest |G| is found in integers: 13 FP64 instructions, 372 us.
__device__ __forceinline__ double tiny(float f)
{
    const int b = __float_as_int(f);
    return __hiloint2double((b >> 3) & (int)0x8fffffff, b << 29);
}
__device__ __forceinline__ GaussTerms64 gauss_terms64(const SiteCoef64 &sc, DF a, DF b, float e1, float e1b, float e2,
                                                      float e2b, float e3, float e3b)
{
    const double div = ((tiny(e1) - tiny(e1b)) + (tiny(e2) - tiny(e2b))) + (tiny(e3) - tiny(e3b));
    const double q = sc.g_phi_tiny * ((tiny(a.h) - tiny(b.h)) + (tiny(a.l) - tiny(b.l)));
    const double s = fma(sc.g_div_tiny, div, q), d = fma(sc.g_div_tiny, div, -q);
    const long long m = 0x7fffffffffffffffLL, sa = __double_as_longlong(s) & m, da = __double_as_longlong(d) & m;
    return { s, __longlong_as_double(max(sa, da)), sa };
}
// Gauss residual and its sums in FP64: of FP64 states, and of FP32 states in passes that
// ask for it (G64).
template <typename real, typename IT, bool G64 = sizeof(real) == 8>
struct DiagTile {
    using G = DiagGeo;
    using Coef = typename PassCoef<real, G64>::type;
    static constexpr int EX = G::EX, NE = G::NE;
    // sums 3..13 of ah_obs (compensated for FP32), Gauss sums and maxima, windings
    Acc<real> s[11];
    double dg2 = 0.0, dgs2 = 0.0, dgmax = 0.0;
    Acc<float> fg2, fgs2;
    DF fgmax{ 0.f, 0.f };
    real tmax = real(0);
    int ic[kNumInt] = { 0, 0, 0, 0, 0, 0, 0, 0 };

    // one column of tiles: planes [z0, z1) of the 32 x 8 sites at (x0, y0)
    __device__ __forceinline__ void column(const View<real> &v, int N, const DiagArgs &da, const Coef &sc, int x0,
                                           int y0, int z0, int z1, unsigned char *smem)
    {
        const int lx = threadIdx.x & 31, wy = threadIdx.x >> 5;
        const IT NN = (IT)N * (IT)N;
        const bool own = x0 + lx < N && y0 + wy < N;
        const int roff = wrapm(x0 + lx, N) + N * wrapm(y0 + wy, N);
        const int e = (wy + 1) * EX + lx + 1;
        // the ring: phi, theta of the row above (warp 7) and of the column to the
        // right with the corner between them (warp 3); E_2 of the row below (warp
        // 0), E_1 of the column to the left (warp 4)
        const bool above = wy == 7, right = wy == 3 && lx <= 8, fwd = above || right;
        const bool back = wy == 0 || (wy == 4 && lx < 8);
        const int rx = wy == 3 ? 32 : wy == 4 ? -1 : lx, ry = wy == 7 ? 8 : wy == 0 ? -1 : lx;
        const bool ring = fwd || back;
        const int hoff = wrapm(x0 + rx, N) + N * wrapm(y0 + ry, N);
        const int he = ring ? (ry + 1) * EX + rx + 1 : 0;
        const int half = (G::bytes<real> + 15) / 16 * 16;
        auto at4 = [&](int b) { return reinterpret_cast<D4<real> *>(smem + b * half); };
        auto at2 = [&](int b) { return reinterpret_cast<D2<real> *>(smem + b * half + NE * 4 * sizeof(real)); };
        auto atw = [&](int b) { return reinterpret_cast<uint2 *>(smem + b * half + NE * 6 * sizeof(real)); };
        auto at1 = [&](int b) { return reinterpret_cast<real *>(smem + b * half + NE * (6 * sizeof(real) + 8)); };
        auto atf = [&](int b) { return reinterpret_cast<float *>(smem + b * half + NE * (7 * sizeof(real) + 8)); };
        auto wrapz = [&](int z) { return (IT)(z < 0 ? z + N : (z >= N ? z - N : z)) * NN; };

        // fields of the next plane, momenta of the current one
        real nf[2], nt[3], rf[2], rt[3], pr, pim, e1, e2, e3, re = real(0);
        auto load_fields = [&](int z) {
            const IT a = wrapz(z) + (IT)roff;
            nf[0] = v.phr[a]; nf[1] = v.phi[a];
            nt[0] = v.th1[a]; nt[1] = v.th2[a]; nt[2] = v.th3[a];
            if (fwd) {
                const IT b = wrapz(z) + (IT)hoff;
                rf[0] = v.phr[b]; rf[1] = v.phi[b];
                rt[0] = v.th1[b]; rt[1] = v.th2[b]; rt[2] = v.th3[b];
            }
        };
        auto load_momenta = [&](int z) {
            const IT a = wrapz(z) + (IT)roff;
            pr = v.pir[a]; pim = v.pii[a];
            e1 = v.e1[a]; e2 = v.e2[a]; e3 = v.e3[a];
            if (back) re = wy == 0 ? v.e2[wrapz(z) + (IT)hoff] : v.e1[wrapz(z) + (IT)hoff];
        };
        real f0[2], t0[3], g0[3];
        float a0, ra;
        real e3m = v.e3[wrapz(z0 - 1) + (IT)roff];
        load_fields(z0);
        load_momenta(z0);
        a0 = site_phase(nf[0], nf[1]);
        ra = fwd ? site_phase(rf[0], rf[1]) : 0.f;
        unsigned wm = 0;                         // own turns and N of plane z - 1
        for (int z = z0; z <= z1; ++z) {
            const int b = z & 1;
            f0[0] = nf[0]; f0[1] = nf[1];
            t0[0] = nt[0]; t0[1] = nt[1]; t0[2] = nt[2];
            g0[0] = rt[0]; g0[1] = rt[1]; g0[2] = rt[2];
            at4(b)[e] = { f0[0], f0[1], t0[2], t0[1] };
            at2(b)[e] = { e1, e2 };
            at1(b)[e] = t0[0];
            atf(b)[e] = a0;
            if (fwd) {
                at4(b)[he] = { rf[0], rf[1], rt[2], rt[1] };
                at1(b)[he] = rt[0];
                atf(b)[he] = ra;
            }
            if (back) {
                if (wy == 0) at2(b)[he].b = re;
                else at2(b)[he].a = re;
            }
            const real mpr = pr, mpi = pim, m1 = e1, m2 = e2, m3 = e3;
            if (z < z1) load_fields(z + 1);
            __syncthreads();

            const D4<real> qx = at4(b)[e + 1], qy = at4(b)[e + EX];
            const real t1y = at1(b)[e + EX];
            const float ax = atf(b)[e + 1], ay = atf(b)[e + EX];
            const real e1x = at2(b)[e - 1].a, e2y = at2(b)[e - EX].b;
            if (z + 1 < z1) load_momenta(z + 1);
            const float an = z < z1 ? site_phase(nf[0], nf[1]) : 0.f;
            int n[3];
            int nc;
            {
                const float bn[3] = { ax, ay, an };
                nc = link_turns(a0, bn, t0, n);
                atw(b)[e] = make_uint2(x_word(n[1], n[2], nc), y_word(n[0], n[2], nc));
            }
            if (fwd) {
                // the row above: n_1, n_3; the column to the right: n_2, n_3
                const float rn = z < z1 ? site_phase(rf[0], rf[1]) : 0.f;
                const float aj = above ? atf(b)[he + 1] : (lx < 8 ? atf(b)[he + EX] : 0.f);
                const float bn[3] = { aj, aj, rn };
                int rk[3];
                const int rc = link_turns(ra, bn, g0, rk);
                atw(b)[he] = make_uint2(x_word(rk[1], rk[2], rc), y_word(rk[0], rk[2], rc));
                ra = rn;
            }
            // windings of plane z - 1 (Eq. 9): its neighbours' turns are in the other copy
            if (z > z0 && own) {
                const unsigned wx = atw(1 - b)[e + 1].x, wyv = atw(1 - b)[e + EX].y, wz = z_word(n, nc);
                const unsigned t = (0u - (wm + wx + wyv + wz)) & 0xffffffu, cuts = (wm | wx | wyv | wz) >> 24;
                if (t | cuts) {
                    int q[3];
                    windings(t, q);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (cuts >> k & 1u) {
                            const unsigned long long at =
                                (unsigned long long)((long long)(z - 1) * N * (long long)N + (long long)roff);
                            const unsigned long long i = atomicAdd(da.list.count, 1ULL);
                            if (i < (unsigned long long)da.list.capacity) da.list.items[i] = at * 4ULL + k;
                        } else {
                            ic[k] += abs(q[k]);
                            ic[3 + k] += q[k];
                            ic[6] += q[k] != 0;
                        }
                    }
                }
            }
            if (z == z1) break;
            // energies and the Gauss residual of plane z
            {
                const real ti[3] = { t0[0], t0[0], t0[1] }, tij[3] = { t1y, nt[0], nt[1] };
                const real tj[3] = { t0[1], t0[2], t0[2] }, tji[3] = { qx.d, qx.c, qy.c };
                unsigned wn;
                const real bsum = xi_terms(ti, tij, tj, tji, &wn);
                const unsigned wo = own_word(n, nc);
                wm = ((wo + wn) & 0xffffffu) | ((wo | wn) & 0x07000000u);
                real sn[3], co[3];
                diag_links(t0, sn, co);
                if (own) site(sc, f0, t0, sn, co, qx, qy, nf, bsum, mpr, mpi, m1, m2, m3, e1x, e2y, e3m);
            }
            e3m = m3;
            a0 = an;
        }
        __syncthreads();                         // the next column reuses the arrays
    }

    __device__ __forceinline__ void site(const Coef &sc, const real f0[2], const real t0[3],
                                         const real sn[3], const real co[3], const D4<real> &qx, const D4<real> &qy,
                                         const real nf[2], real bsum, real pr, real pim, real e1, real e2, real e3,
                                         real e1b, real e2b, real e3b)
    {
        const real fr[3] = { qx.a, qy.a, nf[0] }, fi[3] = { qx.b, qy.b, nf[1] };
        real g = real(0);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const real wr = co[d] * fr[d] - sn[d] * fi[d], wi = co[d] * fi[d] + sn[d] * fr[d];
            const real a = wr - f0[0], b = wi - f0[1];
            g += a * a + b * b;
        }
        const real K = pr * pr + pim * pim;
        const real G2 = g * sc.inv_dx2;
        const real m2 = f0[0] * f0[0] + f0[1] * f0[1] - sc.sigma2;
        const real V = sc.v_coef * m2 * m2;
        const real Eel = sc.eel_coef * (e1 * e1 + e2 * e2 + e3 * e3);
        const real B = sc.b_coef * bsum;
        const real L = K - G2 - V + Eel - B;
        const real rho = K + G2 + V + Eel + B;
        const real pp = K - G2 * real(1.0 / 3.0) - V + (Eel + B) * real(1.0 / 3.0);
        s[0].add(K); s[1].add(G2); s[2].add(V); s[3].add(Eel); s[4].add(B);
        s[5].add(K * V); s[6].add(G2 * V); s[7].add(K * L); s[8].add(G2 * L); s[9].add(pp * L); s[10].add(rho * L);
        tmax = fmax(tmax, fmax(fabs(t0[0]), fmax(fabs(t0[1]), fabs(t0[2]))));
        ic[7] += !(isfinite(L) && isfinite(rho) && isfinite(pp));
        if constexpr (sizeof(real) == 8) {
            const double div = (e1 - e1b) + (e2 - e2b) + (e3 - e3b);
            const double g1 = sc.g_div.h * div;
            const double g2 = sc.g_phi.h * (f0[0] * pim - f0[1] * pr);
            const double Gs = g1 + g2, gs = fabs(g1) + fabs(g2);
            dg2 += Gs * Gs;
            dgs2 += gs * gs;
            dgmax = fmax(dgmax, fabs(Gs));
        } else if constexpr (G64) {
            add(gauss_terms64(sc, two_prod(f0[0], pim), two_prod(f0[1], pr), e1, e1b, e2, e2b, e3, e3b));
        } else {
            const GaussTerms gt = gauss_terms(sc.g_div, sc.g_phi, f0[0], f0[1], pr, pim, e1, e1b, e2, e2b, e3, e3b);
            DF Gs = gt.g;
            if (Gs.h < 0.f) Gs = { -Gs.h, -Gs.l };
            const float gs = gt.scale;
            const float sg = Gs.h * 0x1p30f, ss = gs * 0x1p30f;
            fg2.add(sg * sg);
            fgs2.add(ss * ss);
            if (Gs.h > fgmax.h || (Gs.h == fgmax.h && Gs.l > fgmax.l)) fgmax = Gs;
        }
    }

    __device__ __forceinline__ void add(const GaussTerms64 &t)
    {
        dg2 += t.g * t.g;
        dgs2 += t.scale * t.scale;
        dgmax = __longlong_as_double(max(__double_as_longlong(dgmax), t.size));
    }

    // dg2, dgs2 and dgmax of a column again, with conversions: any fields
    __device__ __forceinline__ void gauss_again(const View<real> &v, int N, const Coef &sc, int x0, int y0, int rows,
                                                int z0, int z1)
    {
        const int x = x0 + (threadIdx.x & 31);
        const IT NN = (IT)N * (IT)N;
        for (int z = z0; z < z1; ++z) {
            for (int y = y0 + (threadIdx.x >> 5); y < min(y0 + rows, N) && x < N; y += 8) {
                const IT s = (IT)z * NN + (IT)(N * y + x), sx = x ? s - 1 : s + (N - 1), sy = y ? s - N : s + (NN - N);
                const IT sz = z ? s - NN : s + (NN * N - NN);
                add(gauss_terms64(sc.g_div64, sc.g_phi64, v.phr[s], v.phi[s], v.pir[s], v.pii[s], v.e1[s], v.e1[sx], v.e2[s],
                                  v.e2[sy], v.e3[s], v.e3[sz]));
            }
        }
    }

    __device__ __forceinline__ void flush(DiagPartial *out)
    {
        double accd[kNumSums];
#pragma unroll
        for (int k = 3; k < 14; ++k) accd[k] = s[k - 3].value();
        // the sums of L, rho and p are linear in those of K, G2, V, E_el, B
        accd[0] = accd[3] - accd[4] - accd[5] + accd[6] - accd[7];
        accd[1] = accd[3] + accd[4] + accd[5] + accd[6] + accd[7];
        accd[2] = accd[3] - accd[4] * (1.0 / 3.0) - accd[5] + (accd[6] + accd[7]) * (1.0 / 3.0);
        if constexpr (!G64) {
            dg2 = fg2.value() * 0x1p-60;
            dgs2 = fgs2.value() * 0x1p-60;
            dgmax = (double)fgmax.h + (double)fgmax.l;
        }
        accd[14] = dg2;
        accd[15] = dgs2;
        double mx[kNumMax] = { dgmax, (double)tmax };
        long long il[kNumInt];
#pragma unroll
        for (int k = 0; k < kNumInt; ++k) il[k] = ic[k];
        block_reduce<256>(accd, mx, il, out);
    }
};

}  // namespace
}  // namespace ah
