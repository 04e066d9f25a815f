// diag_pair.cuh -- the FP32 whole-lattice diagnostics of diag_tile.cuh, two rows per
// thread from planes copied ahead (as the step of feed_tile.cuh).
//
// The pass is bound by instruction issue: energies, compensated sums, the
// double-float Gauss residual and the winding turns of a site take 660
// instructions one site at a time.  Two rows share every packed instruction, and the
// fields of the next plane come by cp.async instead of through registers.  A CTA of
// 256 threads takes 32 x 16 columns of sites.  phi, theta and E come as rows of 40
// floats (16 own rows and one on either side), Pi as rows of 32; one barrier per plane.
// A pass takes 2.80 ms at 512^3 and 0.375 ms at 256^3, 21 ps per site, where the one-row
// walk takes 29 (381^3).
#pragma once
#include "diag_tile.cuh"
#include "feed_tile.cuh"

namespace ah {
namespace {

// packed forms of diag_common.cuh's double-float helpers: the same bits per element
struct DF2 { float2 h, l; };
__device__ __forceinline__ DF2 two_sum2(float2 a, float2 b)
{
    const float2 s = ad(a, b), bb = sb(s, a);
    return { s, ad(sb(a, sb(s, bb)), sb(b, bb)) };
}
__device__ __forceinline__ DF2 two_diff2(float2 a, float2 b)      // two_sum(a, -b)
{
    const float2 s = sb(a, b), bb = sb(s, a), nb = ng(b);
    return { s, ad(sb(a, sb(s, bb)), sb(nb, bb)) };
}
__device__ __forceinline__ DF2 two_prod2(float2 a, float2 b)
{
    const float2 p = ml(a, b);
    return { p, fm(a, b, ng(p)) };
}
__device__ __forceinline__ DF2 df_add2(DF2 a, DF2 b)
{
    const DF2 s = two_sum2(a.h, b.h);
    return two_sum2(s.h, ad(s.l, ad(a.l, b.l)));
}
__device__ __forceinline__ DF2 df_sub2(DF2 a, DF2 b)              // df_add(a, -b)
{
    const DF2 s = two_diff2(a.h, b.h);
    return two_sum2(s.h, ad(s.l, sb(a.l, b.l)));
}
__device__ __forceinline__ DF2 df_mul2(DF a, DF2 b)
{
    const DF2 p = two_prod2(pk(a.h), b.h);
    const float2 t = ad(p.l, fm(pk(a.h), b.l, ml(pk(a.l), b.h))), h = ad(p.h, t);
    return { h, sb(t, sb(h, p.h)) };
}
struct GaussTerms2 { DF2 g; float2 scale; };
__device__ __forceinline__ float2 abs2(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ GaussTerms2 gauss_terms2(DF g_div, DF g_phi, float2 fr, float2 fi, float2 pr, float2 pi,
                                                    float2 e1, float2 e1b, float2 e2, float2 e2b, float2 e3,
                                                    float2 e3b)
{
    const DF2 div = df_add2(df_add2(two_diff2(e1, e1b), two_diff2(e2, e2b)), two_diff2(e3, e3b));
    const DF2 p = df_mul2(g_div, div), q = df_mul2(g_phi, df_sub2(two_prod2(fr, pi), two_prod2(fi, pr)));
    return { df_add2(p, q), ad(abs2(p.h), abs2(q.h)) };
}

// site_phase of both sites
__device__ __forceinline__ float2 site_phase2(float2 r, float2 i)
{
    const float2 x = abs2(r), y = abs2(i);
    const float2 hi = make_float2(fmaxf(x.x, y.x), fmaxf(x.y, y.y)), lo = make_float2(fminf(x.x, y.x), fminf(x.y, y.y));
    const float2 q = make_float2(__fdividef(lo.x, hi.x), __fdividef(lo.y, hi.y)), u = ml(q, q);
    float2 p = fm(u, pk(7.648353930562735e-03f), pk(-3.636043146252632e-02f));
    p = fm(u, p, pk(8.312645554542542e-02f));
    p = fm(u, p, pk(-1.344786435365677e-01f));
    p = fm(u, p, pk(1.9872039556503296e-01f));
    p = fm(u, p, pk(-3.332567811012268e-01f));
    p = fm(u, p, pk(9.999992251396179e-01f));
    const float2 a = ml(q, p);
    auto octant = [](float a, float r, float i, float x, float y, float hi) {
        a = y > x ? 0.5f * kPi32 - a : a;
        a = r < 0.f ? kPi32 - a : a;
        a = i < 0.f ? -a : a;
        return hi > 1e-30f && x + y < 1e30f ? a : __int_as_float(0x7fc00000);
    };
    return make_float2(octant(a.x, r.x, i.x, x.x, y.x, hi.x), octant(a.y, r.y, i.y, x.y, y.y, hi.y));
}

// link_turns of both sites: n[d][row]; the cut bits of row 0, and of row 1 shifted by 3
__device__ __forceinline__ int link_turns2(float2 a, const float2 b[3], const float2 t[3], int n[3][2])
{
    const float m = fmaxf(amax2(t[0]), fmaxf(amax2(t[1]), amax2(t[2])));
    if (__all_sync(__activemask(), m <= 8.f)) {
        bool any = false;
        float2 f[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float2 v = ad(sb(b[d], a), t[d]);
            const float2 kb = fm(v, pk(kInvTwoPi32), pk(kRound)), k = ad(kb, pk(-kRound));
            f[d] = fm(k, pk(-kTwoPi32), v);
            any = any || !(fabsf(f[d].x) <= kPi32 - kCutMargin) || !(fabsf(f[d].y) <= kPi32 - kCutMargin);
            n[d][0] = __float_as_int(kb.x) - kRoundBits;
            n[d][1] = __float_as_int(kb.y) - kRoundBits;
        }
        if (!__any_sync(__activemask(), any)) return 0;
        int cuts = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const bool c0 = !(fabsf(f[d].x) <= kPi32 - kCutMargin), c1 = !(fabsf(f[d].y) <= kPi32 - kCutMargin);
            cuts |= (int)c0 << d | (int)c1 << (3 + d);
            n[d][0] = c0 ? 0 : n[d][0];
            n[d][1] = c1 ? 0 : n[d][1];
        }
        return cuts;
    }
    const float b0[3] = { b[0].x, b[1].x, b[2].x }, b1[3] = { b[0].y, b[1].y, b[2].y };
    const float t0[3] = { t[0].x, t[1].x, t[2].x }, t1[3] = { t[0].y, t[1].y, t[2].y };
    int k0[3], k1[3];
    const int c0 = link_turns(a.x, b0, t0, k0), c1 = link_turns(a.y, b1, t1, k1);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        n[d][0] = k0[d];
        n[d][1] = k1[d];
    }
    return c0 | c1 << 3;
}

// xi_terms of both sites
__device__ __forceinline__ float2 xi_terms2(const float2 *ti, const float2 *tij, const float2 *tj, const float2 *tji,
                                            unsigned word[2])
{
    float2 x[3], sum = pk(0.f);
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 a = sb(ti[k], tij[k]);
        x[k] = ad(a, sb(tji[k], tj[k]));
        m = fmaxf(fmaxf(m, amax2(a)), amax2(x[k]));
    }
    word[0] = word[1] = 0;
    if (__all_sync(__activemask(), m <= 0.78f)) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 u = ml(x[k], x[k]);
            float2 p = fm(u, pk(-2.480158764e-05f), pk(1.388888923e-03f));
            p = fm(u, p, pk(-4.166666791e-02f));
            sum = fm(u, fm(u, p, pk(0.5f)), sum);
        }
        return sum;
    }
    float s[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float a[3], b[3], c[3], d[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a[k] = r ? ti[k].y : ti[k].x;
            b[k] = r ? tij[k].y : tij[k].x;
            c[k] = r ? tj[k].y : tj[k].x;
            d[k] = r ? tji[k].y : tji[k].x;
        }
        s[r] = xi_terms(a, b, c, d, &word[r]);
    }
    return make_float2(s[0], s[1]);
}

struct DiagPairGeo {
    static constexpr int NP = 8, TY = 16, NT = 256, W = 40, RW = 4 * W;
    static constexpr int array = RW * (TY + 2);                // one field of a plane: [TY + 2 rows][W]
    static constexpr int raw_plane = 5 * array, el_plane = 3 * array, pi_array = 128 * TY, pi_plane = 2 * pi_array;
    // phi, theta of three planes, E and Pi of two; alpha and the packed turns in two
    // copies: rows 0 .. TY, columns 0 .. 32
    static constexpr int off_el = 3 * raw_plane, off_pi = off_el + 2 * el_plane, NE = 33 * (TY + 1);
    static constexpr int off_w = off_pi + 2 * pi_plane, off_a = off_w + 2 * 8 * NE;
    static constexpr size_t smem = off_a + 2 * 4 * NE;
};

template <typename IT, bool G64>
struct DiagPair : DiagTile<float, IT, G64> {
    using G = DiagPairGeo;
    using Base = DiagTile<float, IT, G64>;

    // planes [z0, z1) of the 32 x 16 sites at (x0, y0)
    __device__ __forceinline__ void column(const View<float> &v, int N, const DiagArgs &da, const typename Base::Coef &sc,
                                           int x0, int y0, int z0, int z1, unsigned char *smem)
    {
        const int lx = threadIdx.x & 31, wp = threadIdx.x >> 5;
        const IT NN = (IT)N * (IT)N;
        const bool own0 = x0 + lx < N && y0 + 2 * wp < N, own1 = x0 + lx < N && y0 + 2 * wp + 1 < N;
        // copies: 16 bytes of a row of phi, theta, E (10 per row) and of Pi (8 per row,
        // the second half of the threads takes Pi_i)
        const bool raw_copy = threadIdx.x < 10 * (G::TY + 2), second = wp >= G::NP / 2;
        int raw_src = 0, pi_src;
        unsigned raw_dst, pi_dst;
        {
            const unsigned sbase = (unsigned)__cvta_generic_to_shared(smem);
            const int row = threadIdx.x / 10, c4 = 4 * (threadIdx.x % 10);
            if (raw_copy) raw_src = wrapm(x0 - 4 + c4, N) + N * wrapm(y0 - 1 + row, N);
            raw_dst = sbase + row * G::RW + 4 * c4;
            const int q = threadIdx.x % 128, mrow = q / 8, mc4 = 4 * (q % 8);
            pi_src = x0 + mc4 < N ? x0 + mc4 + N * wrapm(y0 + mrow, N) : -1;
            pi_dst = sbase + G::off_pi + (second ? G::pi_array : 0) + mrow * 128 + 4 * mc4;
        }
        auto plane_of = [&](int z) { return (IT)(z < 0 ? z + N : (z >= N ? z - N : z)) * NN; };
        auto copy_raw = [&](int z, int off) {
            if (raw_copy) {
                const IT s = plane_of(z) + (IT)raw_src;
                const unsigned d = raw_dst + off;
                feed_copy(d, v.phr + s);
                feed_copy(d + G::array, v.phi + s);
                feed_copy(d + 2 * G::array, v.th1 + s);
                feed_copy(d + 3 * G::array, v.th2 + s);
                feed_copy(d + 4 * G::array, v.th3 + s);
            }
        };
        auto copy_mom = [&](int z, int m) {
            const IT b = plane_of(z);
            if (raw_copy) {
                const IT s = b + (IT)raw_src;
                const unsigned d = raw_dst + G::off_el + m * G::el_plane;
                feed_copy(d, v.e1 + s);
                feed_copy(d + G::array, v.e2 + s);
                feed_copy(d + 2 * G::array, v.e3 + s);
            }
            if (pi_src >= 0) feed_copy(pi_dst + m * G::pi_plane, (second ? v.pii : v.pir) + b + (IT)pi_src);
        };
        auto commit = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };
        // value of field k at row (from own row 2p) and column of the slot at `off`
        unsigned char *const own = smem + (2 * wp + 1) * G::RW + 4 * (lx + 4);
        auto raw = [&](int off, int k, int row, int col) -> float {
            return *reinterpret_cast<const float *>(own + off + k * G::array + row * G::RW + 4 * col);
        };
        auto raw2 = [&](int off, int k, int col) { return make_float2(raw(off, k, 0, col), raw(off, k, 1, col)); };
        // exchanged values at (row, column), own at e and e + 33
        const int e = 2 * wp * 33 + lx;
        auto al = [&](int k) { return reinterpret_cast<float *>(smem + G::off_a + (k & 1) * 4 * G::NE); };
        auto tw = [&](int k) { return reinterpret_cast<uint2 *>(smem + G::off_w + (k & 1) * 8 * G::NE); };
        // the ring: the row above (warp 7), the column to the right and the corner
        // between them (warp 3, one lane per row)
        const bool above = wp == 7, ring = above || (wp == 3 && lx <= G::TY);
        const int rrow = above ? G::TY : lx, rcol = above ? lx : 32, he = rrow * 33 + rcol;
        unsigned char *const hown = smem + (rrow + 1) * G::RW + 4 * (rcol + 4);
        auto hraw = [&](int off, int k) { return *reinterpret_cast<const float *>(hown + off + k * G::array); };

        int ra = 0, rb = G::raw_plane, rc = 2 * G::raw_plane;       // planes z - 1 (next copied to), z, z + 1
        copy_raw(z0, rb);
        copy_mom(z0, 0);
        commit();
        copy_raw(z0 + 1, rc);
        commit();
        float2 e3m;
        {
            const IT a = plane_of(z0 - 1) + (IT)wrapm(x0 + lx, N);
            e3m = make_float2(v.e3[a + (IT)N * wrapm(y0 + 2 * wp, N)], v.e3[a + (IT)N * wrapm(y0 + 2 * wp + 1, N)]);
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        float2 f0r = raw2(rb, 0, 0), f0i = raw2(rb, 1, 0), t0[3] = { raw2(rb, 2, 0), raw2(rb, 3, 0), raw2(rb, 4, 0) };
        float2 a0 = site_phase2(f0r, f0i);
        float ha = ring ? site_phase(hraw(rb, 0), hraw(rb, 1)) : 0.f;
        al(0)[e] = a0.x;
        al(0)[e + 33] = a0.y;
        if (ring) al(0)[he] = ha;
        unsigned wm0 = 0, wm1 = 0;               // own turns and N of plane z - 1
        for (int z = z0, m = 0;; ++z, m ^= 1) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            if (z < z1 && z + 1 <= z1) {
                if (z + 2 <= z1) copy_raw(z + 2, ra);
                if (z + 1 < z1) copy_mom(z + 1, m ^ 1);
            }
            commit();
            // phases of plane z + 1, turns of plane z
            const float2 fnr = raw2(rc, 0, 0), fni = raw2(rc, 1, 0);
            const bool last = z == z1;           // only n_1, n_2 of this plane are wanted
            const float2 an = last ? pk(0.f) : site_phase2(fnr, fni);
            const float *A = al(m);
            int n[3][2];
            int nc;
            {
                const float ay = A[e + 66];
                const float2 bn[3] = { make_float2(A[e + 1], A[e + 34]), make_float2(a0.y, ay), an };
                nc = link_turns2(a0, bn, t0, n);
            }
            const int n0[3] = { n[0][0], n[1][0], n[2][0] }, n1[3] = { n[0][1], n[1][1], n[2][1] };
            uint2 *const T = tw(m);
            const unsigned y0w = y_word(n0[0], n0[2], nc & 7);
            T[e] = make_uint2(x_word(n0[1], n0[2], nc & 7), y0w);
            const unsigned y1w = y_word(n1[0], n1[2], nc >> 3);
            T[e + 33] = make_uint2(x_word(n1[1], n1[2], nc >> 3), y1w);
            float hn = 0.f;
            if (ring) {
                // the row above: n_1, n_3; the column to the right: n_2, n_3
                hn = last ? 0.f : site_phase(hraw(rc, 0), hraw(rc, 1));
                const float aj = above ? A[he + 1] : (lx < G::TY ? A[he + 33] : 0.f);
                const float bn[3] = { aj, aj, hn }, tf[3] = { hraw(rb, 2), hraw(rb, 3), hraw(rb, 4) };
                int rk[3];
                const int rcut = link_turns(ha, bn, tf, rk);
                T[he] = make_uint2(x_word(rk[1], rk[2], rcut), y_word(rk[0], rk[2], rcut));
                ha = hn;
            }
            // windings of plane z - 1 (Eq. 9): its neighbours' turns are in the other copy
            if (z > z0) {
                const uint2 *U = tw(m ^ 1);
                auto count = [&](unsigned wm, unsigned wx, unsigned wy, unsigned wz, int row) {
                    const unsigned t = (0u - (wm + wx + wy + wz)) & 0xffffffu, cuts = (wm | wx | wy | wz) >> 24;
                    if (t | cuts) {
                        int q[3];
                        windings(t, q);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            if (cuts >> k & 1u) {
                                const unsigned long long at =
                                    (unsigned long long)((long long)(z - 1) * N * (long long)N +
                                                         (long long)N * (y0 + 2 * wp + row) + x0 + lx);
                                const unsigned long long i = atomicAdd(da.list.count, 1ULL);
                                if (i < (unsigned long long)da.list.capacity) da.list.items[i] = at * 4ULL + k;
                            } else {
                                this->ic[k] += abs(q[k]);
                                this->ic[3 + k] += q[k];
                                this->ic[6] += q[k] != 0;
                            }
                        }
                    }
                };
                if (own0) count(wm0, U[e + 1].x, U[e + 33].y, z_word(n0, nc & 7), 0);
                if (own1) count(wm1, U[e + 34].x, U[e + 66].y, z_word(n1, nc >> 3), 1);
            }
            if (last) break;
            // energies and the Gauss residual of plane z
            {
                const float2 tn[2] = { raw2(rc, 2, 0), raw2(rc, 3, 0) };
                const float2 t3y = make_float2(t0[2].y, raw(rb, 4, 2, 0));
                const float2 ti[3] = { t0[0], t0[0], t0[1] };
                const float2 tij[3] = { make_float2(t0[0].y, raw(rb, 2, 2, 0)), tn[0], tn[1] };
                const float2 tj[3] = { t0[1], t0[2], t0[2] };
                const float2 tji[3] = { raw2(rb, 3, 1), raw2(rb, 4, 1), t3y };
                unsigned wn[2];
                const float2 bsum = xi_terms2(ti, tij, tj, tji, wn);
                const unsigned w0 = own_word(n0, nc & 7), w1 = own_word(n1, nc >> 3);
                wm0 = ((w0 + wn[0]) & 0xffffffu) | ((w0 | wn[0]) & 0x07000000u);
                wm1 = ((w1 + wn[1]) & 0xffffffu) | ((w1 | wn[1]) & 0x07000000u);
                U22 u[3];
                link_exps2<3>(t0, u);
                const C22 fx = { raw2(rb, 0, 1), raw2(rb, 1, 1) };
                const C22 fy = { make_float2(f0r.y, raw(rb, 0, 2, 0)), make_float2(f0i.y, raw(rb, 1, 2, 0)) };
                const C22 w1c = fwd(u[0], fx), w2c = fwd(u[1], fy), w3c = fwd(u[2], C22{ fnr, fni });
                float2 d = sb(w1c.r, f0r), g = ml(d, d);
                d = sb(w1c.i, f0i); g = fm(d, d, g);
                d = sb(w2c.r, f0r); g = fm(d, d, g);
                d = sb(w2c.i, f0i); g = fm(d, d, g);
                d = sb(w3c.r, f0r); g = fm(d, d, g);
                d = sb(w3c.i, f0i); g = fm(d, d, g);
                const float *P = reinterpret_cast<const float *>(smem + G::off_pi + m * G::pi_plane) + 64 * wp + lx;
                const float2 pr = make_float2(P[0], P[32]), pim = make_float2(P[G::pi_array / 4], P[G::pi_array / 4 + 32]);
                const int el = G::off_el + m * G::el_plane;
                const float2 e1 = raw2(el, 0, 0), e2 = raw2(el, 1, 0), e3 = raw2(el, 2, 0);
                const float2 e1b = raw2(el, 0, -1), e2b = make_float2(raw(el, 1, -1, 0), e2.x);
                const float2 K = fm(pr, pr, ml(pim, pim));
                const float2 G2 = ml(g, pk(sc.inv_dx2));
                const float2 m2 = ad(fm(f0r, f0r, ml(f0i, f0i)), pk(-sc.sigma2));
                const float2 V = ml(ml(pk(sc.v_coef), m2), m2);
                const float2 Eel = ml(pk(sc.eel_coef), fm(e1, e1, fm(e2, e2, ml(e3, e3))));
                const float2 B = ml(pk(sc.b_coef), bsum);
                const float2 EB = ad(Eel, B), KV_ = sb(K, V);
                const float2 L = sb(ad(sb(KV_, G2), Eel), B);
                const float2 rho = ad(ad(ad(K, G2), V), EB);
                const float2 pp = fm(EB, pk(1.0f / 3.0f), fm(G2, pk(-1.0f / 3.0f), KV_));
                [[maybe_unused]] GaussTerms2 gt;
                [[maybe_unused]] GaussTerms64 ga, gb;
                if constexpr (G64) {
                    const DF2 a = two_prod2(f0r, pim), b = two_prod2(f0i, pr);
                    ga = gauss_terms64(sc, { a.h.x, a.l.x }, { b.h.x, b.l.x }, e1.x, e1b.x, e2.x, e2b.x, e3.x, e3m.x);
                    gb = gauss_terms64(sc, { a.h.y, a.l.y }, { b.h.y, b.l.y }, e1.y, e1b.y, e2.y, e2b.y, e3.y, e3m.y);
                } else {
                    gt = gauss_terms2(sc.g_div, sc.g_phi, f0r, f0i, pr, pim, e1, e1b, e2, e2b, e3, e3m);
                }
                constexpr int sums = G64 ? 11 : 13;
                float2 val[13] = { K, G2, V, Eel, B, ml(K, V), ml(G2, V), ml(K, L), ml(G2, L), ml(pp, L), ml(rho, L) };
                if constexpr (!G64) {
                    const float2 sg = ml(gt.g.h, pk(0x1p30f)), ss = ml(gt.scale, pk(0x1p30f));
                    val[11] = ml(sg, sg);
                    val[12] = ml(ss, ss);
                }
                auto biggest = [&](float h, float l) {
                    if (h < 0.f) { h = -h; l = -l; }
                    if (h > this->fgmax.h || (h == this->fgmax.h && l > this->fgmax.l)) this->fgmax = { h, l };
                };
                auto sum = [&](int k, float x) {
                    if (k < 11) this->s[k].add(x);
                    else if (k == 11) this->fg2.add(x);
                    else this->fgs2.add(x);
                };
                // every term of rho is >= 0, and |L|, |p| <= rho: they are finite if it is
                if (own0) {
                    this->ic[7] += !isfinite(rho.x);
                    if constexpr (G64)
                        this->add(ga);
                    else
                        biggest(gt.g.h.x, gt.g.l.x);
                    this->tmax = fmaxf(this->tmax, fmaxf(fabsf(t0[0].x), fmaxf(fabsf(t0[1].x), fabsf(t0[2].x))));
                    if (own1) {
                        this->ic[7] += !isfinite(rho.y);
                        if constexpr (G64)
                            this->add(gb);
                        else
                            biggest(gt.g.h.y, gt.g.l.y);
                        this->tmax = fmaxf(this->tmax, fmaxf(fabsf(t0[0].y), fmaxf(fabsf(t0[1].y), fabsf(t0[2].y))));
#pragma unroll
                        for (int k = 0; k < sums; ++k) {
                            // one after the other, compensated each: their plain sum would
                            // round (and save 1.5 % of the pass, 512^3 2.86 -> 2.82 ms)
                            sum(k, val[k].x);
                            sum(k, val[k].y);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < sums; ++k) sum(k, val[k].x);
                    }
                }
                e3m = e3;
                t0[0] = tn[0];
                t0[1] = tn[1];
                t0[2] = raw2(rc, 4, 0);
            }
            f0r = fnr;
            f0i = fni;
            a0 = an;
            float *const An = al(m ^ 1);
            An[e] = a0.x;
            An[e + 33] = a0.y;
            if (ring) An[he] = ha;
            const int t = ra;
            ra = rb;
            rb = rc;
            rc = t;
        }
        __syncthreads();                         // the next column reuses the arrays
    }
};

}  // namespace
}  // namespace ah
