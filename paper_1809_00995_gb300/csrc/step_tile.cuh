// step_tile.cuh -- one leapfrog step on a tile of the lattice, marched in z.
//
// A CTA of 32 x TY threads owns a 32 x TY column of sites in the XY plane and a
// chunk of z planes; a thread owns one site of each plane.  What a site needs
// of its neighbours goes through shared memory in the form in which the
// neighbour already has it:
//   phi^{x+1}, phi^{x+y}                        forward products U_d phi^{x+d};
//   U_1, phi of x - 1 and U_2, phi of x - y     backward products conj(U) phi;
//   theta_2, theta_3 of x + 1, theta_1, theta_3 of x + y   plaquette phases;
//   sin Xi_12, sin Xi_13 of x - 1, sin Xi_12, sin Xi_23 of x - y   curls.
// Plane z + 1 is in the thread's own registers (its loads are issued one plane
// ahead) and of plane z - 1 only U_3, phi and two sines are kept there.  One
// buffer serves all planes, with two barriers per plane:
//   B  (after the fields of plane z are in place)  plaquette sines to shared
//      memory; Laplacian, Pi kick and phi drift, stored;
//   C  (after the sines)  curls, E kick and theta drift, stored; then the fields
//      of plane z + 1 into the buffer that B has done with.
// The halo ring needs link exponentials only where a link points into the tile
// (theta_2 of the row below, theta_1 of the column to the left); the row above
// and the column to the right are copies.
//
// What bounds it is the FP64 pipe, at 85 % of which nothing else matters: hence
// links instead of backward products in the buffer (a product costs four FP64
// instructions, its accumulation from link and field four as well, and the two
// adds that it would need after that are saved), and nothing of plane z0 - 1 but
// U_3 in the prologue.  One step at 256^3: 6.84 ms with plaquettes from products
// of link exponentials, 5.4 ms with phases, 5.14 ms with links exchanged;
// 128^3 0.665 ms, 64^3 0.113 ms.
#pragma once
#include "fused_common.cuh"
#include "site_math.cuh"

namespace ah {
namespace {

template <typename real, int TY>
struct TileGeo {
    static constexpr int TX = 32, NT = 32 * TY;
    static constexpr int EX = TX + 2, EY = TY + 2, NE = EX * EY;     // the tile and its ring
    // per site { phi.re, phi.im, theta_3, theta_2 }, then arrays of pairs (one
    // address register serves them all): U_1, U_2,
    // { sin 12, sin 13 }, { sin 12, sin 23 }, theta_1 (first of its pair)
    static constexpr size_t off_pairs = sizeof(V4<real>) * NE, stride = sizeof(V2<real>) * NE;
    static constexpr size_t smem = off_pairs + 5 * stride;
    static_assert(TY >= 6 && TY < 32, "a column of the ring and a corner are one warp's lanes");
};
// One site's place in those arrays.
template <typename real, int TY>
struct TileSite {
    using G = TileGeo<real, TY>;
    unsigned char *q, *p;
    __device__ __forceinline__ TileSite(unsigned char *smem, int e)
        : q(smem + e * (int)sizeof(V4<real>)), p(smem + G::off_pairs + e * (int)sizeof(V2<real>)) {}
    __device__ __forceinline__ V4<real> &field(int d = 0) const { return *(reinterpret_cast<V4<real> *>(q) + d); }
    __device__ __forceinline__ V2<real> &pair(int k, int d = 0) const
    {
        return *(reinterpret_cast<V2<real> *>(p + k * G::stride) + d);
    }
    __device__ __forceinline__ V2<real> &u1(int d = 0) const { return pair(0, d); }
    __device__ __forceinline__ V2<real> &u2(int d = 0) const { return pair(1, d); }
    __device__ __forceinline__ V2<real> &s1(int d = 0) const { return pair(2, d); }
    __device__ __forceinline__ V2<real> &s2(int d = 0) const { return pair(3, d); }
    __device__ __forceinline__ real &th1(int d = 0) const { return pair(4, d).r; }
};

// What a thread does for the ring: its site there (in-plane offset, index in the
// tile), whether it has one, and whether a link of that site points into the
// tile (low: row below, column to the left).  The row below is warp 0's, the
// row above warp TY - 1's, the columns, each with a corner, warp 3's and warp 4's.
struct RingTask { int off, e; bool has, low, below; };
template <int TY>
__device__ __forceinline__ RingTask ring_task(int lx, int wy, int x0, int y0, int N)
{
    constexpr int EX = 34;
    int ex = 0, ey = 0;
    RingTask t;
    t.below = wy == 0;
    t.has = wy == 0 || wy == TY - 1;
    t.low = wy == 0;
    if (wy == 0) { ex = lx + 1; ey = 0; }
    else if (wy == TY - 1) { ex = lx + 1; ey = TY + 1; }
    else if (wy == 3 || wy == 4) {
        t.has = lx <= TY;
        t.low = wy == 3 && lx < TY;
        ex = wy == 3 ? 0 : EX - 1;
        ey = wy == 3 ? (lx < TY ? lx + 1 : TY + 1) : (lx < TY ? lx + 1 : 0);
    }
    t.off = wrapm(x0 + ex - 1, N) + N * wrapm(y0 + ey - 1, N);
    t.e = ey * EX + ex;
    return t;
}

// IT: site-index type (int when N^3 < 2^31, so a field address is one
// 32 x 32 -> 64-bit multiply-add; long long otherwise).
template <typename real, int TY, typename IT>
__device__ __forceinline__ void step_tile(const View<real> &v, int N, int zc, const KickCoef<real> &c, int bx, int by,
                                          int bz, unsigned char *smem_raw)
{
    using G = TileGeo<real, TY>;
    using C = V2<real>;
    constexpr int EX = G::EX;

    const int lx = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int x0 = bx * 32, y0 = by * TY, z0 = bz * zc;
    if (z0 >= N) return;
    const int z1 = min(z0 + zc, N);
    const bool wr = x0 + lx < N && y0 + wy < N;
    const IT plane = (IT)N * (IT)N;
    const IT roff = (IT)(wrapm(x0 + lx, N) + N * wrapm(y0 + wy, N));
    const TileSite<real, TY> S(smem_raw, (wy + 1) * EX + lx + 1);
    const RingTask h = ring_task<TY>(lx, wy, x0, y0, N);
    const TileSite<real, TY> R(smem_raw, h.e);
    const IT hoff = (IT)h.off;

    auto field_of = [](const V4<real> &q) { return C{ q.a, q.b }; };
    // fields of the next plane: own site and ring site
    C fn, hf;
    real tn[3], ht[3];
    auto load_plane = [&](IT base) {
        const IT s = base + roff;
        fn = { v.phr[s], v.phi[s] };
        tn[0] = v.th1[s]; tn[1] = v.th2[s]; tn[2] = v.th3[s];
        if (h.has) {
            const IT r = base + hoff;
            hf = { v.phr[r], v.phi[r] };
            ht[0] = v.th1[r]; ht[1] = v.th2[r]; ht[2] = v.th3[r];
        }
    };
    // the plane that becomes the current one: its fields into shared memory, then
    // the link exponentials
    C f0, u[3];
    real t0[3];
    auto put_fields = [&]() {
        f0 = fn;
        t0[0] = tn[0]; t0[1] = tn[1]; t0[2] = tn[2];
        S.field() = { f0.r, f0.i, t0[2], t0[1] };
        S.th1() = t0[0];
        if (h.has) {
            R.field() = { hf.r, hf.i, ht[2], ht[1] };
            R.th1() = ht[0];
        }
    };
    auto put_ring_link = [&]() {
        if (h.low) {
            const real t = h.below ? ht[1] : ht[0];
            C w;
            link_exps<1>(&t, &w);
            (h.below ? R.u2() : R.u1()) = w;
        }
    };
    auto put_links = [&]() {
        link_exps<3>(t0, u);
        S.u1() = u[0];
        S.u2() = u[1];
    };

    // prologue: of plane z0 - 1 only U_3, phi and the sines of the two plaquettes
    // that reach into plane z0 (whose votes are over fewer phases than the loop's: the
    // last bits of a plane depend on where the chunks begin, which N and the GPU decide)
    C um, fb;
    real p13m, p23m;
    load_plane((IT)(z0 == 0 ? N - 1 : z0 - 1) * plane);
    put_fields();
    link_exps<1>(&t0[2], &um);
    fb = f0;
    IT o0 = (IT)z0 * plane;                                   // planes z, z + 1, z + 2
    IT o1 = z0 + 1 == N ? 0 : o0 + plane;
    load_plane(o0);
    __syncthreads();
    {
        const real ti[2] = { t0[0], t0[1] }, tij[2] = { tn[0], tn[1] }, tj[2] = { t0[2], t0[2] };
        const real tji[2] = { S.field(1).c, S.field(EX).c };
        real p[2];
        plaq_sines<2>(ti, tij, tj, tji, p);
        p13m = p[0];
        p23m = p[1];
    }
    __syncthreads();
    put_fields();
    put_ring_link();
    real pr, pim, e1, e2, e3;
    auto load_momenta = [&](IT base) {
        const IT s = base + roff;
        pr = v.pir[s]; pim = v.pii[s];
        e1 = v.e1[s]; e2 = v.e2[s]; e3 = v.e3[s];
    };
    load_plane(o1);
    load_momenta(o0);
    put_links();

    for (int z = z0;; ++z) {
        IT o2 = o1 + plane;
        if (z + 2 == N) o2 = 0;
        __syncthreads();
        // B: plaquette sines of plane z, own and on the ring's low sides
        const V4<real> qx = S.field(1), qy = S.field(EX);
        real p[3];
        {
            const real ti[3] = { t0[0], t0[0], t0[1] }, tij[3] = { S.th1(EX), tn[0], tn[1] };
            const real tj[3] = { t0[1], t0[2], t0[2] }, tji[3] = { qx.d, qx.c, qy.c };
            plaq_sines<3>(ti, tij, tj, tji, p);
            S.s1() = { p[0], p[1] };
            S.s2() = { p[0], p[2] };
        }
        if (h.low) {
            // (12) and, below, (23), to the left, (13)
            const V4<real> a0 = R.field(), ai = R.field(1), aj = R.field(EX);
            const real h1 = R.th1();
            const real ti[2] = { h1, h.below ? a0.d : h1 }, tij[2] = { R.th1(EX), h.below ? ht[1] : ht[0] };
            const real tj[2] = { a0.d, a0.c }, tji[2] = { ai.d, h.below ? aj.c : ai.c };
            real ph[2];
            plaq_sines<2>(ti, tij, tj, tji, ph);
            (h.below ? R.s2() : R.s1()) = { ph[0], ph[1] };
        }
        const C w1 = fwd(u[0], C{ qx.a, qx.b }), w2 = fwd(u[1], C{ qy.a, qy.b }), w3 = fwd(u[2], fn);
        const PiKick<real> k = pi_kick(c, f0, w1, w2, w3, S.u1(-1), field_of(S.field(-1)), S.u2(-EX),
                                       field_of(S.field(-EX)), um, fb, pr, pim);
        const real l1 = e_local(c, e1, k.c1), l2 = e_local(c, e2, k.c2), l3 = e_local(c, e3, k.c3);
        const real g1 = ad(p[0], sb(p[1], p13m)), g2 = sb(sb(p[2], p23m), p[0]), g3 = ad(p[1], p[2]);
        const IT s = o0 + roff;
        if (wr) {
            v.pir[s] = k.pr;
            v.pii[s] = k.pi;
            v.ophr[s] = fm(c.dt, k.pr, f0.r);
            v.ophi[s] = fm(c.dt, k.pi, f0.i);
        }
        um = u[2];
        fb = f0;
        p13m = p[1];
        p23m = p[2];
        __syncthreads();

        // C: curls, E kick and theta drift of plane z
        const C px = S.s1(-1), py = S.s2(-EX);
        const real ne1 = e_kick(c, l1, sb(g1, py.r));
        const real ne2 = e_kick(c, l2, ad(g2, px.r));
        const real ne3 = e_kick(c, l3, sb(ad(px.i, py.i), g3));
        if (wr) {
            v.e1[s] = ne1;
            v.e2[s] = ne2;
            v.e3[s] = ne3;
            v.oth1[s] = th_drift(c, t0[0], ne1);
            v.oth2[s] = th_drift(c, t0[1], ne2);
            v.oth3[s] = th_drift(c, t0[2], ne3);
        }
        if (z + 1 == z1) break;
        o0 = o1;
        o1 = o2;
        put_fields();                        // plane z + 1, before its registers are reloaded
        put_ring_link();
        load_plane(o1);
        load_momenta(o0);
        put_links();
    }
}

}  // namespace
}  // namespace ah
