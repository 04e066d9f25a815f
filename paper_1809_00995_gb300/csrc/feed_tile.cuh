// feed_tile.cuh -- one FP32 leapfrog step on a tile, two rows per thread, from
// planes copied ahead.
//
// A CTA of 32 x NP threads owns 32 x 2 NP sites of the XY plane and a chunk of z
// planes; thread (x, p) owns rows 2p and 2p + 1 and works on both with packed
// arithmetic (pair_math.cuh): 235 thread-instructions per site against 350 of the
// one-site walk in k_fused.cu.  That takes the registers of a prefetch, and with 16
// warps per SM more bytes have to be in flight, so the fields come through shared
// memory, two planes ahead of use: cp.async of 16 bytes past L1, rows of 40 floats of
// phi and theta (32 own columns and 4 on either side, so the ring's columns come with
// them) and of 32 floats of Pi and E.  16 bytes must not straddle the end of a row,
// nor a window of 40 columns wrap twice: N a multiple of 4, and at least 40.
//
// What it measured (512^3, ms per step): 1.69 = 6.3 TB/s, 0.93 of 6.8 TB/s, against
// 2.06 of the one-site walk; 256^3 0.231 against 0.275; 1024^3 13.8 against 16.4.
// One plane ahead instead of two 1.98 (the copies' latency shows); rows copied whole
// by cp.async.bulk 2.52 (170 copies of 128 or 160 bytes per plane and CTA take 22
// cycles each); one barrier per plane, with the curls of plane z - 1 after the barrier
// of plane z, no faster (more instructions); 8- or 4-byte copies for other N, which
// go through L1, slower than the one-site walk (250^3: 0.388 against 0.262).
//
// Raw phi and theta of a plane and its neighbours are read from the copied rows.
// Exchanged through shared memory are only values that a neighbour has computed:
//   conj(U_1) phi of x - 1, conj(U_2) phi of x - y   backward products, formed by the
//                                                     site that owns the link;
//   sin Xi_12, sin Xi_13 of x - 1, sin Xi_12, sin Xi_23 of x - y   for the curls.
// Two barriers per plane:
//   B  (after plane z + 1 and Pi, E of plane z have arrived) plaquette sines to
//      shared memory; Laplacian, Pi kick and phi drift, stored;
//   C  (after the sines) curls, E kick and theta drift, stored; link exponentials
//      and backward products of plane z + 1.
// The ring's extra work, below and to the left of the tile where links point into
// it, is four tasks on four warps.
#pragma once
#include "fused_common.cuh"
#include "pair_math.cuh"

namespace ah {

inline bool feed_ok(int N) { return N % 4 == 0 && N >= 40; }

namespace {

// 16 bytes past L1 (both addresses 16-byte aligned)
__device__ __forceinline__ void feed_copy(unsigned dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

template <int NP>
struct FeedGeo {
    static constexpr int SR = 4, SM = 3;                       // slots of raw planes and of Pi, E planes
    static constexpr int TX = 32, TY = 2 * NP, NT = 32 * NP, W = 40;
    // phi, theta of a plane: [5][TY + 2 rows][W]; Pi, E: [5][TY][TX]
    static constexpr int raw_array = 4 * W * (TY + 2), raw_plane = 5 * raw_array;
    static constexpr int mom_array = 4 * TX * TY, mom_plane = 5 * mom_array;
    // exchanged values, per (pair of rows, column), pairs and columns -1 .. 31
    static constexpr int EX = TX + 1, NE = EX * (NP + 1);
    static constexpr int off_mom = SR * raw_plane, off_b1 = off_mom + SM * mom_plane;
    static constexpr int off_s1 = off_b1 + 16 * NE, off_hb = off_s1 + 16 * NE, off_hp = off_hb + 8 * NE;
    static constexpr size_t smem = off_hp + 8 * NE;
    static_assert(NP >= 4 && raw_array % 16 == 0 && off_b1 % 16 == 0, "layout");
};
__device__ __forceinline__ float2 lo2(float4 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float2 hi2(float4 a) { return make_float2(a.z, a.w); }
__device__ __forceinline__ float4 cat(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

template <int NP, typename IT, typename VIEW, typename COEF>
__device__ __forceinline__ void feed_tile(const VIEW &v, int N, int zc, const COEF &c, int bx, int by, int bz,
                                          unsigned char *smem)
{
    using G = FeedGeo<NP>;
    constexpr int RW = 4 * G::W;                       // bytes of a raw row
    const int lx = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int x0 = bx * 32, y0 = by * G::TY, z0 = bz * zc;
    if (z0 >= N) return;
    const int z1 = min(z0 + zc, N);
    const IT NN = (IT)N * (IT)N;
    const bool wr0 = x0 + lx < N && y0 + 2 * wp < N, wr1 = x0 + lx < N && y0 + 2 * wp + 1 < N;
    const int roff = x0 + lx + N * (y0 + 2 * wp);       // used where wr0 or wr1 holds
    // ---- copies: this thread's 16 bytes of a plane's phi and theta rows (10 per
    // row), and of the Pi, E rows (8 per row; the second half of the threads takes
    // every other array)
    const bool raw_copy = threadIdx.x < 10 * (G::TY + 2);
    int raw_src = 0, mom_src;
    unsigned raw_dst = 0, mom_dst;
    {
        const unsigned sbase = (unsigned)__cvta_generic_to_shared(smem);
        const int row = threadIdx.x / 10, c4 = 4 * (threadIdx.x % 10);
        if (raw_copy) raw_src = wrapm(x0 - 4 + c4, N) + N * wrapm(y0 - 1 + row, N);
        raw_dst = sbase + row * RW + 4 * c4;
        const int q = threadIdx.x % (G::NT / 2), mrow = q / 8, mc4 = 4 * (q % 8);
        mom_src = x0 + mc4 < N ? x0 + mc4 + N * wrapm(y0 + mrow, N) : -1;
        mom_dst = sbase + G::off_mom + mrow * 128 + 4 * mc4;
    }
    const bool second = wp >= NP / 2;
    auto plane_of = [&](int z) { return (IT)(z < 0 ? z + N : (z >= N ? z - N : z)) * NN; };
    auto copy_raw = [&](int z, int off) {
        if (raw_copy) {
            const IT s = plane_of(z) + (IT)raw_src;
            const unsigned d = raw_dst + off;
            feed_copy(d, v.phr + s);
            feed_copy(d + G::raw_array, v.phi + s);
            feed_copy(d + 2 * G::raw_array, v.th1 + s);
            feed_copy(d + 3 * G::raw_array, v.th2 + s);
            feed_copy(d + 4 * G::raw_array, v.th3 + s);
        }
    };
    auto copy_mom = [&](int z, int m) {
        if (mom_src >= 0) {
            const IT s = plane_of(z) + (IT)mom_src;
            const unsigned d = mom_dst + m * G::mom_plane;
            if (!second) {
                feed_copy(d, v.pir + s);
                feed_copy(d + 2 * G::mom_array, v.e1 + s);
                feed_copy(d + 4 * G::mom_array, v.e3 + s);
            } else {
                feed_copy(d + G::mom_array, v.pii + s);
                feed_copy(d + 3 * G::mom_array, v.e2 + s);
            }
        }
    };
    auto commit = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };

    // own and neighbour values in a raw slot: rows 2p, 2p + 1 are raw rows 2p + 1, 2p + 2
    unsigned char *const own = smem + (2 * wp + 1) * RW + 4 * (lx + 4);
    auto raw = [&](int off, int k, int row, int col) -> float {
        return *reinterpret_cast<const float *>(own + off + k * G::raw_array + row * RW + 4 * col);
    };
    auto raw2 = [&](int off, int k, int row, int col) { return make_float2(raw(off, k, row, col), raw(off, k, row + 1, col)); };
    // exchanged values: entry (pair p, column x) at (p + 1) EX + x + 1
    const int e = (wp + 1) * G::EX + lx + 1;
    float4 *const b1s = reinterpret_cast<float4 *>(smem + G::off_b1) + e;
    float4 *const s1s = reinterpret_cast<float4 *>(smem + G::off_s1) + e;
    float2 *const hbs = reinterpret_cast<float2 *>(smem + G::off_hb) + e;
    float2 *const hps = reinterpret_cast<float2 *>(smem + G::off_hp) + e;
    // the ring's links that point into the tile: theta_2 of the row below, raw row 0
    // (products warp 0, sines warp 1), and theta_1 of the column to the left, one lane
    // per pair of rows (warps 2 and 3)
    auto rowb = [&](int off, int k, int row, int col) {
        return *reinterpret_cast<const float *>(smem + off + k * G::raw_array + row * RW + 4 * (lx + 4 + col));
    };
    auto colf = [&](int off, int k, int row, int col) {
        return *reinterpret_cast<const float *>(smem + off + k * G::raw_array + (2 * lx + 1 + row) * RW + 4 * (3 + col));
    };
    auto colb = [&](int off, int k, int row, int col) { return make_float2(colf(off, k, row, col), colf(off, k, row + 1, col)); };
    const int le = (lx + 1) * G::EX, be = lx + 1;

    C22 f0, b2;
    U22 u[3];
    float2 t0[3];
    // own fields and exchanged products of the plane in raw slot `off`
    auto take_plane = [&](int off) {
        f0.r = raw2(off, 0, 0, 0);
        f0.i = raw2(off, 1, 0, 0);
#pragma unroll
        for (int d = 0; d < 3; ++d) t0[d] = raw2(off, 2 + d, 0, 0);
        link_exps2<3>(t0, u);
        const C22 b1 = bwd(u[0], f0);
        *b1s = cat(b1.r, b1.i);
        b2 = bwd(u[1], f0);
        *hbs = make_float2(b2.r.y, b2.i.y);
        if (wp == 0) {
            const float2 t = pk(rowb(off, 3, 0, 0));
            U22 w;
            link_exps2<1>(&t, &w);
            const C22 b = bwd(w, C22{ pk(rowb(off, 0, 0, 0)), pk(rowb(off, 1, 0, 0)) });
            reinterpret_cast<float2 *>(smem + G::off_hb)[be] = make_float2(b.r.x, b.i.x);
        } else if (wp == 2 && lx < NP) {
            const float2 t = colb(off, 2, 0, 0);
            U22 w;
            link_exps2<1>(&t, &w);
            const C22 b = bwd(w, C22{ colb(off, 0, 0, 0), colb(off, 1, 0, 0) });
            reinterpret_cast<float4 *>(smem + G::off_b1)[le] = cat(b.r, b.i);
        }
    };

    // raw slots of planes z - 1 (the next one to copy to), z, z + 1 and z + 2
    int ra = 0, rb = G::raw_plane, rc = 2 * G::raw_plane, rd = 3 * G::raw_plane;
    copy_raw(z0 - 1, ra);
    copy_raw(z0, rb);
    commit();
    copy_raw(z0 + 1, rc);
    copy_mom(z0, 0);
    commit();
    if (z0 + 1 < z1) {
        copy_raw(z0 + 2, rd);
        copy_mom(z0 + 1, 1);
    }
    commit();
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();
    take_plane(ra);                                    // plane z0 - 1
    C22 b3 = bwd(u[2], f0);
    float2 p13m, p23m;
    {
        // all three plaquettes of plane z0 - 1, though only two of the sines are wanted:
        // the vote in plaq_sines2 has to be the one that the loop takes for this plane,
        // or the bits of plane z0 would depend on where the chunks begin (which, in a
        // batch, the other lattices decide)
        const float2 ti[3] = { t0[0], t0[0], t0[1] };
        const float2 tij[3] = { make_float2(t0[0].y, raw(ra, 2, 2, 0)), raw2(rb, 2, 0, 0), raw2(rb, 3, 0, 0) };
        const float2 tj[3] = { t0[1], t0[2], t0[2] };
        const float2 tji[3] = { raw2(ra, 3, 0, 1), raw2(ra, 4, 0, 1), make_float2(t0[2].y, raw(ra, 4, 2, 0)) };
        float2 p[3];
        plaq_sines2<3>(ti, tij, tj, tji, p);
        p13m = p[1];
        p23m = p[2];
    }
    take_plane(rb);

    for (int z = z0, m = 0, mi = 2;; ++z, m = m + 1 == G::SM ? 0 : m + 1, mi = mi + 1 == G::SM ? 0 : mi + 1) {
        const IT s0 = (IT)z * NN + (IT)roff, s1 = s0 + (IT)N;
        auto put = [&](float *p, float2 x) {
            if (wr0) p[s0] = x.x;
            if (wr1) p[s1] = x.y;
        };
        const bool more = z + 1 < z1;
        // plane z + 1 and Pi, E of plane z have arrived (all but the last group of
        // copies); everybody has done with plane z - 1
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (z + 2 < z1) {
            copy_raw(z + 3, ra);
            copy_mom(z + 2, mi);
        }
        commit();
        // B: plaquette sines of plane z, Pi kick and phi drift
        float2 p[3];
        const C22 fz = { raw2(rc, 0, 0, 0), raw2(rc, 1, 0, 0) };
        {
            const float2 ti[3] = { t0[0], t0[0], t0[1] };
            const float2 tij[3] = { make_float2(t0[0].y, raw(rb, 2, 2, 0)), raw2(rc, 2, 0, 0), raw2(rc, 3, 0, 0) };
            const float2 tj[3] = { t0[1], t0[2], t0[2] };
            const float2 tji[3] = { raw2(rb, 3, 0, 1), raw2(rb, 4, 0, 1), make_float2(t0[2].y, raw(rb, 4, 2, 0)) };
            plaq_sines2<3>(ti, tij, tj, tji, p);
            *s1s = cat(p[0], p[1]);
            *hps = make_float2(p[0].y, p[2].y);
        }
        // and of the ring's plaquettes that the curls reach
        if (wp == 1) {
            const float2 t1 = pk(rowb(rb, 2, 0, 0)), t2 = pk(rowb(rb, 3, 0, 0)), t3 = pk(rowb(rb, 4, 0, 0));
            const float2 ti[2] = { t1, t2 }, tij[2] = { pk(rowb(rb, 2, 1, 0)), pk(rowb(rc, 3, 0, 0)) };
            const float2 tj[2] = { t2, t3 }, tji[2] = { pk(rowb(rb, 3, 0, 1)), pk(rowb(rb, 4, 1, 0)) };
            float2 q[2];
            plaq_sines2<2>(ti, tij, tj, tji, q);
            reinterpret_cast<float2 *>(smem + G::off_hp)[be] = make_float2(q[0].x, q[1].x);
        } else if (wp == 3 && lx < NP) {
            const float2 t1 = colb(rb, 2, 0, 0), t2 = colb(rb, 3, 0, 0), t3 = colb(rb, 4, 0, 0);
            const float2 ti[2] = { t1, t1 }, tij[2] = { colb(rb, 2, 1, 0), colb(rc, 2, 0, 0) };
            const float2 tj[2] = { t2, t3 }, tji[2] = { colb(rb, 3, 0, 1), colb(rb, 4, 0, 1) };
            float2 q[2];
            plaq_sines2<2>(ti, tij, tj, tji, q);
            reinterpret_cast<float4 *>(smem + G::off_s1)[le] = cat(q[0], q[1]);
        }
        float2 l1, l2, l3;
        {
            const unsigned char *q = smem + G::off_mom + m * G::mom_plane + 2 * wp * 128 + 4 * lx;
            auto mom = [&](int k) {
                const float *f = reinterpret_cast<const float *>(q + k * G::mom_array);
                return make_float2(f[0], f[32]);
            };
            const C22 w1 = fwd(u[0], C22{ raw2(rb, 0, 0, 1), raw2(rb, 1, 0, 1) });
            const C22 w2 = fwd(u[1], C22{ make_float2(f0.r.y, raw(rb, 0, 2, 0)), make_float2(f0.i.y, raw(rb, 1, 2, 0)) });
            const C22 w3 = fwd(u[2], fz);
            const float4 bl = b1s[-1];
            const float2 bb = hbs[-G::EX];
            const PiKick2 k = pi_kick(c, f0, w1, w2, w3, C22{ lo2(bl), hi2(bl) },
                                      C22{ make_float2(bb.x, b2.r.x), make_float2(bb.y, b2.i.x) }, b3, mom(0), mom(1));
            put(v.pir, k.pr);
            put(v.pii, k.pi);
            put(v.ophr, fm(c.dt, k.pr, f0.r));
            put(v.ophi, fm(c.dt, k.pi, f0.i));
            l1 = e_local(c, mom(2), k.c1);
            l2 = e_local(c, mom(3), k.c2);
            l3 = e_local(c, mom(4), k.c3);
        }
        const float2 g1 = ad(p[0], sb(p[1], p13m)), g2 = sb(sb(p[2], p23m), p[0]), g3 = ad(p[1], p[2]);
        b3 = bwd(u[2], f0);
        p13m = p[1];
        p23m = p[2];
        __syncthreads();

        // C: curls, E kick and theta drift; then the products of plane z + 1
        {
            const float4 px = s1s[-1];
            const float2 hy = hps[-G::EX];
            const float2 y12 = make_float2(hy.x, p[0].x), y23 = make_float2(hy.y, p[2].x);
            const float2 ne1 = e_kick(c, l1, sb(g1, y12));
            const float2 ne2 = e_kick(c, l2, ad(g2, lo2(px)));
            const float2 ne3 = e_kick(c, l3, sb(ad(hi2(px), y23), g3));
            put(v.e1, ne1);
            put(v.e2, ne2);
            put(v.e3, ne3);
            put(v.oth1, th_drift(c, t0[0], ne1));
            put(v.oth2, th_drift(c, t0[1], ne2));
            put(v.oth3, th_drift(c, t0[2], ne3));
        }
        if (!more) break;
        const int t = ra;
        ra = rb;
        rb = rc;
        rc = rd;
        rd = t;
        take_plane(rb);
    }
}

}  // namespace
}  // namespace ah
