// k_fused.cu -- fused leapfrog step: both kicks and both drifts of one time
// step (Eqs. up_pi, up_E, up_phi, up_A of arXiv:1809.00995) in one z-marching
// kernel.
//
// A CTA owns a TX x TY column of sites in the XY plane and a chunk of z planes.
// For each plane z it keeps, in shared memory, the link exponentials
// U_d = e^{i theta_d} and phi of planes z and z+1 on the tile plus a one-site
// halo ring, and the plaquette sines sin Xi_ij = Im(U_i U_j^{x+i} conj(U_i^{x+j})
// conj(U_j)) of plane z on the tile plus its low halos.  Each link exponential is
// computed once per site and shared by the covariant Laplacian, the scalar
// current and the three plaquettes; each plaquette sine is computed once and
// shared by the four E kicks that use it.  Values of plane z-1 that a site
// needs (phi, U_3, sin Xi_13, sin Xi_23) stay in the owning thread's registers
// as the CTA marches up in z, and the next plane's fields are prefetched into
// registers one plane ahead.
//
// phi and theta are read from one buffer and written to the other (ping-pong),
// Pi and E are updated in place, so every step reads and writes the 10-real
// state exactly once from DRAM; halo re-reads are served by L2.  Periodic
// boundaries are applied in the index arithmetic.
//
// That walk serves k_fused (one lattice, one step) and k_fused_batch (persistent
// CTAs over the tiles of many lattices).  FP32 lattices whose rows can be copied in
// 16 bytes run feed_tile.cuh instead (k_feed, k_feed_batch), FP64 lattices of the
// default shape step_tile.cuh.  The shapes (tile height, sites per thread in x,
// resident CTAs per SM) are chosen by the default of the size or by the autotuner,
// the number of z chunks per column by choose_chunks: each CTA marches a whole
// chunk, so a poorly filled last wave costs a whole march.
#include "ah_internal.cuh"
#include "sincos32.cuh"
#include "fused_common.cuh"
#include "feed_tile.cuh"
#include "step_tile.cuh"

namespace ah {
namespace {

// Each thread owns RX consecutive sites in x times RY rows (y stride 8).
// One work item of the fused step: tile (bx, by) of plane chunk bz, marched in z.

// IT: site-index type (int when N^3 < 2^31, so every field address is one
// 32 x 32 -> 64-bit multiply-add; long long otherwise).
template <typename real, int TY, int RX, typename IT>
__device__ __forceinline__ void fused_tile(const View<real> &v, int N, int zc, const KickCoef<real> &c,
                                           int bx, int by, int bz, unsigned char *smem_raw)
{
    using G = Geo<real, TY, RX>;
    using IO = Row<real, RX>;
    constexpr int TX = G::TX, RY = G::RY, NS = G::NS, EX = G::EX, EY = G::EY, NE = G::NE, PX = G::PX;
    cpx<real> *sU = reinterpret_cast<cpx<real> *>(smem_raw);   // [2 planes][3 dirs][NE]
    cpx<real> *sF = sU + 2 * 3 * NE;                            // [2 planes][NE] phi
    real *sP = reinterpret_cast<real *>(sF + 2 * NE);           // [3][NP] sin Xi_12, _13, _23

    const int tid = threadIdx.x, lx = tid & 31, wy = tid >> 5;
    const int x0 = bx * TX, y0 = by * TY;
    const int z0 = bz * zc;
    if (z0 >= N) return;
    const int z1 = min(z0 + zc, N);
    const IT NN = (IT)N * (IT)N;

    // own rows: in-plane offset of the first of the RX sites, validity
    int roff[RY];
    bool wr[RY];
#pragma unroll
    for (int my = 0; my < RY; ++my) {
        const int gx = x0 + RX * lx, gy = y0 + wy + 8 * my;
        wr[my] = gx < N && gy < N;
        roff[my] = wrapm(gx, N) + N * wrapm(gy, N);
    }
    auto eix = [&](int m) { return (wy + 8 * (m / RX) + 1) * EX + RX * lx + (m % RX) + 1; };
    auto pix = [&](int m) { return (wy + 8 * (m / RX) + 1) * PX + RX * lx + (m % RX) + 1; };
    // halo task (tid < NHALO): one site of the halo ring
    const bool has_halo = tid < G::NHALO;
    int hoff, heix;
    {
        int ex = 0, ey = 0;
        const int h = tid;
        if (h < EX) { ex = h; ey = 0; }
        else if (h < 2 * EX) { ex = h - EX; ey = EY - 1; }
        else if (h < 2 * EX + TY) { ex = 0; ey = 1 + h - 2 * EX; }
        else { ex = EX - 1; ey = 1 + h - 2 * EX - TY; }
        hoff = wrapm(x0 + ex - 1, N) + N * wrapm(y0 + ey - 1, N);
        heix = ey * EX + ex;
    }

    // register prefetch of one plane's phi, theta: own sites [0, NS), halo [NS]
    real fth[NS + 1][3], fph[NS + 1][2];
    auto load_plane = [&](int z) {           // z in [-1, N + 1]
        const int zz = z < 0 ? z + N : (z >= N ? z - N : z);
        const IT base = (IT)zz * NN;
#pragma unroll
        for (int my = 0; my < RY; ++my) {
            const IT s = base + (IT)roff[my];
            real t[RX];
            IO::ld(v.th1 + s, t);
#pragma unroll
            for (int mx = 0; mx < RX; ++mx) fth[my * RX + mx][0] = t[mx];
            IO::ld(v.th2 + s, t);
#pragma unroll
            for (int mx = 0; mx < RX; ++mx) fth[my * RX + mx][1] = t[mx];
            IO::ld(v.th3 + s, t);
#pragma unroll
            for (int mx = 0; mx < RX; ++mx) fth[my * RX + mx][2] = t[mx];
            IO::ld(v.phr + s, t);
#pragma unroll
            for (int mx = 0; mx < RX; ++mx) fph[my * RX + mx][0] = t[mx];
            IO::ld(v.phi + s, t);
#pragma unroll
            for (int mx = 0; mx < RX; ++mx) fph[my * RX + mx][1] = t[mx];
        }
        if (has_halo) {
            const IT s = base + (IT)hoff;
            fth[NS][0] = v.th1[s]; fth[NS][1] = v.th2[s]; fth[NS][2] = v.th3[s];
            fph[NS][0] = v.phr[s]; fph[NS][1] = v.phi[s];
        }
    };
    // U and phi of the prefetched plane into shared buffer b
    auto store_plane = [&](int b) {
#pragma unroll
        for (int t = 0; t <= NS; ++t) {
            if (t < NS || has_halo) {
                const int e = t < NS ? eix(t) : heix;
                real sn[3], co[3];
                sincos_link3(fth[t], sn, co);
#pragma unroll
                for (int d = 0; d < 3; ++d) sU[(b * 3 + d) * NE + e] = { co[d], sn[d] };
                sF[b * NE + e] = { fph[t][0], fph[t][1] };
            }
        }
    };

    // own-site registers carried along z
    cpx<real> ph_m[NS], ph_0[NS], u3_m[NS];
    real th_0[NS][3], p13_m[NS], p23_m[NS];

    // prologue: planes z0-1 and z0
    // ring slot of plane z: (z - z0 + 1) & 1
    load_plane(z0 - 1);
    constexpr int bm = 0, b0 = 1;
    store_plane(bm);
#pragma unroll
    for (int m = 0; m < NS; ++m) ph_m[m] = { fph[m][0], fph[m][1] };
    load_plane(z0);
    store_plane(b0);
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        ph_0[m] = { fph[m][0], fph[m][1] };
        th_0[m][0] = fth[m][0]; th_0[m][1] = fth[m][1]; th_0[m][2] = fth[m][2];
    }
    load_plane(z0 + 1);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        const int e = eix(m);
        const cpx<real> *Um = sU + bm * 3 * NE, *U0 = sU + b0 * 3 * NE;
        u3_m[m] = Um[2 * NE + e];
        p13_m[m] = plaq(Um[e], Um[2 * NE + e + 1], U0[e], Um[2 * NE + e]);
        p23_m[m] = plaq(Um[NE + e], Um[2 * NE + e + EX], U0[NE + e], Um[2 * NE + e]);
    }
    __syncthreads();

    // one plane z; BC (compile time) is the ring slot of plane z
    auto plane_step = [&](int z, auto bc_tag) {
        constexpr int bc = decltype(bc_tag)::value, bn = 1 - bc;
        const IT base = (IT)z * NN;
        // Pi, E of plane z (consumed after two barriers)
        real pr[NS], pim[NS], e1[NS], e2[NS], e3[NS];
#pragma unroll
        for (int my = 0; my < RY; ++my) {
            const IT s = base + (IT)roff[my];
            IO::ld(v.pir + s, pr + my * RX);
            IO::ld(v.pii + s, pim + my * RX);
            IO::ld(v.e1 + s, e1 + my * RX);
            IO::ld(v.e2 + s, e2 + my * RX);
            IO::ld(v.e3 + s, e3 + my * RX);
        }
        // A: links and phi of plane z+1 from the prefetch, then prefetch z+2
        store_plane(bn);
        cpx<real> ph_p[NS];
        real th_p[NS][3];
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            ph_p[m] = { fph[m][0], fph[m][1] };
            th_p[m][0] = fth[m][0]; th_p[m][1] = fth[m][1]; th_p[m][2] = fth[m][2];
        }
        load_plane(z + 2);
        __syncthreads();

        // B: plaquette sines of plane z on the tile (own sites) and its low halos
        const cpx<real> *U0 = sU + bc * 3 * NE, *U1p = sU + bn * 3 * NE;
        real p12[NS], p13[NS], p23[NS];
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            const int e = eix(m), p = pix(m);
            p12[m] = plaq(U0[e], U0[NE + e + 1], U0[e + EX], U0[NE + e]);
            p13[m] = plaq(U0[e], U0[2 * NE + e + 1], U1p[e], U0[2 * NE + e]);
            p23[m] = plaq(U0[NE + e], U0[2 * NE + e + EX], U1p[NE + e], U0[2 * NE + e]);
            sP[p] = p12[m];
            sP[G::NP + p] = p13[m];
            sP[2 * G::NP + p] = p23[m];
        }
        if (tid < G::NPHALO) {
            const int px = tid < PX ? tid : 0, py = tid < PX ? 0 : tid - PX + 1;
            const int e = py * EX + px, p = py * PX + px;
            sP[p] = plaq(U0[e], U0[NE + e + 1], U0[e + EX], U0[NE + e]);
            sP[G::NP + p] = plaq(U0[e], U0[2 * NE + e + 1], U1p[e], U0[2 * NE + e]);
            sP[2 * G::NP + p] = plaq(U0[NE + e], U0[2 * NE + e + EX], U1p[NE + e], U0[2 * NE + e]);
        }
        __syncthreads();

        // C: kicks and drifts of the own sites of plane z
        const cpx<real> *F0 = sF + bc * NE;
        real o_pr[NS], o_pi[NS], o_e1[NS], o_e2[NS], o_e3[NS], o_fr[NS], o_fi[NS], o_t1[NS], o_t2[NS], o_t3[NS];
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            const int e = eix(m), p = pix(m);
            const cpx<real> f0 = ph_0[m];
            const cpx<real> u1 = U0[e], u2 = U0[NE + e], u3 = U0[2 * NE + e];
            const cpx<real> u1m = U0[e - 1], u2m = U0[NE + e - EX], u3m = u3_m[m];
            // forward products U_d phi^{x+d}; backward conj(U_d^{x-d}) phi^{x-d}
            const cpx<real> w1 = mul(u1, F0[e + 1]), w2 = mul(u2, F0[e + EX]), w3 = mul(u3, ph_p[m]);
            const cpx<real> b1 = mul({ u1m.r, -u1m.i }, F0[e - 1]);
            const cpx<real> b2 = mul({ u2m.r, -u2m.i }, F0[e - EX]);
            const cpx<real> b3 = mul({ u3m.r, -u3m.i }, ph_m[m]);
            const real lr = (w1.r + b1.r) + (w2.r + b2.r) + (w3.r + b3.r) - real(6) * f0.r;
            const real li = (w1.i + b1.i) + (w2.i + b2.i) + (w3.i + b3.i) - real(6) * f0.i;
            const real pot = c.c_pot * (f0.r * f0.r + f0.i * f0.i - c.sigma2);
            const real npr = c.c_damp * pr[m] - pot * f0.r + c.c_lap * lr;
            const real npi = c.c_damp * pim[m] - pot * f0.i + c.c_lap * li;
            // current Im[conj(U_i phi^{x+i}) phi^x]
            const real cu1 = w1.r * f0.i - w1.i * f0.r;
            const real cu2 = w2.r * f0.i - w2.i * f0.r;
            const real cu3 = w3.r * f0.i - w3.i * f0.r;
            // curls sum_{j != i} [sin Xi_ij^x - sin Xi_ij^{x-j}], Xi_ji = -Xi_ij
            const real q12 = p12[m], q13 = p13[m], q23 = p23[m];
            const real cl1 = (q12 - sP[p - PX]) + (q13 - p13_m[m]);
            const real cl2 = (sP[p - 1] - q12) + (q23 - p23_m[m]);
            const real cl3 = (sP[G::NP + p - 1] - q13) + (sP[2 * G::NP + p - PX] - q23);
            const real ne1 = c.c_edamp * e1[m] + c.c_cur * cu1 - c.c_curl * cl1;
            const real ne2 = c.c_edamp * e2[m] + c.c_cur * cu2 - c.c_curl * cl2;
            const real ne3 = c.c_edamp * e3[m] + c.c_cur * cu3 - c.c_curl * cl3;
            o_pr[m] = npr; o_pi[m] = npi;
            o_e1[m] = ne1; o_e2[m] = ne2; o_e3[m] = ne3;
            o_fr[m] = f0.r + c.dt * npr;
            o_fi[m] = f0.i + c.dt * npi;
            o_t1[m] = th_0[m][0] + c.dt * ne1;
            o_t2[m] = th_0[m][1] + c.dt * ne2;
            o_t3[m] = th_0[m][2] + c.dt * ne3;
            if (c.wrap) {
                o_t1[m] = wrap_phase(o_t1[m]);
                o_t2[m] = wrap_phase(o_t2[m]);
                o_t3[m] = wrap_phase(o_t3[m]);
            }
            // march: plane z becomes z-1
            ph_m[m] = f0;
            u3_m[m] = u3;
            p13_m[m] = q13;
            p23_m[m] = q23;
            ph_0[m] = ph_p[m];
            th_0[m][0] = th_p[m][0]; th_0[m][1] = th_p[m][1]; th_0[m][2] = th_p[m][2];
        }
#pragma unroll
        for (int my = 0; my < RY; ++my) {
            if (wr[my]) {
                const IT s = base + (IT)roff[my];
                const int k = my * RX;
                IO::st(v.pir + s, o_pr + k); IO::st(v.pii + s, o_pi + k);
                IO::st(v.e1 + s, o_e1 + k); IO::st(v.e2 + s, o_e2 + k); IO::st(v.e3 + s, o_e3 + k);
                IO::st(v.ophr + s, o_fr + k); IO::st(v.ophi + s, o_fi + k);
                IO::st(v.oth1 + s, o_t1 + k); IO::st(v.oth2 + s, o_t2 + k); IO::st(v.oth3 + s, o_t3 + k);
            }
        }
        __syncthreads();
    };
    for (int k = 0; z0 + k < z1; k += 2) {
        plane_step(z0 + k, IC<1>{});
        if (z0 + k + 1 < z1) plane_step(z0 + k + 1, IC<0>{});
    }
}

// Shapes that run step_tile instead of fused_tile: FP64, one site per thread.
// (FP32 issues its link exponentials and plaquette products at 64 times the
// FP64 rate and waits on memory instead, for which fused_tile keeps one more
// plane in flight.)
template <typename real, int TY, int RX>
constexpr bool kStepTile = sizeof(real) == 8 && TY == 8 && RX == 1;

template <typename real, int TY, int RX, int MINB, typename IT>
__global__ void __launch_bounds__(256, MINB) k_fused(View<real> v, int N, int zc, KickCoef<real> c)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (kStepTile<real, TY, RX>)
        step_tile<real, TY, IT>(v, N, zc, c, blockIdx.x, blockIdx.y, blockIdx.z, smem_raw);
    else
        fused_tile<real, TY, RX, IT>(v, N, zc, c, blockIdx.x, blockIdx.y, blockIdx.z, smem_raw);
}

// The step of two rows per thread with copied planes (feed_tile.cuh).
template <int NP, int MINB, typename IT>
__global__ void __launch_bounds__(32 * NP, MINB) k_feed(View<float> v, int N, int zc, KickCoef2 c)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    feed_tile<NP, IT>(v, N, zc, c, blockIdx.x, blockIdx.y, blockIdx.z, smem_raw);
}

// Batched fused step: persistent CTAs take (lattice, tile) work items from a
// shared counter and advance every lattice of the batch by one step.  Lattices
// that have run all their steps are skipped; each lattice's step number, read
// buffer and coefficient table live in device memory (advanced by
// k_batch_advance), so the same launch sequence can be replayed from a graph.
template <int TY, int RX, int MINB>
__global__ void __launch_bounds__(256, MINB)
k_fused_batch(const BatchLattice *lat, BatchState *state, const int2 *items, const int *nitems,
              unsigned int *counter, int mode)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    const int n = *nitems;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= n) break;
        const int L = items[it].x, local = items[it].y;
        const BatchLattice &B = lat[L];
        const int step = state[L].step;
        if (!batch_takes_single(B, step, mode)) continue;
        const int cur = state[L].cur, o = 1 - cur;
        float *const *q = B.q[state[L].pe];
        View<float> v;
        v.phr = B.F.phr[cur]; v.phi = B.F.phi[cur];
        v.th1 = B.F.th[cur][0]; v.th2 = B.F.th[cur][1]; v.th3 = B.F.th[cur][2];
        v.pir = q[0]; v.pii = q[1];
        v.e1 = q[2]; v.e2 = q[3]; v.e3 = q[4];
        v.ophr = B.F.phr[o]; v.ophi = B.F.phi[o];
        v.oth1 = B.F.th[o][0]; v.oth2 = B.F.th[o][1]; v.oth3 = B.F.th[o][2];
        const int bx = local % B.tiles_x, by = (local / B.tiles_x) % B.tiles_y, bz = local / (B.tiles_x * B.tiles_y);
        fused_tile<float, TY, RX, int>(v, B.N, B.zc, B.coefs[step], bx, by, bz, smem_raw);
        __syncthreads();
    }
}

// The same for the lattices that ah_step steps with k_feed (feed_lattice).  The
// item's pointers and coefficients are in shared memory, where they cost no
// registers.
template <int NP, int MINB>
__global__ void __launch_bounds__(32 * NP, MINB)
    k_feed_batch(const BatchLattice *lat, BatchState *state, const int2 *items, const int *nitems,
                 unsigned int *counter, int mode)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    __shared__ View<float> sv;
    __shared__ KickCoef2 sc;
    const int n = *nitems;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int it = s_item;
        if (it >= n) break;
        const int L = items[it].x, local = items[it].y;
        const BatchLattice &B = lat[L];
        const int step = state[L].step;
        const bool takes = batch_takes_single(B, step, mode);
        if (takes && threadIdx.x == 0) {
            const int cur = state[L].cur, o = 1 - cur;
            float *const *q = B.q[state[L].pe];
            sv.phr = B.F.phr[cur]; sv.phi = B.F.phi[cur];
            sv.th1 = B.F.th[cur][0]; sv.th2 = B.F.th[cur][1]; sv.th3 = B.F.th[cur][2];
            sv.pir = q[0]; sv.pii = q[1]; sv.e1 = q[2]; sv.e2 = q[3]; sv.e3 = q[4];
            sv.ophr = B.F.phr[o]; sv.ophi = B.F.phi[o];
            sv.oth1 = B.F.th[o][0]; sv.oth2 = B.F.th[o][1]; sv.oth3 = B.F.th[o][2];
            sc = pair_coef(B.coefs[step]);
        }
        __syncthreads();
        if (takes) {
            const int bx = local % B.tiles_x, by = (local / B.tiles_x) % B.tiles_y;
            feed_tile<NP, int>(sv, B.N, B.zc, sc, bx, by, local / (B.tiles_x * B.tiles_y), smem_raw);
        }
        __syncthreads();
    }
}

// After a batched step: every lattice that took part (batch_takes_single)
// moves to its next step and swaps its phi/theta buffers; the work counters are
// reset.
__global__ void k_batch_advance(const BatchLattice *lat, BatchState *state, int nlat, unsigned int *counter,
                                int mode)
{
    for (int L = threadIdx.x; L < nlat; L += blockDim.x) {
        if (batch_takes_single(lat[L], state[L].step, mode)) {
            state[L].step += 1;
            state[L].cur ^= 1;
        }
    }
    if (threadIdx.x < 2) counter[threadIdx.x] = 0u;
}

// Compile-time shapes of the fused step: tile height TY (TY/8 rows per thread),
// RX sites per thread in x (tile width 32 RX; RX = 2 uses 8-byte vector
// accesses and needs an even N), and the minimum resident CTAs per SM the
// register allocation must allow; min_chunk is the shortest z chunk.  The z
// chunk count is either "about 16 waves of CTAs" or (_w) the wave-quantisation
// model of choose_chunks.
struct VariantInfo { int ty, rx, minb, min_chunk; bool wave_model; const char *name; };
constexpr VariantInfo kVariants32[] = {
    { 16, 1, 2, 16, false, "ty16_b2" }, { 16, 1, 3, 16, false, "ty16_b3" }, { 8, 1, 4, 16, false, "ty8_b4" },
    { 8, 1, 3, 16, false, "ty8_b3" },  { 32, 1, 1, 16, false, "ty32_b1" }, { 16, 1, 2, 64, false, "ty16_b2_z64" },
    { 8, 2, 3, 16, false, "x2_ty8_b3" }, { 8, 2, 2, 16, false, "x2_ty8_b2" }, { 16, 2, 2, 16, false, "x2_ty16_b2" },
    { 16, 2, 1, 16, false, "x2_ty16_b1" }, { 8, 1, 4, 16, true, "ty8_b4_w" }, { 8, 1, 3, 16, true, "ty8_b3_w" },
    { 8, 2, 2, 16, true, "x2_ty8_b2_w" }, { 16, 1, 2, 16, true, "ty16_b2_w" },
};
constexpr VariantInfo kVariants64[] = { { 16, 1, 1, 16, false, "ty16_b1" }, { 8, 1, 2, 16, false, "ty8_b2" },
                                        { 8, 2, 1, 16, false, "x2_ty8_b1" }, { 8, 1, 2, 16, true, "ty8_b2_w" } };

}  // namespace

int device_sm_count()
{
    static int sms[64] = {};
    int &n = sms[device_slot()];
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 152;
    }
    return n;
}

int choose_chunks(int N, long long tiles, int per_sm, int extra, const PlaneTimes &times)
{
    const int nmax = std::min(N, 64);
    const long long sms = device_sm_count(), slots = sms * per_sm;
    int best = 1;
    long long best_cost = -1;
    for (int n = 1; n <= nmax; ++n) {
        const long long zc = (N + n - 1) / n, ctas = tiles * ((N + zc - 1) / zc);
        const long long last = ctas % slots;
        const long long wave = ctas / slots * times.t[per_sm - 1] + (last ? times.t[(last - 1) / sms] : 0);
        const long long cost = (zc + extra) * wave;
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = n;
        }
    }
    return best;
}

namespace {

// FP32 step, microseconds x 100 per plane measured at 64^3 to 256^3 (113 with one
// CTA on an SM, 255 with four)
constexpr PlaneTimes kStepTimes32 = { { 113, 156, 199, 255 } };
// FP64 step: bound by the FP64 pipe, which one CTA fills to 0.88
constexpr PlaneTimes kStepTimes64 = { { 123, 216, 324, 432 } };

// z chunks of the k_feed grid: at most 64 planes, since CTAs of longer marches
// drift apart until the rows they share no longer meet in L2 (1024^3: 4 chunks read
// 62 B per site and take 17.3 ms, 16 chunks 13.8).
constexpr PlaneTimes kFeedTimes = { { 140, 214 } };
constexpr int kFeedMaxChunk = 64;

template <typename IT>
cudaError_t launch_feed_it(const View<float> &v, int N, const KickCoef<float> &c, cudaStream_t st)
{
    constexpr int NP = 8, MINB = 2;
    using G = FeedGeo<NP>;
    static unsigned long long configured = 0;   // per device, once per instantiation
    const unsigned long long dev_bit = 1ULL << device_slot();
    if (!(configured & dev_bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_feed<NP, MINB, IT>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem);
        if (e != cudaSuccess) return e;
        configured |= dev_bit;
    }
    const int tx = (N + 31) / 32, ty = (N + G::TY - 1) / G::TY;
    const int n = std::max(choose_chunks(N, (long long)tx * ty, MINB, 2, kFeedTimes),
                           (N + kFeedMaxChunk - 1) / kFeedMaxChunk);
    const int zc = (N + n - 1) / n;
    k_feed<NP, MINB, IT><<<dim3(tx, ty, (N + zc - 1) / zc), G::NT, G::smem, st>>>(v, N, zc, pair_coef(c));
    return cudaGetLastError();
}
cudaError_t launch_feed(const View<float> &v, int N, const KickCoef<float> &c, cudaStream_t st)
{
    return (long long)N * N * N < (1LL << 31) ? launch_feed_it<int>(v, N, c, st) : launch_feed_it<long long>(v, N, c, st);
}

template <typename real, int TY, int RX, int MINB>
cudaError_t launch_shape(const View<real> &v, int N, const KickCoef<real> &c, int min_chunk, bool wave_model,
                         cudaStream_t st)
{
    using G = Geo<real, TY, RX>;
    constexpr size_t smem = kStepTile<real, TY, RX> ? TileGeo<real, 8>::smem : G::smem;
    if (RX > 1 && (N & 1)) return cudaErrorInvalidValue;
    const bool idx32 = (long long)N * N * N < (1LL << 31);
    static unsigned long long configured = 0;   // per device, once per instantiation
    const unsigned long long dev_bit = 1ULL << device_slot();
    if (!(configured & dev_bit)) {
        cudaError_t e = cudaFuncSetAttribute(k_fused<real, TY, RX, MINB, int>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fused<real, TY, RX, MINB, long long>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured |= dev_bit;
    }
    const int tx = (N + G::TX - 1) / G::TX, ty = (N + TY - 1) / TY;
    int nch;
    if (wave_model) {
        nch = choose_chunks(N, (long long)tx * ty, MINB, 1, sizeof(real) == 4 ? kStepTimes32 : kStepTimes64);
    } else {
        // enough z chunks for several waves of CTAs, chunks of at least min_chunk planes
        nch = (int)((16LL * device_sm_count() + (long long)tx * ty - 1) / ((long long)tx * ty));
        nch = max(1, min(nch, N / min_chunk));
    }
    const int zc = (N + nch - 1) / nch;
    nch = (N + zc - 1) / zc;
    if (idx32) k_fused<real, TY, RX, MINB, int><<<dim3(tx, ty, nch), G::NT, smem, st>>>(v, N, zc, c);
    else k_fused<real, TY, RX, MINB, long long><<<dim3(tx, ty, nch), G::NT, smem, st>>>(v, N, zc, c);
    return cudaGetLastError();
}

}  // namespace

// Shape used when a simulation is not autotuned.  FP32: from 64^3 on, where rows can
// be copied in 16 bytes, ty16_b2_w (feed_tile.cuh; it ties at 64^3, 10.3 us, and wins
// from 96^3 on, 18.5 against 20.6 us), else ty8_b4_w, the fastest of the others at
// every measured size from 24^3 to 1024^3.
template <>
int fused_default_variant<float>(int N) { return feed_ok(N) && N >= 64 ? 13 : 10; }
template <>
int fused_default_variant<double>(int) { return 3; }      // ty8_b2_w

template <>
int fused_variant_count<float>() { return (int)(sizeof(kVariants32) / sizeof(kVariants32[0])); }
template <>
int fused_variant_count<double>() { return (int)(sizeof(kVariants64) / sizeof(kVariants64[0])); }
template <>
const char *fused_variant_name<float>(int k) { return kVariants32[k].name; }
template <>
const char *fused_variant_name<double>(int k) { return kVariants64[k].name; }

template <>
bool fused_variant_ok<float>(int k, int N) { return kVariants32[k].rx == 1 || (N % 2 == 0); }
template <>
bool fused_variant_ok<double>(int k, int N) { return kVariants64[k].rx == 1 || (N % 2 == 0); }

template <>
cudaError_t launch_fused_step<float>(const View<float> &v, int N, const KickCoef<float> &c, int variant,
                                     cudaStream_t st)
{
    if (variant < 0 || variant >= fused_variant_count<float>()) return cudaErrorInvalidValue;
    const int mc = kVariants32[variant].min_chunk;
    const bool wm = kVariants32[variant].wave_model;
    // ty16_b2_w: two rows per thread; where rows can be copied in 16 bytes, from
    // copied planes
    if (variant == 13 && feed_ok(N)) return launch_feed(v, N, c, st);
    switch (variant) {
    case 0: return launch_shape<float, 16, 1, 2>(v, N, c, mc, wm, st);
    case 1: return launch_shape<float, 16, 1, 3>(v, N, c, mc, wm, st);
    case 2: return launch_shape<float, 8, 1, 4>(v, N, c, mc, wm, st);
    case 3: return launch_shape<float, 8, 1, 3>(v, N, c, mc, wm, st);
    case 4: return launch_shape<float, 32, 1, 1>(v, N, c, mc, wm, st);
    case 5: return launch_shape<float, 16, 1, 2>(v, N, c, mc, wm, st);
    case 6: return launch_shape<float, 8, 2, 3>(v, N, c, mc, wm, st);
    case 7: return launch_shape<float, 8, 2, 2>(v, N, c, mc, wm, st);
    case 8: return launch_shape<float, 16, 2, 2>(v, N, c, mc, wm, st);
    case 9: return launch_shape<float, 16, 2, 1>(v, N, c, mc, wm, st);
    case 10: return launch_shape<float, 8, 1, 4>(v, N, c, mc, wm, st);
    case 11: return launch_shape<float, 8, 1, 3>(v, N, c, mc, wm, st);
    case 12: return launch_shape<float, 8, 2, 2>(v, N, c, mc, wm, st);
    case 13: return launch_shape<float, 16, 1, 2>(v, N, c, mc, wm, st);
    default: return cudaErrorInvalidValue;
    }
}
template <>
cudaError_t launch_fused_step<double>(const View<double> &v, int N, const KickCoef<double> &c, int variant,
                                      cudaStream_t st)
{
    if (variant < 0 || variant >= fused_variant_count<double>()) return cudaErrorInvalidValue;
    const int mc = kVariants64[variant].min_chunk;
    const bool wm = kVariants64[variant].wave_model;
    switch (variant) {
    case 0: return launch_shape<double, 16, 1, 1>(v, N, c, mc, wm, st);
    case 1: return launch_shape<double, 8, 1, 2>(v, N, c, mc, wm, st);
    case 2: return launch_shape<double, 8, 2, 1>(v, N, c, mc, wm, st);
    case 3: return launch_shape<double, 8, 1, 2>(v, N, c, mc, wm, st);
    default: return cudaErrorInvalidValue;
    }
}


// ---- batched step ----
namespace {
struct BatchShape { int ty, rx, minb; };
constexpr BatchShape kBatchShapes[] = { { 8, 1, 4 }, { 16, 1, 2 }, { 8, 2, 2 } };

template <int TY, int RX, int MINB>
cudaError_t launch_batch_shape(const BatchLattice *lat, BatchState *state, const int2 *items, const int *nitems,
                               unsigned int *counter, int num_sms, cudaStream_t st, int mode)
{
    using G = Geo<float, TY, RX>;
    static int blocks_per_sm_dev[64] = {};      // per device
    int &blocks_per_sm = blocks_per_sm_dev[device_slot()];
    if (!blocks_per_sm) {
        cudaError_t e = cudaFuncSetAttribute(k_fused_batch<TY, RX, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)G::smem);
        if (e != cudaSuccess) return e;
        int b = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_fused_batch<TY, RX, MINB>, 256, G::smem);
        if (e != cudaSuccess) return e;
        blocks_per_sm = b < 1 ? 1 : b;
    }
    k_fused_batch<TY, RX, MINB><<<num_sms * blocks_per_sm, 256, G::smem, st>>>(lat, state, items, nitems, counter,
                                                                              mode);
    return cudaGetLastError();
}

cudaError_t launch_feed_batch(const BatchLattice *lat, BatchState *state, const int2 *items, const int *nitems,
                              unsigned int *counter, int num_sms, cudaStream_t st, int mode)
{
    using G = FeedGeo<8>;
    static unsigned long long configured = 0;   // per device
    const unsigned long long dev_bit = 1ULL << device_slot();
    if (!(configured & dev_bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_feed_batch<8, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)G::smem);
        if (e != cudaSuccess) return e;
        configured |= dev_bit;
    }
    k_feed_batch<8, 2><<<num_sms * 2, G::NT, G::smem, st>>>(lat, state, items, nitems, counter, mode);
    return cudaGetLastError();
}
}  // namespace

int batch_shape_count() { return (int)(sizeof(kBatchShapes) / sizeof(kBatchShapes[0])); }

// Per-shape one-time set-up (shared-memory attribute, occupancy) done outside
// any stream capture: a launch of an empty work list.
cudaError_t batch_shape_prepare(int shape, int num_sms, cudaStream_t st, bool two)
{
    // a few bytes of device scratch per device, kept for the life of the process
    static BatchState *d_dummy_dev[64] = {};
    static int *d_zero_dev[64] = {};
    static unsigned int *d_cnt_dev[64] = {};
    const int ds = device_slot();
    BatchState *&d_dummy = d_dummy_dev[ds];
    int *&d_zero = d_zero_dev[ds];
    unsigned int *&d_cnt = d_cnt_dev[ds];
    if (!d_dummy) {
        BatchState *a = nullptr;
        int *z = nullptr;
        unsigned int *c = nullptr;
        cudaError_t e = cudaMalloc(&a, sizeof(BatchState));
        if (e == cudaSuccess) e = cudaMalloc(&z, sizeof(int));
        if (e == cudaSuccess) e = cudaMalloc(&c, 2 * sizeof(unsigned int));
        if (e == cudaSuccess) e = cudaMemsetAsync(z, 0, sizeof(int), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(c, 0, 2 * sizeof(unsigned int), st);
        if (e != cudaSuccess) {
            cudaFree(a); cudaFree(z); cudaFree(c);
            return e;
        }
        d_dummy = a; d_zero = z; d_cnt = c;
    }
    // nlat = 0: the advance kernel touches no lattice; nitems = 0: no work
    if (two) return launch_fused2_batch(shape, nullptr, d_dummy, 0, nullptr, d_zero, d_cnt, num_sms, st);
    const BatchItems none = { nullptr, d_zero, true };
    return launch_fused_batch(shape, nullptr, d_dummy, 0, none, none, d_cnt, num_sms, st);
}

bool feed_lattice(int N) { return fused_default_variant<float>(N) == 13; }

void batch_tiles(int shape, int N, int *tx, int *ty)
{
    if (feed_lattice(N)) {
        *tx = (N + 31) / 32;
        *ty = (N + FeedGeo<8>::TY - 1) / FeedGeo<8>::TY;
        return;
    }
    const BatchShape &b = kBatchShapes[shape];
    *tx = (N + 32 * b.rx - 1) / (32 * b.rx);
    *ty = (N + b.ty - 1) / b.ty;
}

int batch_resident_ctas(int shape, bool feed) { return feed ? 2 : kBatchShapes[shape].minb; }

bool batch_shape_ok(int shape, int N) { return kBatchShapes[shape].rx == 1 || N % 2 == 0; }

cudaError_t launch_fused_batch(int shape, const BatchLattice *lat, BatchState *state, int nlat,
                               const BatchItems &plain, const BatchItems &feed, unsigned int *counter, int num_sms,
                               cudaStream_t st, int mode)
{
    cudaError_t e = cudaSuccess;
    if (plain.any) {
        switch (shape) {
        case 0: e = launch_batch_shape<8, 1, 4>(lat, state, plain.items, plain.count, counter, num_sms, st, mode); break;
        case 1: e = launch_batch_shape<16, 1, 2>(lat, state, plain.items, plain.count, counter, num_sms, st, mode); break;
        case 2: e = launch_batch_shape<8, 2, 2>(lat, state, plain.items, plain.count, counter, num_sms, st, mode); break;
        default: e = cudaErrorInvalidValue;
        }
    }
    if (e == cudaSuccess && feed.any)
        e = launch_feed_batch(lat, state, feed.items, feed.count, counter + 1, num_sms, st, mode);
    if (e != cudaSuccess) return e;
    k_batch_advance<<<1, 256, 0, st>>>(lat, state, nlat, counter, mode);
    return cudaGetLastError();
}

}  // namespace ah
