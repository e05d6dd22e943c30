// blocksolve.cuh -- the persistent block-solver kernel (K6); instantiated per storage policy and
// block length in bs_<policy><l>.cu so that the instantiations compile in parallel.
#pragma once

#include <cooperative_groups.h>

#include "blas.cuh"
#include "ctx.h"
#include "lowprec.cuh"
#include "split64.cuh"
#include "stencil.cuh"

namespace ddrw {

template <class P> struct BlkArgs {
    using E = typename P::SElem;
    const E *b;
    E *x;
    E *r, *rh, *p, *v;
    long rstride;
    const typename P::UElem *U;
    const typename P::CElem *Cl;
    int rpm, nrhs;
    typename P::R mass4[MAXM];
    const typename P::CElem *Ainv[MAXM];
    int blk0;
    double tol2;
    const double *tol2_dev = nullptr;  // if set, the tolerance is read from device memory (captured graphs)
    int maxiter;
    int *stat;  // [0] max iterations, [1] blocks that missed the tolerance
};

// One cluster of C CTAs owns one (block, right-hand side) pair and runs the whole even-odd BiCGStab on
// it; CTA q of the cluster holds the q-th part of the block's sites in time (BL / C time slices of
// each parity), one even and one odd site per thread.
//
// What bounds it: the eight-neighbour gathers.  With the vectors in global memory (one CTA per block, the
// six vectors of an 8^4 block 1.2 MB) the kernel waited on L2: 27 % of the issue slots, 16 MB through
// L1 and L2 per iteration against 9.7 TB/s of L2 bandwidth for the whole chip, and its sums and scalars
// in FP64 on every warp took a fifth of the time (GB300 issues FP64 at 1/64 of its FP32 rate).  So
//   * the two vectors that are gathered from -- G (p, then s) on the even sites, T (A_oo^-1 H_oe G) on
//     the odd ones -- live in the cluster's shared memory, and a time hop into the neighbouring CTA's
//     part reads distributed shared memory.  The others are read and written once by the thread that
//     owns the site: v and t stay in registers over the reduction that follows them;
//   * inner products are summed in float pairs (RunSum), and one thread of each CTA does the FP64
//     scalars;
//   * more CTAs per block than one also spread a small lattice over the chip: an FP64 solve of
//     the 8 blocks of 4^4 sites of one colour with 4 right-hand sides kept 32 SMs busy, now 128.

constexpr int BLK_KMAX = 7;  // inner products of one reduction

template <class P, int BL, int C> struct BlkShape {
    static constexpr int HL = BlockShape<BL>::VBH / C;  // sites of one parity per CTA
    // 16-byte elements of one vector of the CTA
    static constexpr int FE = P::ID == 64 ? 12 * HL : P::ID == 32 ? 6 * HL : 3 * HL + (HL + 3) / 4;
    static constexpr size_t SMEM = (size_t)2 * FE * 16;  // G and T of one right-hand side
};

template <int C> __device__ __forceinline__ void blk_sync()
{
    if constexpr (C == 1) __syncthreads();
    else cooperative_groups::this_cluster().sync();
}

// acc += the hop of direction MU, DIR (forward: (1 - g) U(s) F(s + mu), backward: (1 + g) U(s - mu)^dag
// F(s - mu)) of the site with in-block coordinates c, half index h and internal index s, if it
// stays inside the block.  F: the other parity's part of the vector held by this CTA (q).
template <class P, int BL, int C, int MU, int DIR>
__device__ __forceinline__ void hop_shared(const int (&c)[4], int lb, int s, int nbase, int q, int V,
                                           const typename P::SElem *F, const typename P::UElem *__restrict__ U,
                                           Spinor<typename P::R> &acc)
{
    using R = typename P::R;
    constexpr int HL = BlkShape<P, BL, C>::HL;
    constexpr int STEP = MU == 0 ? BL * BL * BL : MU == 1 ? BL * BL : MU == 2 ? BL : 1;
    if (DIR > 0 ? c[MU] == BL - 1 : c[MU] == 0) return;
    const int hn = (lb + DIR * STEP) >> 1;  // half index of the neighbour in the block
    Link<R> L;
    P::load_link(U, V, MU, DIR > 0 ? s : nbase + hn, L);
    Spinor<R> p;
    const int own = hn - q * HL;
    if (C == 1 || MU != 0 || (own >= 0 && own < HL)) {
        P::load_spinor_rw(F, HL, own, p);
    } else {
        const int q2 = q + DIR;
        P::load_spinor_rw(cooperative_groups::this_cluster().map_shared_rank(F, q2), HL, hn - q2 * HL, p);
    }
    Half<R> h, w;
    project<MU, -DIR>(p, h);
    if constexpr (sizeof(R) == 4) link_mul_packed<(DIR < 0)>(L, h, w);
    else if (DIR > 0) link_mul(L, h, w);
    else link_dag_mul(L, h, w);
    reconstruct_add<MU, -DIR>(acc, w);
}

// shared scratch of the reductions: per warp, and per CTA of the cluster (two sets used in turn)
template <typename R, int C, int NT> struct BlkRed {
    typename RunSum<R>::Raw warp[NT / 32][BLK_KMAX], tot[2][C][BLK_KMAX];
};

// K totals over the cluster, in out[] of thread 0 of every CTA (the same bits in each).  Every thread of
// the cluster takes part.  With C > 1 it ends with a cluster barrier.
template <int K, int NT, int C, typename R>
__device__ __forceinline__ void cluster_totals(RunSum<R> (&v)[K], double (&out)[K], BlkRed<R, C, NT> &red, int &buf, int q)
{
    using Raw = typename RunSum<R>::Raw;
    constexpr int NW = NT / 32, W2 = NW <= 1 ? 1 : NW <= 2 ? 2 : NW <= 4 ? 4 : NW <= 8 ? 8 : 16;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    using WS = WarpSums<K, R>;
    {
        const RunSum<R> t = WS::total(v);
        const int k = lane >> WS::SHIFT;
        if ((lane & ((1 << WS::SHIFT) - 1)) == 0 && k < K) red.warp[w][k] = t.raw();
    }
    if (NW == 1) {
        __syncwarp();
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; k++) {
                v[k] = RunSum<R>();
                v[k].join(red.warp[0][k]);
            }
    } else {
        __syncthreads();
        if (w == 0)
#pragma unroll
            for (int k = 0; k < K; k++) {
                v[k] = RunSum<R>();
                if (lane < NW) v[k].join(red.warp[lane][k]);
                v[k].template shuffle_sum<W2>();
            }
    }
    if constexpr (C > 1) {
        auto cl = cooperative_groups::this_cluster();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int j = 0; j < C; j++) {
                Raw *d = cl.map_shared_rank(&red.tot[buf][q][0], j);
#pragma unroll
                for (int k = 0; k < K; k++) d[k] = v[k].raw();
            }
        }
        cl.sync();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                v[k] = RunSum<R>();
#pragma unroll
                for (int j = 0; j < C; j++) v[k].join(red.tot[buf][j][k]);
            }
        }
        buf ^= 1;
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < K; k++) out[k] = v[k].value();
}

// FP32 arithmetic: at most 128 registers, so that 512 threads fit an SM
template <class P, int BL, int C, int NT>
__global__ void __launch_bounds__(NT, sizeof(typename P::R) == 4 ? 512 / NT : 1) k_block_solve(GeomDev g, BlkArgs<P> a)
{
    using R = typename P::R;
    using E = typename P::SElem;
    constexpr int VBH = BlockShape<BL>::VBH, HL = BlkShape<P, BL, C>::HL;
    static_assert(HL <= NT && BL % C == 0 && NT % 32 == 0, "one site of each parity per thread, whole time slices per CTA");
    extern __shared__ __align__(16) unsigned char blk_smem[];
    __shared__ BlkRed<R, C, NT> red;
    __shared__ R scal[6];   // alpha, omega, beta
    __shared__ double fs[5]; // thread 0's FP64 scalars: rho, alpha, the threshold of ||r||^2
    __shared__ int live;    // 0 once converged or broken down
    E *G = reinterpret_cast<E *>(blk_smem), *T = G + BlkShape<P, BL, C>::FE;
    const int q = C == 1 ? 0 : (int)(blockIdx.x % C), id = C == 1 ? (int)blockIdx.x : (int)(blockIdx.x / C);
    // right-hand side fastest: the clusters of one block run together and share its links in L2
    const int rhs = id % a.nrhs, blk = a.blk0 + id / a.nrhs;
    const long ro = (long)rhs * a.rstride;
    const int slot = rhs / a.rpm;
    const R mass4 = a.mass4[slot];
    const typename P::CElem *Ainv = a.Ainv[slot];
    const int V = (int)g.V, vh = (int)g.vh;

    const bool act = (int)threadIdx.x < HL;
    const int hl = act ? threadIdx.x : 0;  // site of either parity: own slot
    const int be = blk * VBH, bo = vh + be;

    double &rho_x = fs[0], &rho_y = fs[1], &al_x = fs[2], &al_y = fs[3], &thresh = fs[4];
    int it = 0, buf = 0;
    bool ok = false;
    // the solution becomes the gather source of the odd sites
    auto finish = [&](int se) {
        if (act) {
            Spinor<R> s;
            P::load_spinor_rw(a.x + ro, V, se, s);
            P::store_spinor(G, HL, hl, s);
        }
    };
    // the passes of the loop: start (btil, r = rh = p), v = S p, t = S s, and the odd sites of x
    enum { START, V_OF_P, T_OF_S, FINISH };
    int stage = START;
    while (true) {
        // index in the block, opaque to the compiler: the neighbours' addresses are cheaper to form again in
        // every pass than to keep in registers (or spill) across the loop
        int h = q * HL + hl;
        asm volatile("" : "+r"(h));
        const int se = be + h, so = bo + h;
        int c[4];  // in-block coordinates; z depends on the parity
        int zr = h / (BL / 2);
        const int z0 = 2 * (h - zr * (BL / 2));
        c[2] = zr % BL;
        zr /= BL;
        c[1] = zr % BL;
        c[0] = zr / BL;
        const int odd_row = (c[0] + c[1] + c[2]) & 1;
        if (act) {
            // ---- odd site:  T = A_oo^-1 ( y + coef H_oe G ),  y = b_o at the start and the end
            Spinor<R> acc;
            zero(acc);
            if (stage != START) {
                c[3] = z0 + (odd_row ^ 1);
                const int lb = 2 * h + (c[3] & 1);
                hop_shared<P, BL, C, 0, +1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 0, -1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 1, +1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 1, -1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 2, +1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 2, -1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 3, +1>(c, lb, so, be, q, V, G, a.U, acc);
                hop_shared<P, BL, C, 3, -1>(c, lb, so, be, q, V, G, a.U, acc);
            }
            if (stage == START || stage == FINISH) {
                Spinor<R> y;
                P::load_spinor(a.b + ro, V, so, y);
                if (stage == FINISH) scale(acc, R(0.5));
                axpy(acc, R(1), y);
            }
            clover_apply<P>(Ainv, V, so, R(0), acc);
            if (stage == FINISH) P::store_spinor(a.x + ro, V, so, acc);
            else P::store_spinor(T, HL, hl, acc);
        }
        if (stage == FINISH) break;
        blk_sync<C>();
        // ---- even site:  acc = D own + coef H_eo T  (D = 1, coef 1/2 at the start; A(m), -1/4 after)
        Spinor<R> acc;
        zero(acc);
        if (act) {
            c[3] = z0 + odd_row;
            const int lb = 2 * h + (c[3] & 1);
            hop_shared<P, BL, C, 0, +1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 0, -1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 1, +1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 1, -1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 2, +1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 2, -1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 3, +1>(c, lb, se, bo, q, V, T, a.U, acc);
            hop_shared<P, BL, C, 3, -1>(c, lb, se, bo, q, V, T, a.U, acc);
            scale(acc, stage == START ? R(0.5) : R(-0.25));
            Spinor<R> own;
            if (stage == START) {
                P::load_spinor(a.b + ro, V, se, own);
            } else {
                P::load_spinor_rw(G, HL, hl, own);
                clover_apply<P>(a.Cl, V, se, mass4, own);
            }
            axpy(acc, R(1), own);
        }
        if (stage == V_OF_P) {
            // (rh, v) and rho = (rh, r): the difference that beta is formed with is rounded relative to |s|
            RunSum<R> d[4];
            Spinor<R> s;
            if (act) {
                Spinor<R> w;
                P::load_spinor_rw(a.rh + ro, V, se, w);
                P::load_spinor_rw(a.r + ro, V, se, s);
                SiteDot<R> z, y;
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    z.add(k, w.v[k / 3][k % 3], acc.v[k / 3][k % 3]);
                    y.add(k, w.v[k / 3][k % 3], s.v[k / 3][k % 3]);
                }
                d[0].add(z.total().re);
                d[1].add(z.total().im);
                d[2].add(y.total().re);
                d[3].add(y.total().im);
                P::store_spinor(a.v + ro, V, se, acc);
            }
            double o[4];
            cluster_totals<4, NT, C, R>(d, o, red, buf, q);
            if (threadIdx.x == 0) {  // alpha = rho / (rh, v); a zero or NaN is a breakdown: x as it is
                rho_x = o[2];
                rho_y = o[3];
                const double den = o[0] * o[0] + o[1] * o[1];
                live = !(den == 0.0 || !(den == den));
                const double iv = 1.0 / den;
                al_x = (rho_x * o[0] + rho_y * o[1]) * iv;
                al_y = (rho_y * o[0] - rho_x * o[1]) * iv;
                scal[0] = R(al_x);
                scal[1] = R(al_y);
            }
            __syncthreads();
            if (!live) {
                finish(se);
                stage = FINISH;
            } else {
                if (act) {  // s = r - alpha v
                    const cpx<R> al = {scal[0], scal[1]};
#pragma unroll
                    for (int k = 0; k < 12; k++) cmsub(s.v[k / 3][k % 3], al, acc.v[k / 3][k % 3]);
                    P::store_spinor(G, HL, hl, s);
                }
                stage = T_OF_S;
            }
            blk_sync<C>();
            continue;
        }
        // r = rh = p at the start; the end of an iteration after t
        RunSum<R> rr[2];  // ||r||^2 and, at the start, ||b||^2
        if (stage == START) {
            if (act) {
                SiteNorm<R> n, be2, bo2;
                Spinor<R> o;
#pragma unroll
                for (int k = 0; k < 12; k++) n.add(k, acc.v[k / 3][k % 3]);
                P::load_spinor(a.b + ro, V, se, o);
#pragma unroll
                for (int k = 0; k < 12; k++) be2.add(k, o.v[k / 3][k % 3]);
                P::load_spinor(a.b + ro, V, so, o);
#pragma unroll
                for (int k = 0; k < 12; k++) bo2.add(k, o.v[k / 3][k % 3]);
                rr[0].add(n.total());
                rr[1].add(be2.total());
                rr[1].add(bo2.total());
                P::store_spinor(a.r + ro, V, se, acc);
                P::store_spinor(a.rh + ro, V, se, acc);
                P::store_spinor(a.p + ro, V, se, acc);
                P::store_spinor(G, HL, hl, acc);
                zero(acc);
                P::store_spinor(a.x + ro, V, se, acc);
            }
        } else {
            RunSum<R> d[7];
            if (act) {
                Spinor<R> w;
                P::load_spinor_rw(G, HL, hl, w);
                SiteDot<R> ts, hs, ht;
                SiteNorm<R> tt;
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    const cpx<R> z = acc.v[k / 3][k % 3];
                    ts.add(k, z, w.v[k / 3][k % 3]);
                    tt.add(k, z);
                }
                Spinor<R> hh;
                P::load_spinor_rw(a.rh + ro, V, se, hh);
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    hs.add(k, hh.v[k / 3][k % 3], w.v[k / 3][k % 3]);
                    ht.add(k, hh.v[k / 3][k % 3], acc.v[k / 3][k % 3]);
                }
                d[0].add(ts.total().re);
                d[1].add(ts.total().im);
                d[2].add(tt.total());
                d[3].add(hs.total().re);
                d[4].add(hs.total().im);
                d[5].add(ht.total().re);
                d[6].add(ht.total().im);
            }
            double o[7];
            cluster_totals<7, NT, C, R>(d, o, red, buf, q);
            if (threadIdx.x == 0) {
                // omega = (t, s) / (t, t), rho' = (rh, s) - omega (rh, t), beta = rho' alpha / (rho omega); a zero
                // denominator (rho = 0) ends the recurrence after this iteration
                const double tt = o[2];
                const bool go = !(tt == 0.0 || !(tt == tt));
                live = go;
                const double iv = go ? 1.0 / tt : 0.0;
                const double ox = o[0] * iv, oy = o[1] * iv;
                const double rx = o[3] - (ox * o[5] - oy * o[6]), ry = o[4] - (ox * o[6] + oy * o[5]);
                const double nx = rx * al_x - ry * al_y, ny = rx * al_y + ry * al_x;
                const double dx = rho_x * ox - rho_y * oy, dy = rho_x * oy + rho_y * ox;
                const double d2 = dx * dx + dy * dy, jv = d2 > 0.0 ? 1.0 / d2 : 0.0;
                scal[2] = R(ox);
                scal[3] = R(oy);
                scal[4] = R((nx * dx + ny * dy) * jv);
                scal[5] = R((ny * dx - nx * dy) * jv);
                rho_x = d2 > 0.0 ? rx : 0.0;
                rho_y = d2 > 0.0 ? ry : 0.0;
            }
            __syncthreads();
            if (!live) {
                finish(se);
                stage = FINISH;
                blk_sync<C>();
                continue;
            }
            if (act) {  // x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v)
                const cpx<R> al = {scal[0], scal[1]}, om = {scal[2], scal[3]}, bt = {scal[4], scal[5]};
                Spinor<R> s, pv, y;
                P::load_spinor_rw(G, HL, hl, s);
                P::load_spinor_rw(a.p + ro, V, se, pv);
                P::load_spinor_rw(a.x + ro, V, se, y);
                SiteNorm<R> n;
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    cpx<R> &sk = s.v[k / 3][k % 3], &xk = y.v[k / 3][k % 3];
                    cmac(xk, al, pv.v[k / 3][k % 3]);
                    cmac(xk, om, sk);
                    cmsub(sk, om, acc.v[k / 3][k % 3]);
                    n.add(k, sk);
                }
                P::store_spinor(a.x + ro, V, se, y);
                P::store_spinor(a.r + ro, V, se, s);
                P::load_spinor_rw(a.v + ro, V, se, y);
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    cpx<R> &pk = pv.v[k / 3][k % 3];
                    cmsub(pk, om, y.v[k / 3][k % 3]);
                    cmac(s.v[k / 3][k % 3], bt, pk);
                }
                P::store_spinor(a.p + ro, V, se, s);
                P::store_spinor(G, HL, hl, s);
                rr[0].add(n.total());
            }
            it++;
        }
        double o[2];
        cluster_totals<2, NT, C, R>(rr, o, red, buf, q);
        if (threadIdx.x == 0) {
            if (stage == START) {
                thresh = (a.tol2_dev ? *a.tol2_dev : a.tol2) * o[1];
                rho_x = o[0];
                rho_y = 0.0;
            }
            ok = o[0] <= thresh;
            const bool dead = !(o[0] == o[0]) || it >= a.maxiter || (rho_x == 0.0 && rho_y == 0.0);
            live = !ok && !dead;
        }
        __syncthreads();
        stage = V_OF_P;
        if (!live) {
            finish(se);
            stage = FINISH;
            blk_sync<C>();
        }
    }
    if (threadIdx.x == 0 && q == 0) {
        atomicMax(a.stat, it);
        if (!ok) atomicAdd(a.stat + 1, 1);
    }
    blk_sync<C>();  // no CTA leaves while another may read its part
}

// ---- FP64, eight lanes per site (split64.cuh), for 2^4 and 4^4 blocks.  With one thread per site a warp's
// chain of FP64 instructions takes 180 us per iteration, whether it has an SM to itself (8 blocks of 4^4
// sites and 4 right-hand sides: 128 CTAs of one warp) or shares it with three others; a 2^4 block fills
// 8 of a warp's 32 lanes.  Here lane u does hop u, then its share of spin u & 3; the Krylov vectors stay in
// registers for the whole solve (lane (al, q) owns colours 0, 1 of spin al for q = 0, colour 2 for q = 1).
// ms per launch of a colour, one thread per site / split: 8^4 in 4^4 blocks, 4 right-hand sides 3.47 / 1.42,
// 16 right-hand sides 3.64 / 5.58, 16^4, 4 right-hand sides 13.1 / 20.5 (block_form chooses).
template <int BL, int C> struct SplitShape {
    static constexpr int HL = BlockShape<BL>::VBH / C, NT = 8 * HL;
    static constexpr size_t SMEM = (size_t)HL * (2 * 12 + 48) * sizeof(double2);  // G, T, the half spinors
};

template <int BL, int C>
__global__ void __launch_bounds__(SplitShape<BL, C>::NT) k_block_split(GeomDev g, BlkArgs<PrecD> a)
{
    constexpr int VBH = BlockShape<BL>::VBH, HL = SplitShape<BL, C>::HL, NT = SplitShape<BL, C>::NT;
    static_assert(HL % 4 == 0 && BL % C == 0, "whole warps, whole time slices per CTA");
    extern __shared__ __align__(16) unsigned char blk_smem[];
    __shared__ BlkRed<double, C, NT> red;
    __shared__ double scal[6], fs[5];
    __shared__ int live;
    double2 *G = reinterpret_cast<double2 *>(blk_smem), *T = G + 12 * HL;  // [site][12]
    const int q = C == 1 ? 0 : (int)(blockIdx.x % C), id = C == 1 ? (int)blockIdx.x : (int)(blockIdx.x / C);
    const int rhs = id % a.nrhs, blk = a.blk0 + id / a.nrhs;
    const long ro = (long)rhs * a.rstride, V = g.V;
    const int slot = rhs / a.rpm;
    const double mass4 = a.mass4[slot];
    const double2 *Ainv = a.Ainv[slot];

    const int u = threadIdx.x & 7, al = u & 3, hf = u >> 2, hl = threadIdx.x >> 3, h = q * HL + hl;
    double2 *w = T + 12 * HL + hl * 48;  // [hop][6]
    const long be = (long)blk * VBH, bo = g.vh + be, se = be + h, so = bo + h;
    const int mu = u >> 1;
    const bool fwd = (u & 1) == 0;
    // coordinate and half-index step of this lane's hop, for each parity of the output site
    int zr = h / (BL / 2);
    const int z0 = 2 * (h - zr * (BL / 2)), cy = zr % BL, cx = (zr / BL) % BL, ct = zr / (BL * BL);
    const int odd_row = (ct + cx + cy) & 1;

    // this lane's hop into the site of parity par, gathered from F, then its share of the hop sum
    auto hops = [&](int par, const double2 *F, cpx<double> (&o)[3]) {
        const int cz = z0 + (odd_row ^ par), cm = mu == 0 ? ct : mu == 1 ? cx : mu == 2 ? cy : cz;
        const int step = mu == 0 ? BL * BL * BL : mu == 1 ? BL * BL : mu == 2 ? BL : 1;
        Half<double> hw;
        if (fwd ? cm < BL - 1 : cm > 0) {
            const int hn = (2 * h + (cz & 1) + (fwd ? step : -step)) >> 1;
            const long s = par ? so : se, sn = (par ? be : bo) + hn;
            const int own = hn - q * HL;
            const double2 *src = F + 12 * own;
            if (C > 1 && (own < 0 || own >= HL)) {
                const int q2 = own < 0 ? q - 1 : q + 1;
                src = cooperative_groups::this_cluster().map_shared_rank(F, q2) + 12 * (hn - q2 * HL);
            }
            split_hop(src, 1, a.U + (long)mu * 9 * V + (fwd ? s : sn), V, mu, fwd, hw);
        } else {
#pragma unroll
            for (int k = 0; k < 6; k++) hw.v[k / 3][k % 3] = {0.0, 0.0};
        }
#pragma unroll
        for (int k = 0; k < 6; k++) w[u * 6 + k] = make_double2(hw.v[k / 3][k % 3].re, hw.v[k / 3][k % 3].im);
        __syncwarp();
        split_sum(w, al, hf, o);
        __syncwarp();
    };
    // the two components a lane owns (the second is zero for hf = 1), and back to shared memory
    const int k0 = 3 * al + 2 * hf;
    auto own2 = [&](const cpx<double> (&o)[3], cpx<double> (&e)[2]) {
        e[0] = hf ? o[2] : o[0];
        e[1] = hf ? cpx<double>{0.0, 0.0} : o[1];
    };
    auto put = [&](double2 *F, const cpx<double> (&e)[2]) {
        F[12 * hl + k0] = make_double2(e[0].re, e[0].im);
        if (!hf) F[12 * hl + k0 + 1] = make_double2(e[1].re, e[1].im);
    };
    auto put_global = [&](double2 *f, long s, const cpx<double> (&e)[2]) {
        f[(long)k0 * V + s] = make_double2(e[0].re, e[0].im);
        if (!hf) f[(long)(k0 + 1) * V + s] = make_double2(e[1].re, e[1].im);
    };
    auto add_b = [&](long s, cpx<double> (&o)[3]) {  // by one lane of a spin, before the halves join
        if (hf == 0)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const double2 t = __ldg(a.b + ro + (long)(3 * al + c) * V + s);
                o[c].re += t.x;
                o[c].im += t.y;
            }
    };

    double &rho_x = fs[0], &rho_y = fs[1], &al_x = fs[2], &al_y = fs[3], &thresh = fs[4];
    int it = 0, buf = 0;
    bool ok = false;
    cpx<double> x[2] = {{0.0, 0.0}, {0.0, 0.0}}, r[2], rh[2], p[2], v[2], s[2];
    enum { START, V_OF_P, T_OF_S, FINISH };
    int stage = START;
    while (true) {
        cpx<double> o[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}}, f3[3], e[2];
        // ---- odd site:  T = A_oo^-1 ( y + coef H_oe G )
        if (stage != START) hops(1, G, o);
        if (stage == FINISH)
#pragma unroll
            for (int c = 0; c < 3; c++) o[c] = 0.5 * o[c];
        if (stage == START || stage == FINISH) add_b(so, o);
        split_join(o);
        split_fetch(o, al, hf, f3);
        split_herm(Ainv + so, V, al, hf, 0.0, f3, o);
        split_join(o);
        own2(o, e);
        if (stage == FINISH) {
            put_global(a.x + ro, so, e);
            break;
        }
        put(T, e);
        blk_sync<C>();
        // ---- even site
        hops(0, T, o);
        const double coef = stage == START ? 0.5 : -0.25;
#pragma unroll
        for (int c = 0; c < 3; c++) o[c] = coef * o[c];
        if (stage == START) {
            add_b(se, o);
        } else {
            cpx<double> d[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const double2 t = G[12 * hl + 3 * ((al & 2) + hf) + c];
                f3[c] = {t.x, t.y};
            }
            split_herm(a.Cl + se, V, al, hf, mass4, f3, d);
#pragma unroll
            for (int c = 0; c < 3; c++) o[c] = o[c] + d[c];
        }
        split_join(o);
        own2(o, e);
        if (stage == V_OF_P) {
            RunSum<double> d[4];  // (rh, v) and rho = (rh, r)
            cpx<double> z = {0.0, 0.0}, y = {0.0, 0.0};
#pragma unroll
            for (int k = 0; k < 2; k++) {
                v[k] = e[k];
                cmacc(z, rh[k], v[k]);
                cmacc(y, rh[k], r[k]);
            }
            d[0].s = z.re;
            d[1].s = z.im;
            d[2].s = y.re;
            d[3].s = y.im;
            double t[4];
            cluster_totals<4, NT, C, double>(d, t, red, buf, q);
            if (threadIdx.x == 0) {  // alpha = rho / (rh, v); a zero or NaN is a breakdown: x as it is
                rho_x = t[2];
                rho_y = t[3];
                const double den = t[0] * t[0] + t[1] * t[1];
                live = !(den == 0.0 || !(den == den));
                const double iv = 1.0 / den;
                scal[0] = al_x = (rho_x * t[0] + rho_y * t[1]) * iv;
                scal[1] = al_y = (rho_y * t[0] - rho_x * t[1]) * iv;
            }
            __syncthreads();
            if (!live) {
                put(G, x);
                stage = FINISH;
            } else {  // s = r - alpha v
                const cpx<double> alp = {scal[0], scal[1]};
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    s[k] = r[k];
                    cmsub(s[k], alp, v[k]);
                }
                put(G, s);
                stage = T_OF_S;
            }
            blk_sync<C>();
            continue;
        }
        RunSum<double> rr[2];  // ||r||^2 and, at the start, ||b||^2
        if (stage == START) {
            double n = 0, nb = 0;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                r[k] = rh[k] = p[k] = e[k];
                n = fma(e[k].re, e[k].re, fma(e[k].im, e[k].im, n));
                if (k == 0 || !hf) {
                    const double2 t0 = __ldg(a.b + ro + (long)(k0 + k) * V + se), t1 = __ldg(a.b + ro + (long)(k0 + k) * V + so);
                    nb = fma(t0.x, t0.x, fma(t0.y, t0.y, fma(t1.x, t1.x, fma(t1.y, t1.y, nb))));
                }
            }
            rr[0].s = n;
            rr[1].s = nb;
            put(G, p);
        } else {
            RunSum<double> d[7];
            cpx<double> ts = {0.0, 0.0}, hs = {0.0, 0.0}, ht = {0.0, 0.0};
            double tt = 0;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                cmacc(ts, e[k], s[k]);
                tt = fma(e[k].re, e[k].re, fma(e[k].im, e[k].im, tt));
                cmacc(hs, rh[k], s[k]);
                cmacc(ht, rh[k], e[k]);
            }
            d[0].s = ts.re;
            d[1].s = ts.im;
            d[2].s = tt;
            d[3].s = hs.re;
            d[4].s = hs.im;
            d[5].s = ht.re;
            d[6].s = ht.im;
            double t[7];
            cluster_totals<7, NT, C, double>(d, t, red, buf, q);
            if (threadIdx.x == 0) {  // as in k_block_solve
                const double n2 = t[2];
                const bool go = !(n2 == 0.0 || !(n2 == n2));
                live = go;
                const double iv = go ? 1.0 / n2 : 0.0;
                const double ox = t[0] * iv, oy = t[1] * iv;
                const double rx = t[3] - (ox * t[5] - oy * t[6]), ry = t[4] - (ox * t[6] + oy * t[5]);
                const double nx = rx * al_x - ry * al_y, ny = rx * al_y + ry * al_x;
                const double dx = rho_x * ox - rho_y * oy, dy = rho_x * oy + rho_y * ox;
                const double d2 = dx * dx + dy * dy, jv = d2 > 0.0 ? 1.0 / d2 : 0.0;
                scal[2] = ox;
                scal[3] = oy;
                scal[4] = (nx * dx + ny * dy) * jv;
                scal[5] = (ny * dx - nx * dy) * jv;
                rho_x = d2 > 0.0 ? rx : 0.0;
                rho_y = d2 > 0.0 ? ry : 0.0;
            }
            __syncthreads();
            if (!live) {
                put(G, x);
                stage = FINISH;
                blk_sync<C>();
                continue;
            }
            // x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v)
            const cpx<double> alp = {scal[0], scal[1]}, om = {scal[2], scal[3]}, bt = {scal[4], scal[5]};
            double n = 0;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                cmac(x[k], alp, p[k]);
                cmac(x[k], om, s[k]);
                r[k] = s[k];
                cmsub(r[k], om, e[k]);
                n = fma(r[k].re, r[k].re, fma(r[k].im, r[k].im, n));
                cmsub(p[k], om, v[k]);
                cpx<double> pn = r[k];
                cmac(pn, bt, p[k]);
                p[k] = pn;
            }
            put(G, p);
            rr[0].s = n;
            it++;
        }
        double t[2];
        cluster_totals<2, NT, C, double>(rr, t, red, buf, q);
        if (threadIdx.x == 0) {
            if (stage == START) {
                thresh = (a.tol2_dev ? *a.tol2_dev : a.tol2) * t[1];
                rho_x = t[0];
                rho_y = 0.0;
            }
            ok = t[0] <= thresh;
            const bool dead = !(t[0] == t[0]) || it >= a.maxiter || (rho_x == 0.0 && rho_y == 0.0);
            live = !ok && !dead;
        }
        __syncthreads();
        stage = V_OF_P;
        if (!live) {
            put(G, x);
            stage = FINISH;
            blk_sync<C>();
        }
    }
    put_global(a.x + ro, se, x);
    if (threadIdx.x == 0 && q == 0) {
        atomicMax(a.stat, it);
        if (!ok) atomicAdd(a.stat + 1, 1);
    }
    blk_sync<C>();  // no CTA leaves while another may read its part
}

// Launch shapes: C CTAs of NT threads per block and right-hand side.  Form 0 is the wider CTA, form 1 the
// smaller one (more CTAs for few blocks and right-hand sides, more distributed-memory hops).
// Measured on FP32 storage, ms per launch of a colour, form 0 / form 1 / the kernel with its vectors in
// global memory: 24x12^3 in 6^4 blocks, 5 right-hand sides 0.38 / 0.40 / 1.07; 16^4 in 4^4 blocks, 16
// right-hand sides 0.85 / 1.57 / 1.54; 32x16^3 in 8^4 blocks, 24 right-hand sides 5.5 / 6.2; 48x24^3 in 6^4
// blocks, 6 right-hand sides 5.8 / 6.3 / 9.1; 64x32^3 in 8^4 blocks, 4 right-hand sides 14.9 / 25.2 (form 0 / global).
// What bounds it now is waiting at 16 warps per SM (8^4 blocks, 16 right-hand sides: of 10.4 cycles between
// a warp's instructions 2.4 at cluster barriers and 2.2 for loads; issue 0.33, L1 0.45, L2 0.24 of their
// rates).  Two or four right-hand sides in a CTA, to share the links through L1, lost (22.8 ms on
// 64x32^3, 4 right-hand sides): their barriers couple them.
template <int BL> struct BlkForms;
template <> struct BlkForms<2> { static constexpr int C[2] = {1, 1}, N[2] = {32, 32}; };
template <> struct BlkForms<4> { static constexpr int C[2] = {1, 4}, N[2] = {128, 32}; };
template <> struct BlkForms<6> { static constexpr int C[2] = {3, 6}, N[2] = {224, 128}; };
template <> struct BlkForms<8> { static constexpr int C[2] = {4, 8}, N[2] = {512, 256}; };

// The form of a launch of n clusters (blocks of a colour times right-hand sides): a rule on sizes, so that every
// context, captured or not, adds in the same order and no launch is spent on timing.  One GB300, ms
// per launch with near-unit links.
//   * 4^4 blocks, 32- and 16-bit storage: form 0 at every size (8 clusters 0.149 / 0.191, 2048 0.85 / 1.57).
//   * 6^4 and 8^4, 32- and 16-bit: form 1 while its CTAs have SMs to themselves (6^4: 8 clusters 0.315 / 0.291, 16 0.300 /
//     0.284, 24 0.314 / 0.316; 8^4: 8 0.518 / 0.456, 16 0.537 / 0.524, 24 0.553 / 0.587), then form 0 (at most
//     3 % behind in FP32, 7 % in 16-bit storage, where its last wave is short).
//   * FP64, where a CTA has an SM to itself and a launch takes whole waves of clusters.  6^4: form 0 runs 45
//     clusters per wave of 7.9 ms, form 1 22 of 4.5 (16 clusters 8.2 / 5.0, 40 8.2 / 9.2, 64 15.9 / 13.4, 80 16.2 /
//     18.6); 8^4: 34 of 22.5 ms and 15 of 11.4 (8 clusters 23.0 / 11.9, 32 23.1 / 34.3, 40 44.7 / 34.7).
//     4^4: eight lanes per site (form 2) take waves of 36 clusters of 1.3 ms, form 0 of 152 of 3.3 (64
//     clusters 3.29 / 2.61, 80 3.46 / 3.79); form 1, four CTAs of a warp, fills the SMs that form 0's second wave
//     leaves idle (160 clusters 6.0 / 5.0, 192 6.0 to 6.2 / 5.4 to 5.7, 256 6.2 / 7.3 to 7.9).
inline int block_form(int id, int bl, long n)
{
    if (bl == 2) return 0;
    if (id != 64) return bl != 4 && n <= 16;
    if (bl == 4) return n <= 72 ? 2 : n > 152 && n <= 200 ? 1 : 0;
    const long per0 = bl == 6 ? 45 : 34, per1 = bl == 6 ? 22 : 15;
    const double t0 = bl == 6 ? 7.9 : 22.5, t1 = bl == 6 ? 4.5 : 11.4;
    return t1 * (double)((n + per1 - 1) / per1) < t0 * (double)((n + per0 - 1) / per0);
}

template <class P>
void launch_clusters(ddrw_ctx *ctx, void (*kernel)(GeomDev, BlkArgs<P>), int C, int NT, size_t smem, const BlkArgs<P> &a,
                     int nrhs)
{
    BlkArgs<P> b = a;
    b.nrhs = nrhs;
    if (smem > 40 * 1024)  // (static shared memory counts towards the default limit of 48 KB)
        cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((long)C * nrhs * ctx->nblk_c));
    lc.blockDim = dim3(NT);
    lc.dynamicSmemBytes = smem;
    lc.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = C > 1 ? 1 : 0;
    ++ctx->launches;
    cudaLaunchKernelEx(&lc, kernel, geom_dev(ctx), b);
}

template <class P, int BL, int C, int NT>
void launch_block_shape(ddrw_ctx *ctx, const BlkArgs<P> &a, int nrhs)
{
    launch_clusters<P>(ctx, k_block_solve<P, BL, C, NT>, C, NT, BlkShape<P, BL, C>::SMEM, a, nrhs);
}

template <class P, int BL>
void launch_block_kernel(ddrw_ctx *ctx, const BlkArgs<P> &a, int nrhs)
{
    using F = BlkForms<BL>;
    // pinned (ddrw_block_config), else by size
    const int form = ctx->blk_form >= 0 ? ctx->blk_form : block_form(P::ID, BL, (long)ctx->nblk_c * nrhs);
    ProfScope ps(ctx, P::ID == 64 ? PROF_BLOCK64 : P::ID == 32 ? PROF_BLOCK32 : PROF_BLOCK16, 0.0);
    if constexpr (P::ID == 64 && BL == 2) {
        launch_clusters<P>(ctx, k_block_split<2, 1>, 1, SplitShape<2, 1>::NT, SplitShape<2, 1>::SMEM, a, nrhs);
    } else {
        if constexpr (P::ID == 64 && BL == 4) {
            if (form == 2) {
                launch_clusters<P>(ctx, k_block_split<4, 4>, 4, SplitShape<4, 4>::NT, SplitShape<4, 4>::SMEM, a, nrhs);
                return;
            }
        }
        if (BL > 2 && form) launch_block_shape<P, BL, F::C[1], F::N[1]>(ctx, a, nrhs);
        else launch_block_shape<P, BL, F::C[0], F::N[0]>(ctx, a, nrhs);
    }
}

}  // namespace ddrw
