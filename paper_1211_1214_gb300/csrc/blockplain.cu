// blockplain.cu -- the FP32 block solver with one CTA per block and right-hand side, for the adjoint force.
//
// The force of one noise vector is the difference of two nearly equal terms (target masses m1 and m2), which
// magnifies what the block solves leave behind a hundredfold: at a block tolerance of 1e-11 a force is known to
// 1e-9, and another order of the sums gives another, equally good one 1.3e-9 away (either is 1.1e-9 from
// the exact one).  The FP32 block solves of the force keep this kernel's order of operations, so that its results
// stay within that distance of those of earlier versions; it makes them no more exact.  FP64 block solves,
// 16-bit ones (ddrw_set_low_precision) and block method 1 (ddrw_set_block_solver) take the
// solvers they take elsewhere, whose order follows from the sizes.  It costs a tenth of the force (16^4, 4^4
// blocks, 4 noise vectors: 39.7 ms, with the cluster kernel of blocksolve.cuh 35.9).
//
// One CTA of NT threads owns one (block, right-hand side) pair and runs the whole even-odd BiCGStab with the
// vectors in global memory; it waits on L2.
#include "blocksolve.cuh"

namespace ddrw {

namespace {

template <class P> struct PlainArgs : BlkArgs<P> {
    typename P::SElem *t, *tmp;
};

template <int K, int NT>
__device__ __forceinline__ void cta_sum(double (&v)[K], double (*sm)[K])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; k++) {
        double a = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        v[k] = a;
    }
    __syncthreads();  // earlier readers of sm are done
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; k++) sm[w][k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; k++) {
        double s = 0;
#pragma unroll
        for (int i = 0; i < NT / 32; i++) s += sm[i][k];
        v[k] = s;
    }
}

template <typename R>
__device__ __forceinline__ void sp_norm_dot(const Spinor<R> &a, const Spinor<R> &b, R &re, R &im)
{  // += conj(a) b
#pragma unroll
    for (int sp = 0; sp < 4; sp++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            cpx<R> z = cmulc(a.v[sp][c], b.v[sp][c]);
            re += z.re;
            im += z.im;
        }
}

template <typename R>
__device__ __forceinline__ R sp_norm2(const Spinor<R> &a)
{
    R s = 0;
#pragma unroll
    for (int sp = 0; sp < 4; sp++)
#pragma unroll
        for (int c = 0; c < 3; c++) s += a.v[sp][c].re * a.v[sp][c].re + a.v[sp][c].im * a.v[sp][c].im;
    return s;
}

// Per-site pieces of the block operator, kept out of line so that every phase of the kernel
// reuses one register allocation (the fully unrolled stencil is large).

// odd site s:  out(s) = A_oo^-1 ( y(s) + coef * H_intra in (s) )    (y may be null, coef 0 skips the hop)
template <class P, int BL>
__device__ __noinline__ void site_odd(const GeomDev &g, long s, const typename P::SElem *in,
                                      const typename P::SElem *y, typename P::R coef,
                                      const typename P::UElem *__restrict__ U,
                                      const typename P::CElem *__restrict__ Ainv, typename P::SElem *out)
{
    using R = typename P::R;
    Spinor<R> acc;
    zero(acc);
    if (coef != R(0)) {
        Site<BL> st;
        decode_site<BL>(s, g, st);
        hop_sum<P, BL, 1, false>(g, st, s, in, U, acc);
        scale(acc, coef);
    }
    if (y) {
        Spinor<R> q;
        P::load_spinor_rw(y, g.V, s, q);
        axpy(acc, R(1), q);
    }
    clover_apply<P>(Ainv, g.V, s, R(0), acc);
    P::store_spinor(out, g.V, s, acc);
}

template <typename R> struct Dot3 {
    R a, b, c;
};

// even site s:  out(s) = D(x)(s) + coef * H_intra tmp (s), D = A(m) (diag) or 1, and the partial
// inner products of the phase: mode 1 -> conj(w) out; mode 2 -> conj(out) x and |out|^2.
template <class P, int BL>
__device__ __noinline__ Dot3<typename P::R> site_even(const GeomDev &g, long s, const typename P::SElem *tmp,
                                                      const typename P::SElem *x, typename P::R coef, bool diag,
                                                      typename P::R mass4, const typename P::UElem *__restrict__ U,
                                                      const typename P::CElem *__restrict__ Cl,
                                                      const typename P::SElem *w, int mode, typename P::SElem *out)
{
    using R = typename P::R;
    Spinor<R> acc, q;
    zero(acc);
    Site<BL> st;
    decode_site<BL>(s, g, st);
    hop_sum<P, BL, 1, false>(g, st, s, tmp, U, acc);
    scale(acc, coef);
    P::load_spinor_rw(x, g.V, s, q);
    Dot3<R> d{R(0), R(0), R(0)};
    if (diag) {
        Spinor<R> dq = q;
        clover_apply<P>(Cl, g.V, s, mass4, dq);
        axpy(acc, R(1), dq);
    } else {
        axpy(acc, R(1), q);
    }
    P::store_spinor(out, g.V, s, acc);
    if (mode == 1) {
        P::load_spinor_rw(w, g.V, s, q);
        sp_norm_dot(q, acc, d.a, d.b);
    } else if (mode == 2) {
        sp_norm_dot(acc, q, d.a, d.b);
        d.c = sp_norm2(acc);
    }
    return d;
}

template <class P, int BL, int NT>
// 32-bit arithmetic: at most 128 registers (170 for 128 threads) -- two 256-thread CTAs or one
// 512-thread CTA per SM -- so the register allocation keeps the occupancy of the out-of-line site
// functions
__global__ void __launch_bounds__(NT, sizeof(typename P::R) == 4 ? (NT >= 512 ? 1 : NT >= 256 ? 2 : NT >= 128 ? 3 : 1) : 1)
    k_block_plain(GeomDev g, PlainArgs<P> a)
{
    using R = typename P::R;
    using E = typename P::SElem;
    constexpr int VBH = BlockShape<BL>::VBH;
    constexpr int NP = P::NCHUNK, CW = P::CW;
    __shared__ double sm[NT / 32][3];
    // right-hand side fastest: the CTAs of one block run together and share its links in L2
    const int rhs = blockIdx.x;
    const int blk = a.blk0 + blockIdx.y;
    const long ro = (long)rhs * a.rstride;
    const int slot = rhs / a.rpm;
    const R mass4 = a.mass4[slot];
    const typename P::CElem *Ainv = a.Ainv[slot];
    const long e0 = (long)blk * VBH, o0 = g.vh + (long)blk * VBH;
    const long V = g.V;
    const E *b = a.b + ro;
    E *x = a.x + ro, *r = a.r + ro, *rh = a.rh + ro, *p = a.p + ro, *v = a.v + ro, *t = a.t + ro, *tmp = a.tmp + ro;

    // ||b||^2 over the block; tmp_o = A_oo^-1 b_o
    R bbl = 0;
    for (int h = threadIdx.x; h < VBH; h += NT)
        for (int k = 0; k < NP; k++) {
            cpx<R> c[CW], d[CW];
            P::ld_chunk(b, V, e0 + h, k, c);
            P::ld_chunk(b, V, o0 + h, k, d);
#pragma unroll
            for (int q = 0; q < CW; q++)
                bbl += c[q].re * c[q].re + c[q].im * c[q].im + d[q].re * d[q].re + d[q].im * d[q].im;
        }
    for (int h = threadIdx.x; h < VBH; h += NT) site_odd<P, BL>(g, o0 + h, nullptr, b, R(0), a.U, Ainv, tmp);
    double red[3] = {(double)bbl, 0, 0};
    cta_sum<3, NT>(red, sm);
    const double bb = red[0];
    // r = b_e + 1/2 H_eo tmp_o ; rh = p = r ; x_e = 0
    for (int h = threadIdx.x; h < VBH; h += NT)
        site_even<P, BL>(g, e0 + h, tmp, b, R(0.5), false, mass4, a.U, a.Cl, nullptr, 0, r);
    R rl = 0;
    for (int h = threadIdx.x; h < VBH; h += NT)
        for (int k = 0; k < NP; k++) {
            cpx<R> c[CW], z[CW];
            P::ld_chunk(r, V, e0 + h, k, c);
#pragma unroll
            for (int q = 0; q < CW; q++) {
                rl += c[q].re * c[q].re + c[q].im * c[q].im;
                z[q] = {R(0), R(0)};
            }
            P::st_chunk(rh, V, e0 + h, k, c);
            P::st_chunk(p, V, e0 + h, k, c);
            P::st_chunk(x, V, e0 + h, k, z);
        }
    red[0] = (double)rl;
    cta_sum<3, NT>(red, sm);
    double rr = red[0];
    double2 rho = make_double2(rr, 0.0);
    const double thresh = (a.tol2_dev ? *a.tol2_dev : a.tol2) * bb;
    int it = 0;
    bool ok = rr <= thresh;
    while (!ok && it < a.maxiter) {
        // v = S p  and  (rh, v)
        for (int h = threadIdx.x; h < VBH; h += NT) site_odd<P, BL>(g, o0 + h, p, nullptr, R(1), a.U, Ainv, tmp);
        __syncthreads();
        R are = 0, aim = 0;
        for (int h = threadIdx.x; h < VBH; h += NT) {
            Dot3<R> d = site_even<P, BL>(g, e0 + h, tmp, p, R(-0.25), true, mass4, a.U, a.Cl, rh, 1, v);
            are += d.a;
            aim += d.b;
        }
        red[0] = (double)are;
        red[1] = (double)aim;
        cta_sum<3, NT>(red, sm);
        double den = red[0] * red[0] + red[1] * red[1];
        if (den == 0.0 || !(den == den)) break;
        double2 alpha = make_double2((rho.x * red[0] + rho.y * red[1]) / den, (rho.y * red[0] - rho.x * red[1]) / den);
        const cpx<R> al = {R(alpha.x), R(alpha.y)};
        // s = r - alpha v (in r)
        for (int h = threadIdx.x; h < VBH; h += NT)
            for (int k = 0; k < NP; k++) {
                    cpx<R> c[CW], d[CW];
                P::ld_chunk(r, V, e0 + h, k, c);
                P::ld_chunk(v, V, e0 + h, k, d);
#pragma unroll
                for (int q = 0; q < CW; q++) c[q] = c[q] - cmul(al, d[q]);
                P::st_chunk(r, V, e0 + h, k, c);
            }
        __syncthreads();
        // t = S s  and  (t, s), (t, t)
        for (int h = threadIdx.x; h < VBH; h += NT) site_odd<P, BL>(g, o0 + h, r, nullptr, R(1), a.U, Ainv, tmp);
        __syncthreads();
        R tsr = 0, tsi = 0, tt = 0;
        for (int h = threadIdx.x; h < VBH; h += NT) {
            Dot3<R> d = site_even<P, BL>(g, e0 + h, tmp, r, R(-0.25), true, mass4, a.U, a.Cl, nullptr, 2, t);
            tsr += d.a;
            tsi += d.b;
            tt += d.c;
        }
        red[0] = (double)tsr;
        red[1] = (double)tsi;
        red[2] = (double)tt;
        cta_sum<3, NT>(red, sm);
        if (red[2] == 0.0 || !(red[2] == red[2])) break;
        double2 omega = make_double2(red[0] / red[2], red[1] / red[2]);
        const cpx<R> om = {R(omega.x), R(omega.y)};
        // x += alpha p + omega s ; r = s - omega t ; rho' = (rh, r) ; rr = (r, r)
        R hre = 0, him = 0, rrl = 0;
        for (int h = threadIdx.x; h < VBH; h += NT)
            for (int k = 0; k < NP; k++) {
                    cpx<R> xv[CW], pv[CW], sv[CW], tv[CW], hv[CW];
                P::ld_chunk(x, V, e0 + h, k, xv);
                P::ld_chunk(p, V, e0 + h, k, pv);
                P::ld_chunk(r, V, e0 + h, k, sv);
                P::ld_chunk(t, V, e0 + h, k, tv);
                P::ld_chunk(rh, V, e0 + h, k, hv);
#pragma unroll
                for (int q = 0; q < CW; q++) {
                    xv[q] = xv[q] + cmul(al, pv[q]) + cmul(om, sv[q]);
                    sv[q] = sv[q] - cmul(om, tv[q]);
                    cpx<R> z = cmulc(hv[q], sv[q]);
                    hre += z.re;
                    him += z.im;
                    rrl += sv[q].re * sv[q].re + sv[q].im * sv[q].im;
                }
                P::st_chunk(x, V, e0 + h, k, xv);
                P::st_chunk(r, V, e0 + h, k, sv);
            }
        red[0] = (double)hre;
        red[1] = (double)him;
        red[2] = (double)rrl;
        cta_sum<3, NT>(red, sm);
        it++;
        rr = red[2];
        if (!(rr == rr)) break;
        if (rr <= thresh) {
            ok = true;
            break;
        }
        double2 rn = make_double2(red[0], red[1]);
        double d1 = rho.x * rho.x + rho.y * rho.y, d2 = omega.x * omega.x + omega.y * omega.y;
        if (d1 == 0.0 || d2 == 0.0) break;
        double2 q1 = make_double2((rn.x * rho.x + rn.y * rho.y) / d1, (rn.y * rho.x - rn.x * rho.y) / d1);
        double2 q2 = make_double2((alpha.x * omega.x + alpha.y * omega.y) / d2, (alpha.y * omega.x - alpha.x * omega.y) / d2);
        const cpx<R> be = {R(q1.x * q2.x - q1.y * q2.y), R(q1.x * q2.y + q1.y * q2.x)};
        rho = rn;
        // p = r + beta (p - omega v)
        for (int h = threadIdx.x; h < VBH; h += NT)
            for (int k = 0; k < NP; k++) {
                    cpx<R> pv[CW], rv[CW], vv[CW];
                P::ld_chunk(p, V, e0 + h, k, pv);
                P::ld_chunk(r, V, e0 + h, k, rv);
                P::ld_chunk(v, V, e0 + h, k, vv);
#pragma unroll
                for (int q = 0; q < CW; q++) pv[q] = rv[q] + cmul(be, pv[q] - cmul(om, vv[q]));
                P::st_chunk(p, V, e0 + h, k, pv);
            }
        __syncthreads();
    }
    __syncthreads();
    // x_o = A_oo^-1 (b_o + 1/2 H_oe x_e)
    for (int h = threadIdx.x; h < VBH; h += NT) site_odd<P, BL>(g, o0 + h, x, b, R(0.5), a.U, Ainv, x);
    if (threadIdx.x == 0) {
        atomicMax(a.stat, it);
        if (!ok) atomicAdd(a.stat + 1, 1);
    }
}

template <int BL> void launch_plain(ddrw_ctx *ctx, const PlainArgs<PrecS> &a, int nrhs)
{
    constexpr int VBH = BlockShape<BL>::VBH, NT = VBH <= 32 ? 32 : VBH <= 128 ? 128 : VBH <= 648 ? 256 : 512;
    ++ctx->launches;
    k_block_plain<PrecS, BL, NT><<<dim3((unsigned)nrhs, (unsigned)ctx->nblk_c), NT, 0, ctx->stream>>>(geom_dev(ctx), a);
}

}  // namespace

ddrw_status block_plain32(ddrw_ctx *ctx, const BlkArgs<PrecS> &args, int nrhs)
{
    PlainArgs<PrecS> a;
    static_cast<BlkArgs<PrecS> &>(a) = args;
    const size_t f32 = sizeof(float4) * (size_t)a.rstride * nrhs;
    ddrw_status st;
    if ((st = workspace(ctx, "blk32_t", f32, (void **)&a.t))) return st;
    if ((st = workspace(ctx, "blk32_tmp", f32, (void **)&a.tmp))) return st;
    ProfScope ps(ctx, PROF_BLOCK32, 0.0);
    switch (ctx->l) {
    case 2: launch_plain<2>(ctx, a, nrhs); break;
    case 4: launch_plain<4>(ctx, a, nrhs); break;
    case 6: launch_plain<6>(ctx, a, nrhs); break;
    default: launch_plain<8>(ctx, a, nrhs); break;
    }
    return DDRW_OK;
}

}  // namespace ddrw
