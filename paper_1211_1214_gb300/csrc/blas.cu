// blas.cu -- vector kernels and reductions of the Krylov solvers (K7).
//
// A vector is a site range [off, off + n) of a field (all planes), for nrhs right-hand sides along
// gridDim.y.  Reductions: products are formed and summed over a storage chunk (at most a site) in the
// storage precision's arithmetic type; threads, warps, CTAs and the grid sum these in FP64 for FP64
// fields and in float pairs (RunSum, blas.cuh) for FP32 arithmetic, the last CTA of a right-hand side to
// finish (atomic ticket after a fence) in a fixed order, so the result does not depend on
// scheduling.  The solver scalars stay on the device; the last CTA
// also performs the scalar update of the Krylov recurrence.
#include <algorithm>

#include "blas.cuh"
#include "ctx.h"
#include "lowprec.cuh"

namespace ddrw {

// ----------------------------------------------------------------------------- element access

template <class P> struct VecArgs {
    long V, off, n, rs;  // plane stride, first site, sites, rhs stride (elements)
};

constexpr int NT = 256;

// body(j, k) for every site j of [0, n) and storage chunk k.  The units of work are (chunk, tile of NT
// sites), dealt to the CTAs of a right-hand side in turn: a short range (a 4096-site lattice in FP64 has
// 16 tiles of 12 chunks) still reaches all SMs, and a long one gives each thread several units, so that
// the reductions that follow run over few warps.
template <class P, class Body> __device__ __forceinline__ void for_chunks(long n, Body body)
{
    const int nt = (int)((n + NT - 1) / NT), nu = nt * P::NCHUNK;
    for (int u = blockIdx.x; u < nu; u += gridDim.x) {
        const int k = P::NCHUNK == 1 ? 0 : u / nt;
        const long j = (long)(u - k * nt) * NT + threadIdx.x;
        if (j < n) body(j, k);
    }
}

// ----------------------------------------------------------------------------- BiCGStab steps
// Scalars per right-hand side in KScal (blas.cuh).  r holds s = r - alpha v after the s-step.

template <class P>
__global__ void __launch_bounds__(NT) k_bicg_init(VecArgs<P> va, typename P::SElem *r, typename P::SElem *rh,
                                                  typename P::SElem *p, typename P::SElem *x, KScal *sc,
                                                  double *part, unsigned *ticket)
{
    using R = typename P::R;
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> acc;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], z[P::CW];
        SiteNorm<R> a;
        P::ld_chunk(r + rb, va.V, va.off + j, k, c);
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            a.add(q, c[q]);
            z[q] = {R(0), R(0)};
        }
        P::st_chunk(rh + rb, va.V, va.off + j, k, c);
        P::st_chunk(p + rb, va.V, va.off + j, k, c);
        P::st_chunk(x + rb, va.V, va.off + j, k, z);
        acc.add(a.total());
    });
    RunSum<R> sums[1] = {acc};
    double v[1];
    if (grid_sum_run<1, NT, R>(sums, v, part, ticket)) {
        KScal &s = sc[blockIdx.y];
        s.rho = make_double2(v[0], 0.0);
        s.rr = v[0];
        s.iters = 0;
        s.breakdown = 0;
        s.active = (v[0] > s.thresh) ? 1 : 0;
    }
}

template <class P>
__global__ void __launch_bounds__(NT) k_bicg_alpha(VecArgs<P> va, const typename P::SElem *rh,
                                                   const typename P::SElem *v, KScal *sc, double *part,
                                                   unsigned *ticket)
{
    using R = typename P::R;
    if (!sc[blockIdx.y].active) return;
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> are, aim;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], d[P::CW];
        SiteDot<R> a;
        P::ld_chunk(rh + rb, va.V, va.off + j, k, c);
        P::ld_chunk(v + rb, va.V, va.off + j, k, d);
#pragma unroll
        for (int q = 0; q < P::CW; q++) a.add(q, c[q], d[q]);
        are.add(a.total().re);
        aim.add(a.total().im);
    });
    RunSum<R> sums[2] = {are, aim};
    double val[2];
    if (grid_sum_run<2, NT, R>(sums, val, part, ticket)) {
        KScal &s = sc[blockIdx.y];
        double den = val[0] * val[0] + val[1] * val[1];
        if (den == 0.0 || !(den == den)) {
            s.breakdown = 1;
            s.active = 0;
            s.alpha = make_double2(0.0, 0.0);
            return;
        }
        // alpha = rho / (rh, v)
        s.alpha = make_double2((s.rho.x * val[0] + s.rho.y * val[1]) / den, (s.rho.y * val[0] - s.rho.x * val[1]) / den);
    }
}

template <class P>
__global__ void __launch_bounds__(NT) k_bicg_s(VecArgs<P> va, typename P::SElem *r, const typename P::SElem *v,
                                               const KScal *sc)
{
    using R = typename P::R;
    const KScal &s = sc[blockIdx.y];
    if (!s.active) return;
    const cpx<R> al = {R(s.alpha.x), R(s.alpha.y)};
    const long rb = (long)blockIdx.y * va.rs;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], d[P::CW];
        P::ld_chunk(r + rb, va.V, va.off + j, k, c);
        P::ld_chunk(v + rb, va.V, va.off + j, k, d);
#pragma unroll
        for (int q = 0; q < P::CW; q++) cmsub(c[q], al, d[q]);
        P::st_chunk(r + rb, va.V, va.off + j, k, c);
    });
}

// omega = (t, s) / (t, t) and, from the same pass over t, s and rh, the next direction's beta = (rho' alpha) /
// (rho omega) with rho' = (rh, s - omega t) = (rh, s) - omega (rh, t).  With beta known here, the updates of
// x, r and p need one kernel (k_bicg_xrp) instead of two that read and write r twice: 17 passes over a
// vector and 4 vector kernels per iteration, not 18 and 5.  The difference is rounded relative to |s|, which
// exceeds |r| where BiCGStab stagnates, so the rho that the next alpha divides by is the
// product (rh, r) itself, from the kernel that forms r (one pass, 0.4 to 1.4 % of the cases).  With the difference as rho
// too, FP64 solves of thousands of steps took 1.6 times as many (8^4, m = -0.11, eight fields, geometric
// mean: (rh, r) in both 4813, in rho 4716, in neither 9540); below 700 steps there is nothing to see.
// val: (t, s) re, im, (t, t), (rh, s) re, im, (rh, t) re, im
__device__ __forceinline__ void omega_beta(KScal &s, const double *val)
{
    if (val[2] == 0.0 || !(val[2] == val[2])) {
        s.breakdown = 2;
        s.active = 0;
        s.omega = make_double2(0.0, 0.0);
        return;
    }
    const double it = 1.0 / val[2];
    const double2 om = make_double2(val[0] * it, val[1] * it);
    const double2 rn = make_double2(val[3] - (om.x * val[5] - om.y * val[6]), val[4] - (om.x * val[6] + om.y * val[5]));
    const double2 num = make_double2(rn.x * s.alpha.x - rn.y * s.alpha.y, rn.x * s.alpha.y + rn.y * s.alpha.x);
    const double2 den = make_double2(s.rho.x * om.x - s.rho.y * om.y, s.rho.x * om.y + s.rho.y * om.x);
    const double d2 = den.x * den.x + den.y * den.y;
    s.omega = om;
    s.beta = d2 > 0.0 ? make_double2((num.x * den.x + num.y * den.y) / d2, (num.y * den.x - num.x * den.y) / d2)
                      : make_double2(0.0, 0.0);
    // a zero denominator ends the recurrence after this iteration's x and r (k_bicg_xrp)
    if (!(d2 > 0.0)) s.rho = make_double2(0.0, 0.0);
}

template <class P>
__global__ void __launch_bounds__(NT) k_bicg_omega(VecArgs<P> va, const typename P::SElem *t,
                                                   const typename P::SElem *r, const typename P::SElem *rh, KScal *sc,
                                                   double *part, unsigned *ticket)
{
    using R = typename P::R;
    if (!sc[blockIdx.y].active) return;
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> sums[7];
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], d[P::CW], h[P::CW];
        SiteDot<R> ts, hs, ht;
        SiteNorm<R> b;
        P::ld_chunk(t + rb, va.V, va.off + j, k, c);
        P::ld_chunk(r + rb, va.V, va.off + j, k, d);
        P::ld_chunk(rh + rb, va.V, va.off + j, k, h);
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            ts.add(q, c[q], d[q]);
            b.add(q, c[q]);
            hs.add(q, h[q], d[q]);
            ht.add(q, h[q], c[q]);
        }
        sums[0].add(ts.total().re);
        sums[1].add(ts.total().im);
        sums[2].add(b.total());
        sums[3].add(hs.total().re);
        sums[4].add(hs.total().im);
        sums[5].add(ht.total().re);
        sums[6].add(ht.total().im);
    });
    double val[7];
    if (grid_sum_run<7, NT, R>(sums, val, part, ticket)) omega_beta(sc[blockIdx.y], val);
}

// x += alpha p + omega s;  r = s - omega t;  p = r + beta (p - omega v);  rr = (r, r), rho = (rh, r)
template <class P>
__global__ void __launch_bounds__(NT, 2) k_bicg_xrp(VecArgs<P> va, typename P::SElem *x, typename P::SElem *p,
                                                    typename P::SElem *r, const typename P::SElem *t,
                                                    const typename P::SElem *v, const typename P::SElem *rh, KScal *sc,
                                                    double *part, unsigned *ticket)
{
    using R = typename P::R;
    const KScal &s0 = sc[blockIdx.y];
    if (!s0.active) return;
    const cpx<R> al = {R(s0.alpha.x), R(s0.alpha.y)}, om = {R(s0.omega.x), R(s0.omega.y)};
    const cpx<R> be = {R(s0.beta.x), R(s0.beta.y)};
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> rr[3];
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> xv[P::CW], pv[P::CW], sv[P::CW], tv[P::CW], vv[P::CW], hv[P::CW];
        SiteNorm<R> b;
        SiteDot<R> z;
        P::ld_chunk(x + rb, va.V, va.off + j, k, xv);
        P::ld_chunk(p + rb, va.V, va.off + j, k, pv);
        P::ld_chunk(r + rb, va.V, va.off + j, k, sv);
        P::ld_chunk(t + rb, va.V, va.off + j, k, tv);
        P::ld_chunk(v + rb, va.V, va.off + j, k, vv);
        P::ld_chunk(rh + rb, va.V, va.off + j, k, hv);
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            cmac(xv[q], al, pv[q]);
            cmac(xv[q], om, sv[q]);
            cmsub(sv[q], om, tv[q]);
            b.add(q, sv[q]);
            z.add(q, hv[q], sv[q]);
            cmsub(pv[q], om, vv[q]);
            tv[q] = sv[q];
            cmac(tv[q], be, pv[q]);
        }
        P::st_chunk(x + rb, va.V, va.off + j, k, xv);
        P::st_chunk(r + rb, va.V, va.off + j, k, sv);
        P::st_chunk(p + rb, va.V, va.off + j, k, tv);
        rr[0].add(b.total());
        rr[1].add(z.total().re);
        rr[2].add(z.total().im);
    });
    double val[3];
    if (grid_sum_run<3, NT, R>(rr, val, part, ticket)) {
        KScal &s = sc[blockIdx.y];
        s.rr = val[0];
        s.iters += 1;
        if (s.rho.x * s.rho.x + s.rho.y * s.rho.y != 0.0) s.rho = make_double2(val[1], val[2]);
        if (!(val[0] == val[0])) {
            s.breakdown = 3;
            s.active = 0;
        } else if (val[0] <= s.thresh || s.iters >= s.maxiter) {
            s.active = 0;
        } else if (s.rho.x * s.rho.x + s.rho.y * s.rho.y == 0.0) {
            s.breakdown = 4;
            s.active = 0;
        }
    }
}

// alpha (MODE 1) or omega and beta (MODE 2) from the per-warp partial sums (float pairs) a fused stencil
// epilogue wrote: part[(r * nwt + j) * RED_PARTS + k], in a fixed order (one CTA per right-hand side)
template <int MODE>
__global__ void __launch_bounds__(NT) k_bicg_fin(const float2 *part, long nwt, KScal *sc)
{
    constexpr int K = MODE == 1 ? 2 : RED_PARTS;
    __shared__ float2 sm[NT / 32][K], tot[K];
    const int r = blockIdx.x;
    if (!sc[r].active) return;
    RunSum<float> v[K];
#pragma unroll 2
    for (long j = threadIdx.x; j < nwt; j += NT) {
        const float2 *pp = part + ((long)r * nwt + j) * RED_PARTS;
#pragma unroll
        for (int k = 0; k < K; k++) v[k].join(pp[k]);
    }
    cta_sum_run<K, NT, float>(v, sm, tot);
    if (threadIdx.x >= 32) return;
    __syncwarp();
    if (threadIdx.x != 0) return;
    double val[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
        RunSum<float> q;
        q.join(tot[k]);
        val[k] = q.value();
    }
    KScal &s = sc[r];
    if constexpr (MODE == 1) {  // alpha = rho / (rh, v)
        const double den = val[0] * val[0] + val[1] * val[1];
        if (den == 0.0 || !(den == den)) {
            s.breakdown = 1;
            s.active = 0;
            s.alpha = make_double2(0.0, 0.0);
            return;
        }
        s.alpha = make_double2((s.rho.x * val[0] + s.rho.y * val[1]) / den, (s.rho.y * val[0] - s.rho.x * val[1]) / den);
    } else {
        omega_beta(s, val);
    }
}

void bicg_fin(ddrw_ctx *ctx, int mode, int nrhs, const double *part, long nwt, KScal *sc)
{
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    if (mode == 1) k_bicg_fin<1><<<nrhs, NT, 0, ctx->stream>>>((const float2 *)part, nwt, sc);
    else k_bicg_fin<2><<<nrhs, NT, 0, ctx->stream>>>((const float2 *)part, nwt, sc);
}

// ----------------------------------------------------------------------------- generic kernels

// out[r] = sum |f|^2 over the range (FP64 result per right-hand side)
template <class P>
__global__ void __launch_bounds__(NT) k_norm2(VecArgs<P> va, const typename P::SElem *f, double *out,
                                              double *part, unsigned *ticket)
{
    using R = typename P::R;
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> acc;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW];
        SiteNorm<R> a;
        P::ld_chunk(f + rb, va.V, va.off + j, k, c);
#pragma unroll
        for (int q = 0; q < P::CW; q++) a.add(q, c[q]);
        acc.add(a.total());
    });
    RunSum<R> sums[1] = {acc};
    double v[1];
    if (grid_sum_run<1, NT, R>(sums, v, part, ticket)) out[blockIdx.y] = v[0];
}

// out[3r .. 3r+2] = (sum |d|^2, Re sum conj(d) e, Im sum conj(d) e) -- the exponents
// ||delta||^2 + 2 Re <eta, delta> and <eta, delta>
template <class P>
__global__ void __launch_bounds__(NT) k_norm_dot(VecArgs<P> va, const typename P::SElem *d,
                                                 const typename P::SElem *e, double *out, double *part,
                                                 unsigned *ticket)
{
    using R = typename P::R;
    const long rb = (long)blockIdx.y * va.rs;
    RunSum<R> nn, dr, di;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], f[P::CW];
        SiteDot<R> a;
        SiteNorm<R> b;
        P::ld_chunk(d + rb, va.V, va.off + j, k, c);
        P::ld_chunk(e + rb, va.V, va.off + j, k, f);
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            b.add(q, c[q]);
            a.add(q, c[q], f[q]);
        }
        nn.add(b.total());
        dr.add(a.total().re);
        di.add(a.total().im);
    });
    RunSum<R> sums[3] = {nn, dr, di};
    double v[3];
    if (grid_sum_run<3, NT, R>(sums, v, part, ticket)) {
        out[3 * blockIdx.y] = v[0];
        out[3 * blockIdx.y + 1] = v[1];
        out[3 * blockIdx.y + 2] = v[2];
    }
}

// y = a x + b y with real per-launch scalars
template <class P>
__global__ void __launch_bounds__(NT) k_axpby(VecArgs<P> va, double a, const typename P::SElem *x, double b,
                                              typename P::SElem *y)
{
    using R = typename P::R;
    const long rb = (long)blockIdx.y * va.rs;
    for_chunks<P>(va.n, [&](long j, int k) {
        cpx<R> c[P::CW], d[P::CW];
        P::ld_chunk(x + rb, va.V, va.off + j, k, c);
        P::ld_chunk(y + rb, va.V, va.off + j, k, d);
#pragma unroll
        for (int q = 0; q < P::CW; q++) d[q] = R(a) * c[q] + R(b) * d[q];
        P::st_chunk(y + rb, va.V, va.off + j, k, d);
    });
}

// FP64 -> storage precision P with a per-right-hand-side scale: out = in * scale[r]
template <class P>
__global__ void __launch_bounds__(NT) k_to_low(long V, long off, long n, long rs64, long rsl, const double2 *in,
                                               typename P::SElem *out, const double *scale)
{
    using R = typename P::R;
    static_assert(sizeof(R) == 4, "");
    const double sc = scale ? scale[blockIdx.y] : 1.0;
    const double2 *ib = in + (long)blockIdx.y * rs64;
    typename P::SElem *ob = out + (long)blockIdx.y * rsl;
    for_chunks<P>(n, [&](long j, int k) {
        cpx<R> c[P::CW];
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            double2 a = ib[(long)(k * P::CW + q) * V + off + j];
            c[q] = {to_f32(a.x * sc), to_f32(a.y * sc)};
        }
        P::st_chunk(ob, V, off + j, k, c);
    });
}

// x64 += scale[r] * e (e in storage precision P), or x64 = scale[r] * e (FIRST); SPLIT: also the split copy of
// x64 that the double-single residual reads next, which saves its own pass
template <class P, bool FIRST, bool SPLIT>
__global__ void __launch_bounds__(NT) k_add_low(long V, long off, long n, long rs64, long rsl,
                                                const typename P::SElem *e, double2 *x, float4 *xs, const double *scale)
{
    using R = typename P::R;
    const double sc = scale ? scale[blockIdx.y] : 1.0;
    const typename P::SElem *eb = e + (long)blockIdx.y * rsl;
    double2 *xb = x + (long)blockIdx.y * rs64;
    float4 *sb = xs + (SPLIT ? (long)blockIdx.y * rs64 : 0);
    for_chunks<P>(n, [&](long j, int k) {
        cpx<R> c[P::CW];
        P::ld_chunk(eb, V, off + j, k, c);
#pragma unroll
        for (int q = 0; q < P::CW; q++) {
            const long i = (long)(k * P::CW + q) * V + off + j;
            double2 v = FIRST ? make_double2(0.0, 0.0) : xb[i];
            v = make_double2(fma(sc, to_f64(c[q].re), v.x), fma(sc, to_f64(c[q].im), v.y));
            xb[i] = v;
            if (SPLIT) {
                const float xh = to_f32(v.x), yh = to_f32(v.y);
                sb[i] = make_float4(xh, yh, to_f32(v.x - to_f64(xh)), to_f32(v.y - to_f64(yh)));
            }
        }
    });
}

// FP32 link / clover planes -> 16-bit planes of the same order
template <bool BF> __global__ void k_f32_to_low(long n, const float4 *__restrict__ in, uint2 *out)
{
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 v = in[i];
    out[i] = make_uint2(Pack16<BF>::pack(v.x, v.y), Pack16<BF>::pack(v.z, v.w));
}

// ----------------------------------------------------------------------------- host side

// CTAs per right-hand side for a range of n sites in nch chunks: one unit of for_chunks per CTA while
// nrhs of them fit the chip (152 SMs, 8 CTAs of 256 threads each), else the same
// number of units for each; at most 608, which the partial sums have room for
static unsigned grid_for(long n, int nch, int nrhs)
{
    const long units = std::max(1L, (n + NT - 1) / NT) * nch;
    const long most = std::min(608L, std::max(1L, (1216L + nrhs - 1) / nrhs));
    long per = (units + most - 1) / most;
    // FP64 fields (12 chunks): two units per CTA once every SM has work, the sums of a warp cost as much
    // FP64 time as a unit
    if (nch == 12) per = std::max(per, std::min(2L, units * nrhs / 152));
    return (unsigned)((units + per - 1) / per);
}

ddrw_status reduce_ws(ddrw_ctx *ctx, int nrhs, double **part, unsigned **ticket)
{
    void *p;
    ddrw_status st = workspace(ctx, "red_part", sizeof(double) * 8 * 608 * (size_t)nrhs, &p);
    if (st) return st;
    *part = (double *)p;
    DevBuf &t = ctx->ws["red_ticket"];
    if (t.bytes < sizeof(unsigned) * (size_t)nrhs) {
        clear_graphs(ctx);
        if (t.p) cudaFree(t.p);
        t.p = nullptr;
        t.bytes = 0;
        size_t bytes = sizeof(unsigned) * (size_t)(nrhs < 64 ? 64 : nrhs);
        if (cudaMalloc(&t.p, bytes) != cudaSuccess) return set_error(ctx, DDRW_ENOMEM, "ticket buffer");
        cudaMemsetAsync(t.p, 0, bytes, ctx->stream);
        t.bytes = bytes;
    }
    *ticket = (unsigned *)t.p;
    return DDRW_OK;
}

template <class P>
ddrw_status Blas<P>::bicg_init(ddrw_ctx *ctx, const VecRange &vr, E *r, E *rh, E *p, E *x, KScal *sc)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    dim3 g(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs);
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_bicg_init<P><<<g, NT, 0, ctx->stream>>>(va, r, rh, p, x, sc, part, tk);
    return DDRW_OK;
}

template <class P>
ddrw_status Blas<P>::bicg_alpha(ddrw_ctx *ctx, const VecRange &vr, const E *rh, const E *v, KScal *sc)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_bicg_alpha<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, rh, v, sc, part, tk);
    return DDRW_OK;
}

template <class P>
void Blas<P>::bicg_s(ddrw_ctx *ctx, const VecRange &vr, E *r, const E *v, const KScal *sc)
{
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_bicg_s<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, r, v, sc);
}

template <class P>
ddrw_status Blas<P>::bicg_omega(ddrw_ctx *ctx, const VecRange &vr, const E *t, const E *r, const E *rh, KScal *sc)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_bicg_omega<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, t, r, rh, sc, part, tk);
    return DDRW_OK;
}

template <class P>
ddrw_status Blas<P>::bicg_xrp(ddrw_ctx *ctx, const VecRange &vr, E *x, E *p, E *r, const E *t, const E *v, const E *rh,
                              KScal *sc)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_bicg_xrp<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, x, p, r, t, v, rh, sc, part,
                                                                                         tk);
    return DDRW_OK;
}

template <class P>
ddrw_status Blas<P>::norm2(ddrw_ctx *ctx, const VecRange &vr, const E *f, double *out)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_norm2<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, f, out, part, tk);
    return DDRW_OK;
}

template <class P>
ddrw_status Blas<P>::norm_dot(ddrw_ctx *ctx, const VecRange &vr, const E *d, const E *e, double *out)
{
    double *part;
    unsigned *tk;
    ddrw_status st = reduce_ws(ctx, vr.nrhs, &part, &tk);
    if (st) return st;
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_norm_dot<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, d, e, out, part, tk);
    return DDRW_OK;
}

template <class P>
void Blas<P>::axpby(ddrw_ctx *ctx, const VecRange &vr, double a, const E *x, double b, E *y)
{
    VecArgs<P> va{vr.V, vr.off, vr.n, vr.rs};
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_axpby<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(va, a, x, b, y);
}

template <class P>
void to_low(ddrw_ctx *ctx, const VecRange &vr, long rsl, const double2 *in, typename P::SElem *out,
            const double *scale)
{
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_to_low<P><<<dim3(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rsl, in, out, scale);
}

template <class P>
void add_low(ddrw_ctx *ctx, const VecRange &vr, long rsl, const typename P::SElem *e, double2 *x, const double *scale,
             bool first, float4 *xs)
{
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    const dim3 g(grid_for(vr.n, P::NCHUNK, vr.nrhs), vr.nrhs);
    if (first && xs) k_add_low<P, true, true><<<g, NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rsl, e, x, xs, scale);
    else if (first) k_add_low<P, true, false><<<g, NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rsl, e, x, xs, scale);
    else if (xs) k_add_low<P, false, true><<<g, NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rsl, e, x, xs, scale);
    else k_add_low<P, false, false><<<g, NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rsl, e, x, xs, scale);
}

void f32_to_low(ddrw_ctx *ctx, const float4 *in, uint2 *out, long n, bool bf)
{
    ++ctx->launches;
    unsigned g = (unsigned)((n + 255) / 256);
    if (bf) k_f32_to_low<true><<<g, 256, 0, ctx->stream>>>(n, in, out);
    else k_f32_to_low<false><<<g, 256, 0, ctx->stream>>>(n, in, out);
}

// FP32 field -> 16-bit field over a site range (the 16-bit spinor takes its per-site norm anew)
template <class P16>
__global__ void __launch_bounds__(NT) k_f32_to_16(long V, long off, long n, long rs32, long rs16, const float4 *in,
                                                  typename P16::SElem *out)
{
    const float4 *ib = in + (long)blockIdx.y * rs32;
    typename P16::SElem *ob = out + (long)blockIdx.y * rs16;
    for (long j = (long)blockIdx.x * NT + threadIdx.x; j < n; j += (long)gridDim.x * NT) {
        Spinor<float> p;
        PrecS::load_spinor_rw(ib, (int)V, (int)(off + j), p);
        P16::store_spinor(ob, (int)V, (int)(off + j), p);
    }
}

// x32 += x16 over a site range, then x16 = 0 (the reliable update of a 16-bit Krylov solve)
template <class P16>
__global__ void __launch_bounds__(NT) k_fold_16_into_32(long V, long off, long n, long rs16, long rs32,
                                                        typename P16::SElem *x16, float4 *x32)
{
    typename P16::SElem *hb = x16 + (long)blockIdx.y * rs16;
    float4 *fb = x32 + (long)blockIdx.y * rs32;
    Spinor<float> z;
    zero(z);
    for (long j = (long)blockIdx.x * NT + threadIdx.x; j < n; j += (long)gridDim.x * NT) {
        const int sj = (int)(off + j);
        Spinor<float> a, b;
        P16::load_spinor_rw(hb, (int)V, sj, a);
        PrecS::load_spinor_rw(fb, (int)V, sj, b);
#pragma unroll
        for (int sp = 0; sp < 4; sp++)
#pragma unroll
            for (int c = 0; c < 3; c++) b.v[sp][c] = b.v[sp][c] + a.v[sp][c];
        PrecS::store_spinor(fb, (int)V, sj, b);
        P16::store_spinor(hb, (int)V, sj, z);
    }
}

template <class P16>
void f32_to_16(ddrw_ctx *ctx, const VecRange &vr, long rs16, const float4 *in, typename P16::SElem *out)
{
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_f32_to_16<P16><<<dim3(grid_for(vr.n, 1, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, vr.rs, rs16, in, out);
}

template <class P16>
void fold_16_into_32(ddrw_ctx *ctx, const VecRange &vr, long rs16, typename P16::SElem *x16, float4 *x32)
{
    ProfScope ps(ctx, PROF_BLAS, 0.0);
    ++ctx->launches;
    k_fold_16_into_32<P16><<<dim3(grid_for(vr.n, 1, vr.nrhs), vr.nrhs), NT, 0, ctx->stream>>>(vr.V, vr.off, vr.n, rs16, vr.rs, x16,
                                                                                   x32);
}
template void f32_to_16<PrecH>(ddrw_ctx *, const VecRange &, long, const float4 *, PrecH::SElem *);
template void f32_to_16<PrecB>(ddrw_ctx *, const VecRange &, long, const float4 *, PrecB::SElem *);
template void fold_16_into_32<PrecH>(ddrw_ctx *, const VecRange &, long, PrecH::SElem *, float4 *);
template void fold_16_into_32<PrecB>(ddrw_ctx *, const VecRange &, long, PrecB::SElem *, float4 *);

#define DDRW_LOW_INST(P)                                                                                      \
    template void to_low<P>(ddrw_ctx *, const VecRange &, long, const double2 *, P::SElem *, const double *); \
    template void add_low<P>(ddrw_ctx *, const VecRange &, long, const P::SElem *, double2 *, const double *, bool, float4 *);
DDRW_LOW_INST(PrecS)
DDRW_LOW_INST(PrecH)
DDRW_LOW_INST(PrecB)

template struct Blas<PrecD>;
template struct Blas<PrecS>;
template struct Blas<PrecH>;
template struct Blas<PrecB>;

}  // namespace ddrw
