// FP64 instantiations of the stencil (see dslash.cuh), the split form for small lattices (split64.cuh), and
// D applied to fields in the boundary layout.
#include "dslash.cuh"
#include "split64.cuh"

namespace ddrw {

namespace {

// Output site updates (sites x right-hand sides) up to which a launch takes the split form.  One thread per
// site takes 40 us for its chain of FP64 instructions however small the launch, then 2.2 us per 1000 site
// updates; eight lanes per site take 8 us and 2.5 us per 1000.  Measured on D, us, one thread per site /
// split: 256 updates 43 / 9, 4096 42 / 19, 8192 43 / 31, 16384 46 / 50, 131072 286 / 330.
constexpr long SPLIT_MOST = 12000;

// the block lengths with launches that small: 8^4 blocks come in launches of at least 16384 updates (a colour and
// parity of the smallest lattice, 16^4), D on the whole lattice with 6^4 blocks in 20736 (12^4)
template <bool LEX> constexpr int split_longest() { return LEX ? 4 : 6; }

// ---- one thread per site, boundary layout (in / out: [rhs][lexicographic site][12] complex): FP64 issue
// bounds the stencil (0.92 of it), so the strided 16-byte accesses of 192-byte spinors cost nothing, and
// the two layout passes over the fields are gone.

// internal-order neighbour geometry with lexicographic spinor access
template <int BL, int MU, int DIR>
__device__ __forceinline__ void hop_lex(const GeomDev &g, const Site<BL> &st, const int (&x)[4], int s,
                                        const double2 *__restrict__ in, const double2 *__restrict__ U, Spinor<double> &acc)
{
    bool cross;
    int ph;
    const int sn = neighbour<BL>(st, MU, DIR, g, &cross, &ph);
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[MU] += DIR;
    if (y[MU] < 0) y[MU] += g.L[MU];
    if (y[MU] >= g.L[MU]) y[MU] -= g.L[MU];
    const long ln = (((long)y[0] * g.L[1] + y[1]) * g.L[2] + y[2]) * g.L[3] + y[3];
    Spinor<double> p;
    PrecD::load_spinor(in + 12 * ln, 1, 0, p);
    Half<double> h, w;
    project<MU, -DIR>(p, h);
    Link<double> L;
    PrecD::load_link(U, (int)g.V, MU, DIR > 0 ? s : sn, L);
    if (DIR > 0) link_mul(L, h, w);
    else link_dag_mul(L, h, w);
    if (ph < 0)
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int c = 0; c < 3; c++) w.v[a][c] = -w.v[a][c];
    reconstruct_add<MU, -DIR>(acc, w);
}

template <int BL>
__global__ void __launch_bounds__(64) k_apply_lex(GeomDev g, const double2 *__restrict__ in, double2 *out, double mass4,
                                                  const double2 *__restrict__ U, const double2 *__restrict__ Cl, int nrhs)
{
    // right-hand sides fastest: the CTAs of one tile run together and share its links in L2
    const int rhs = blockIdx.x % nrhs;
    const long i = (long)(blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
    if (i >= g.V) return;
    const int s = (int)i;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int *o = g.blk_org + st.blk * 4;
    const int x[4] = {o[0] + st.c[0], o[1] + st.c[1], o[2] + st.c[2], o[3] + st.c[3]};
    in += (long)rhs * 12 * g.V;
    out += (long)rhs * 12 * g.V;
    Spinor<double> acc;
    zero(acc);
    hop_lex<BL, 0, +1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 0, -1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 1, +1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 1, -1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 2, +1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 2, -1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 3, +1>(g, st, x, s, in, U, acc);
    hop_lex<BL, 3, -1>(g, st, x, s, in, U, acc);
    const long lx = (((long)x[0] * g.L[1] + x[1]) * g.L[2] + x[2]) * g.L[3] + x[3];
#pragma unroll
    for (int ch = 0; ch < 2; ch++) {
        double c[36];
        cpx<double> v6[6], o6[6];
        PrecD::load_clover(Cl, (int)g.V, s, ch, c);
        PrecD::load_chiral(in + 12 * lx, 1, 0, ch, v6);
        herm6_mul<double>(c, mass4, v6, o6);
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const cpx<double> a = acc.v[2 * ch + k / 3][k % 3];
            out[12 * lx + 6 * ch + k] = make_double2(fma(-0.5, a.re, o6[k].re), fma(-0.5, a.im, o6[k].im));
        }
    }
}

// ---- split form: four sites per warp, one warp per CTA.  LEX: fields in the boundary layout.
struct SplitArgs {
    const double2 *in, *x;
    double2 *out;
    long rstride;
    const double2 *U, *Cl;
    double alpha, beta;
    int diag, post, hopsel, par0, npar, blk0, nblk, nrhs, rpm;
    double mass4[MAXM];
    const double2 *Ainv[MAXM];
};

template <int BL, bool LEX>
__global__ void __launch_bounds__(32) k_dslash_split(GeomDev g, SplitArgs a)
{
    __shared__ double2 w[4][8][6];
    const int u = threadIdx.x & 7, al = u & 3, q = u >> 2, sub = threadIdx.x >> 3;
    const int rhs = blockIdx.x % a.nrhs;
    const long nper = (long)a.nblk * BlockShape<BL>::VBH, n = nper * a.npar;
    const long i0 = (long)(blockIdx.x / a.nrhs) * 4 + sub;
    const bool live = i0 < n;
    const long i = live ? i0 : n - 1;  // (a last part of a warp repeats a site and stores nothing)
    const int pp = (int)(i / nper);
    const long s = (long)(a.par0 + pp) * g.vh + (long)a.blk0 * BlockShape<BL>::VBH + (i - pp * nper);
    const long V = g.V;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int slot = rhs / a.rpm;
    const double2 *in = a.in + (long)rhs * a.rstride;
    long lx = 0;
    if (LEX) lx = lex_index<BL>(st, g);
    if (a.beta != 0.0) {
        const int mu = u >> 1;
        const bool fwd = (u & 1) == 0;
        bool cross;
        int ph;
        const int sn = neighbour<BL>(st, mu, fwd ? 1 : -1, g, &cross, &ph);
        Half<double> h;
        if (a.hopsel == 0 || (a.hopsel == 1) != cross) {
            const double2 *lnk = a.U + (long)mu * 9 * V + (fwd ? s : (long)sn);
            if (LEX) {
                Site<BL> sy;
                decode_site<BL>(sn, g, sy);
                split_hop(in + 12 * lex_index<BL>(sy, g), 1, lnk, V, mu, fwd, h);
            } else {
                split_hop(in + sn, V, lnk, V, mu, fwd, h);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 6; k++) h.v[k / 3][k % 3] = {0.0, 0.0};
        }
#pragma unroll
        for (int k = 0; k < 6; k++)
            w[sub][u][k] = make_double2(flip_sign(h.v[k / 3][k % 3].re, ph < 0), flip_sign(h.v[k / 3][k % 3].im, ph < 0));
    }
    __syncwarp();
    cpx<double> o[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
    if (a.beta != 0.0) {
        split_sum(&w[sub][0][0], al, q, o);
#pragma unroll
        for (int c = 0; c < 3; c++) o[c] = a.beta * o[c];
    }
    if (a.diag) {
        const double2 *x = a.x + (long)rhs * a.rstride;
        cpx<double> v[3], t[3];
        const int sp = a.diag == 1 ? (al & 2) + q : al;  // the half row's input spin, or the own spin
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 e = LEX ? x[12 * lx + 3 * sp + c] : x[(long)(3 * sp + c) * V + s];
            v[c] = {e.x, e.y};
        }
        if (a.diag == 1) split_herm(a.Cl + s, V, al, q, a.mass4[slot], v, t);
        if (a.diag == 1 || q == 0)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const cpx<double> z = a.diag == 1 ? t[c] : v[c];
                o[c] = {fma(a.alpha, z.re, o[c].re), fma(a.alpha, z.im, o[c].im)};
            }
    }
    split_join(o);
    if (a.post) {
        cpx<double> v[3];
        split_fetch(o, al, q, v);
        split_herm(a.Ainv[slot] + s, V, al, q, 0.0, v, o);
        split_join(o);
    }
    if (live) {
        double2 *out = a.out + (long)rhs * a.rstride;
#pragma unroll
        for (int c = 0; c < 3; c++)
            if ((c == 2) == (q == 1)) {  // colours 0, 1 by the first half's lane, 2 by the second's
                double2 *d = LEX ? out + 12 * lx + 3 * al + c : out + (long)(3 * al + c) * V + s;
                *d = make_double2(o[c].re, o[c].im);
            }
    }
}

template <bool LEX> void run_split(ddrw_ctx *ctx, const SplitArgs &a)
{
    const long vbh = (long)ctx->l * ctx->l * ctx->l * ctx->l / 2, n = (long)a.npar * a.nblk * vbh;
    const unsigned grid = (unsigned)((n + 3) / 4 * a.nrhs);
    const GeomDev g = geom_dev(ctx);
    ++ctx->launches;
    switch (ctx->l) {
    case 2: k_dslash_split<2, LEX><<<grid, 32, 0, ctx->stream>>>(g, a); break;
    case 4: k_dslash_split<4, LEX><<<grid, 32, 0, ctx->stream>>>(g, a); break;
    default:
        if constexpr (!LEX) k_dslash_split<6, LEX><<<grid, 32, 0, ctx->stream>>>(g, a);
    }
}

SplitArgs split_args(const ddrw_ctx *ctx, const DslashCall &c)
{
    SplitArgs a;
    a.in = (const double2 *)c.in;
    a.x = (const double2 *)c.x;
    a.out = (double2 *)c.out;
    a.rstride = c.rstride;
    a.U = ctx->U64;
    a.Cl = ctx->C64;
    a.alpha = c.alpha;
    a.beta = c.beta;
    a.diag = c.diag;
    a.post = c.post;
    a.hopsel = c.hopsel;
    a.par0 = c.par0;
    a.npar = c.npar;
    a.blk0 = c.blk0;
    a.nblk = c.nblk;
    a.nrhs = c.nrhs;
    const int nm = c.nmass < 1 ? 1 : c.nmass;
    a.rpm = (c.nrhs + nm - 1) / nm;
    for (int k = 0; k < MAXM; k++) {
        const int kk = k < nm ? k : nm - 1;
        a.mass4[k] = 4.0 + c.masses[kk];
        a.Ainv[k] = (const double2 *)c.Ainv[kk];
    }
    return a;
}

}  // namespace

void dslash64(ddrw_ctx *ctx, const DslashCall &c)
{
    const long n = (long)c.npar * c.nblk * ctx->l * ctx->l * ctx->l * ctx->l / 2;
    if (n == 0 || c.nrhs == 0) return;
    // (a pinned launch form, ddrw_stencil_config, selects among the forms of k_dslash)
    if (n * c.nrhs <= SPLIT_MOST && ctx->l <= split_longest<false>() && ctx->pinned_nr == 0) {
        ProfScope ps(ctx, PROF_DSLASH64 + (c.hopsel != 0 ? 2 : 0), compulsory_bytes<PrecD>(c, n), (double)n * c.nrhs);
        run_split<false>(ctx, split_args(ctx, c));
        return;
    }
    launch<PrecD>(ctx, c);
}

void apply_D_lex64(ddrw_ctx *ctx, double m, const double2 *in, double2 *out, int nrhs)
{
    DslashCall c;  // D on every site
    c.in = in;
    c.x = in;
    c.out = out;
    c.rstride = 12 * ctx->V;
    c.nrhs = nrhs;
    c.masses[0] = m;
    c.alpha = 1.0;
    c.beta = -0.5;
    c.diag = 1;
    c.par0 = 0;
    c.npar = 2;
    c.blk0 = 0;
    c.nblk = ctx->nblk;
    ProfScope ps(ctx, PROF_DSLASH64, compulsory_bytes<PrecD>(c, ctx->V), (double)ctx->V * nrhs);
    if (ctx->V * nrhs <= SPLIT_MOST && ctx->l <= split_longest<true>()) {
        run_split<true>(ctx, split_args(ctx, c));
        return;
    }
    const GeomDev g = geom_dev(ctx);
    const unsigned grid = (unsigned)((ctx->V + 63) / 64 * nrhs);
    ++ctx->launches;
    switch (ctx->l) {
    case 2: k_apply_lex<2><<<grid, 64, 0, ctx->stream>>>(g, in, out, 4.0 + m, ctx->U64, ctx->C64, nrhs); break;
    case 4: k_apply_lex<4><<<grid, 64, 0, ctx->stream>>>(g, in, out, 4.0 + m, ctx->U64, ctx->C64, nrhs); break;
    case 6: k_apply_lex<6><<<grid, 64, 0, ctx->stream>>>(g, in, out, 4.0 + m, ctx->U64, ctx->C64, nrhs); break;
    default: k_apply_lex<8><<<grid, 64, 0, ctx->stream>>>(g, in, out, 4.0 + m, ctx->U64, ctx->C64, nrhs); break;
    }
}

}  // namespace ddrw
