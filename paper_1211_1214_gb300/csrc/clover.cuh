// clover.cuh -- the O(a) improvement term C(x) = csw (i/4) sum sigma_{mu nu} Fhat_{mu nu}(x) from the
// plaquette leaves around each site (K2); instantiated per block length in clover_<l>.cu.
//
// Fhat_{mu nu} = (Q - Q^dag) / 8, Q the sum of the four counter-clockwise leaves at x.  A plaquette loop
// W_0 W_1 W_2 W_3 = U_mu(y) U_nu(y+mu) U_mu(y+nu)^dag U_nu(y)^dag gives one leaf to each of its corners, the loop
// begun there: with S_j = W_j W_{j+1} they are S_0 S_2, S_1 S_3, S_2 S_0, S_3 S_1.  So a plane takes 8 matrix
// products per site (one kernel for the leaves of every plaquette, kept as the 9 reals of their
// anti-Hermitian parts, one that sums the four at a site) instead of 12.  Bound by FP64 issue (GB300: 1/64 of
// the FP32 rate); 32x16^3: 1.32 ms for the six planes and the assembly, 3.01 ms when each site formed
// its own 24 leaves with unfused multiply-adds.
#pragma once

#include "ctx.h"

namespace ddrw {

// planes (mu, nu): 01 02 03 12 13 23
__host__ __device__ constexpr int plane_mu(int pl) { return pl < 3 ? 0 : pl < 5 ? 1 : 2; }
__host__ __device__ constexpr int plane_nu(int pl) { return pl < 3 ? pl + 1 : pl < 5 ? pl - 1 : 3; }

// internal index of x + da mu + db nu (da, db in -1 .. 1)
template <int BL>
__device__ __forceinline__ long site_near(const GeomDev &g, const int (&x)[4], int mu, int da, int nu, int db)
{
    int c[4];
#pragma unroll
    for (int d = 0; d < 4; d++) {
        const int v = x[d] + (d == mu ? da : 0) + (d == nu ? db : 0);
        c[d] = v < 0 ? v + g.L[d] : v >= g.L[d] ? v - g.L[d] : v;
    }
    return internal_index<BL>(g, c[0], c[1], c[2], c[3]);
}

// Thread row j of 32 sites: W_j, then S_j and the leaf S_j S_{j+2} of corner j; leaf[(j * 9 + k) V + x] the
// k-th real of leaf - leaf^dag: the imaginary parts of the diagonal (k = 0..2), then (re, im) of 01, 02, 12.
// The loop's lower left corner is x, V a multiple of 32.
template <int BL>
__global__ void __launch_bounds__(128) k_leaves(GeomDev g, const double2 *__restrict__ U64, int mu, int nu, double *leaf)
{
    __shared__ double2 sh[4][9][32];
    const int j = threadIdx.y, t = threadIdx.x;
    const long V = g.V, s = (long)blockIdx.x * 32 + t;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int *o = g.blk_org + st.blk * 4;
    const int x[4] = {o[0] + st.c[0], o[1] + st.c[1], o[2] + st.c[2], o[3] + st.c[3]};
    // the site that holds link j: corner j for j < 2, the next corner for the links run backwards
    const int k = j < 2 ? j : (j + 1) & 3;
    const long sl = site_near<BL>(g, x, mu, k == 1 || k == 2, nu, k >= 2);
    const double2 *b = U64 + (long)((j & 1) ? nu : mu) * 9 * V + sl;
    cpx<double> W[3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 v = __ldg(b + (long)(j < 2 ? 3 * a + c : 3 * c + a) * V);
            W[a][c] = {v.x, j < 2 ? v.y : -v.y};
        }
    auto share = [&](const cpx<double> (&m)[3][3]) {
#pragma unroll
        for (int e = 0; e < 9; e++) sh[j][e][t] = make_double2(m[e / 3][e % 3].re, m[e / 3][e % 3].im);
    };
    auto times = [&](const cpx<double> (&m)[3][3], int q, cpx<double> (&r)[3][3]) {  // r = m * (row q's matrix)
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int c = 0; c < 3; c++) r[a][c] = {0.0, 0.0};
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const double2 v = sh[q & 3][e][t];
#pragma unroll
            for (int a = 0; a < 3; a++) cmac(r[a][e % 3], m[a][e / 3], cpx<double>{v.x, v.y});
        }
    };
    cpx<double> S[3][3], Q[3][3];
    share(W);
    __syncthreads();
    times(W, j + 1, S);
    __syncthreads();
    share(S);
    __syncthreads();
    times(S, j + 2, Q);
    double *d = leaf + (long)j * 9 * V + s;
    d[0] = Q[0][0].im + Q[0][0].im;
    d[V] = Q[1][1].im + Q[1][1].im;
    d[2 * V] = Q[2][2].im + Q[2][2].im;
    d[3 * V] = Q[0][1].re - Q[1][0].re;
    d[4 * V] = Q[0][1].im + Q[1][0].im;
    d[5 * V] = Q[0][2].re - Q[2][0].re;
    d[6 * V] = Q[0][2].im + Q[2][0].im;
    d[7 * V] = Q[1][2].re - Q[2][1].re;
    d[8 * V] = Q[1][2].im + Q[2][1].im;
}

// F[k V + x] = the k-th real of Fhat_{mu nu}(x): corner 0 of the loop at x, 1 at x - mu, 2 at x - mu - nu, 3 at x - nu
template <int BL>
__global__ void __launch_bounds__(128) k_field_strength(GeomDev g, const double *__restrict__ leaf, int mu, int nu, double *F)
{
    const long V = g.V, s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int *o = g.blk_org + st.blk * 4;
    const int x[4] = {o[0] + st.c[0], o[1] + st.c[1], o[2] + st.c[2], o[3] + st.c[3]};
    const long s1 = site_near<BL>(g, x, mu, -1, nu, 0), s2 = site_near<BL>(g, x, mu, -1, nu, -1);
    const long s3 = site_near<BL>(g, x, mu, 0, nu, -1);
#pragma unroll
    for (int k = 0; k < 9; k++)
        F[k * V + s] = 0.125 * ((leaf[k * V + s] + leaf[(9 + k) * V + s1]) + (leaf[(18 + k) * V + s2] + leaf[(27 + k) * V + s3]));
}

// In the chiral basis sigma_{0k} = diag(s_k, -s_k) and sigma_{jk} = -eps_{jkl} diag(s_l, s_l), so
//   C_+ = csw (i/2) sum_l s_l (x) Y+_l,  Y+ = (F01 - F23, F02 + F13, F03 - F12)
//   C_- = csw (i/2) sum_l s_l (x) Y-_l,  Y- = (-F01 - F23, -F02 + F13, -F03 - F12)
// and with G_l = (i/2) csw Y_l (Hermitian):  C_ch = [[G3, G1 - i G2], [G1 + i G2, -G3]].
static __global__ void __launch_bounds__(128) k_clover_assemble(long V, const double *__restrict__ F, double csw,
                                                                double2 *C64, float4 *C32)
{
    const long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
#pragma unroll 1
    for (int ch = 0; ch < 2; ch++) {
        const double sg = ch == 0 ? 1.0 : -1.0, h = 0.5 * csw;
        // G_l from the reals y of Y_l: diagonal -h y, entries above it (i h)(re + i im) = (-h im, h re)
        double gd[3][3];
        cpx<double> go[3][3];  // [l][01, 02, 12]
#pragma unroll
        for (int l = 0; l < 3; l++) {
            const int pe = l, pm = l == 0 ? 5 : l == 1 ? 4 : 3;  // F_0l and F23, F13, F12
            const double m = l == 1 ? 1.0 : -1.0;
            double y[9];
#pragma unroll
            for (int k = 0; k < 9; k++) y[k] = sg * F[(long)(pe * 9 + k) * V + s] + m * F[(long)(pm * 9 + k) * V + s];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                gd[l][k] = -h * y[k];
                go[l][k] = {-h * y[4 + 2 * k], h * y[3 + 2 * k]};
            }
        }
        double r[36];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            r[k] = gd[2][k];
            r[3 + k] = -gd[2][k];
        }
        auto put = [&](int i, int j, cpx<double> z) {
            const int q = 6 + 2 * herm_off(i, j);
            r[q] = z.re;
            r[q + 1] = z.im;
        };
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const int a = k == 2 ? 1 : 0, b = k == 0 ? 1 : 2;
            put(a, b, go[2][k]);
            put(3 + a, 3 + b, -go[2][k]);
            const cpx<double> lo1 = {go[0][k].re, -go[0][k].im}, lo2 = {go[1][k].re, -go[1][k].im};  // below the diagonal
            put(a, 3 + b, go[0][k] - timesI(go[1][k]));
            put(b, 3 + a, lo1 - timesI(lo2));
            put(k, 3 + k, cpx<double>{gd[0][k], -gd[1][k]});
        }
#pragma unroll
        for (int k = 0; k < 18; k++) C64[((long)ch * 18 + k) * V + s] = make_double2(r[2 * k], r[2 * k + 1]);
#pragma unroll
        for (int k = 0; k < 9; k++)
            C32[((long)ch * 9 + k) * V + s] =
                make_float4(to_f32(r[4 * k]), to_f32(r[4 * k + 1]), to_f32(r[4 * k + 2]), to_f32(r[4 * k + 3]));
    }
}

// The scratch is the context's split copies of links and clover term, which the caller rebuilds afterwards:
// the leaves of one plane (288 bytes per site) in Cdd, the field strength (432) in Udd (576 each).
template <int BL>
void clover_launch(ddrw_ctx *ctx)
{
    const GeomDev g = geom_dev(ctx);
    double *leaf = reinterpret_cast<double *>(ctx->Cdd), *F = reinterpret_cast<double *>(ctx->Udd);
    const unsigned gl = (unsigned)(ctx->V / 32), gs = (unsigned)((ctx->V + 127) / 128);
    for (int pl = 0; pl < 6; pl++) {
        ctx->launches += 2;
        k_leaves<BL><<<gl, dim3(32, 4), 0, ctx->stream>>>(g, ctx->U64, plane_mu(pl), plane_nu(pl), leaf);
        k_field_strength<BL><<<gs, 128, 0, ctx->stream>>>(g, leaf, plane_mu(pl), plane_nu(pl), F + (long)pl * 9 * ctx->V);
    }
    ++ctx->launches;
    k_clover_assemble<<<gs, 128, 0, ctx->stream>>>(ctx->V, F, ctx->csw, ctx->C64, ctx->C32);
}

}  // namespace ddrw
