// force.cu -- the adjoint of the estimate (K11): derivatives of e = eta^dag (Mh^dag Mh - 1) eta
// (Eq. 3, Eq. 8 with N = 1) with respect to every link and to the target mass m2.
//
// Reverse mode, with y = Mh eta = eta + delta and Mh = A2^-1 A1 (A_k = A(m_k) = P Dhat(m_k) P):
//
//   de = 2 Re <y, d Mh eta> = 2 Re <z, dA1 eta - dA2 y>,   z = A2^-dag y,
//   z  = y - P g5 D_bw u'_w,   D(m2) u' = g5 y          (A^-1 = P(1 - Dcal_bw D_wb)P and D^dag = g5 D g5)
//
// and, for A = P(1 - B^-1 C W^-1 E)P with B = D_bb, C = D_bw, W = D_ww, E = D_wb at one mass,
//
//   <z, dA v> = <zt, dD rho> + <wt, dD sigma>,
//   a = W^-1 E v,  q = B^-1 C a,  zt = B^-dag z = g5 B^-1 g5 z,  wt = W^-dag C^dag zt = g5 W^-1 E g5 zt,
//   rho = q (black) - a (white),  sigma = a (white) - v (black).
//
// So de = 2 Re sum_k c_k <L_k, dD R_k> over four (L, R) pairs per noise vector (c = +w for the m1
// pair, -w for the m2 pair, w the caller's weight of that e_j).  Per link U_mu(x), with the
// direction dU = i T_a U (T_a = lambda_a / 2, left multiplication):
//
//   hopping:  de_a = Im tr(T_a (U Y - Z U^dag)),  Y = sum c [(1-g_mu) R(x+mu)] L(x)^dag,
//                                                  Z = sum c [(1+g_mu) R(x)] L(x+mu)^dag  (spin summed)
//   clover:   de = -(csw/8) sum_{x, mu<nu} Im tr(dQ_{mu nu}(x) Omega_{mu nu}(x)),
//             Omega = Lambda + Lambda^dag,  Lambda_{mu nu} = sum c sigma_{mu nu} R L^dag (spin summed);
//             for a link W_k = U of a plaquette loop W_0 W_1 W_2 W_3 with Omega_j at the corner
//             before W_j:  E_k = O_{k+1} W_{k+1} W_{k+2} W_{k+3} + W_{k+1} O_{k+2} W_{k+2} W_{k+3}
//                                + W_{k+1} W_{k+2} O_{k+3} W_{k+3} + W_{k+1} W_{k+2} W_{k+3} O_k,
//             K += -(csw/8) i U E_k  (and +(csw/8) i E_k U^dag where the loop holds U^dag),
//   and de_a = Im tr(T_a K) for the total K of the link.
//
//   mass:     de/dm2 = -2 Re [<zt_2, q_2> + <wt_2, a_2>]   (m1 fixed).
//
// Solutions are recomputed (forward chain, one adjoint full solve, eight block solves batched as
// two mass slots), not stored from the forward pass.  The force kernels run in FP64.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <vector>

#include "blas.cuh"
#include "ctx.h"
#include "stencil.cuh"

namespace ddrw {

ddrw_status estimate_fields_for_force(ddrw_ctx *ctx, int nhit, uint64_t seed, uint64_t hit0, const double *eta_user,
                                      double2 *eta, double2 *delta, double *exponents, SolveStats &stats);

namespace {

struct M3c {
    cpx<double> m[3][3];
};

__device__ __forceinline__ M3c m3_zero()
{
    M3c r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) r.m[i][j] = {0.0, 0.0};
    return r;
}
__device__ __forceinline__ M3c m3_mul(const M3c &a, const M3c &b)
{
    M3c c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cpx<double> t = cmul(a.m[i][0], b.m[0][j]);
            t = t + cmul(a.m[i][1], b.m[1][j]);
            t = t + cmul(a.m[i][2], b.m[2][j]);
            c.m[i][j] = t;
        }
    return c;
}
__device__ __forceinline__ M3c m3_dag(const M3c &a)
{
    M3c c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) c.m[i][j] = {a.m[j][i].re, -a.m[j][i].im};
    return c;
}
__device__ __forceinline__ void m3_acc(M3c &a, const M3c &b, double s)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) a.m[i][j] = a.m[i][j] + s * b.m[i][j];
}
__device__ __forceinline__ M3c load_link64(const double2 *U64, long V, int mu, long s)
{
    M3c r;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        double2 v = __ldg(U64 + ((long)mu * 9 + k) * V + s);
        r.m[k / 3][k % 3] = {v.x, v.y};
    }
    return r;
}

// K += a (x) b^dag for the colour vectors of one spin component
__device__ __forceinline__ void outer_mac(M3c &K, const cpx<double> *a, const cpx<double> *b)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) cmacc(K.m[i][j], b[j], a[i]);
}

struct ForceArgs {
    const double2 *L1, *R1, *L2, *R2;  // nrhs fields each
    const double *c;                   // per rhs coefficient
    int nrhs;
    long rs;
    const double2 *U64;
    double2 *omega;  // [6 planes][9][V]
    double *plaq[6]; // per plane [4 links of the loop][8][V]
    double csw;
    double *out;     // [V lexicographic][4][8]
};

// Omega_{mu nu}(x) = Lambda + Lambda^dag, Lambda = sum_rhs c sum_pairs sigma_{mu nu} R L^dag.  In the chiral
// basis sigma_{0l} = diag(s_l, -s_l) and sigma_{jk} = -eps_{jkl} diag(s_l, s_l), so the six planes are
// combinations of X_l = sum s_l R L^dag per chirality, l = 1..3: 36 colour outer products per pair of
// spinors instead of a dense spin product and 4 outer products for each plane.  Bound by FP64
// issue (about 5000 FP64 instructions per site at 8 right-hand sides).
__global__ void __launch_bounds__(64) k_omega(long V, ForceArgs a)
{
    const long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    M3c Lam[6];  // planes 01 02 03 12 13 23; the first chirality's X_l wait in the electric planes
#pragma unroll 1
    for (int ch = 0; ch < 2; ch++) {
        M3c D = m3_zero(), T01 = m3_zero(), T10 = m3_zero();  // T_ab = sum c R_a L_b^dag, D = T00 - T11
#pragma unroll 1
        for (int r = 0; r < 2 * a.nrhs; r++) {
            const int rr = r >> 1;
            const double2 *L = ((r & 1) ? a.L2 : a.L1) + rr * a.rs + (long)6 * ch * V + s;
            const double2 *R = ((r & 1) ? a.R2 : a.R1) + rr * a.rs + (long)6 * ch * V + s;
            const double c = a.c[rr];
            cpx<double> l[2][3], q[2][3];
#pragma unroll
            for (int k = 0; k < 6; k++) {
                const double2 u = L[(long)k * V], v = R[(long)k * V];
                l[k / 3][k % 3] = {u.x, u.y};
                q[k / 3][k % 3] = {c * v.x, c * v.y};
            }
            outer_mac(D, q[0], l[0]);
            outer_mac(T01, q[0], l[1]);
            outer_mac(T10, q[1], l[0]);
#pragma unroll
            for (int k = 0; k < 3; k++) q[1][k] = -q[1][k];
            outer_mac(D, q[1], l[1]);
        }
        // X_1 = T10 + T01, X_2 = -i T10 + i T01, X_3 = D
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const int i = k / 3, j = k % 3;
            const cpx<double> x1 = T10.m[i][j] + T01.m[i][j], x2 = timesI(T01.m[i][j] - T10.m[i][j]), x3 = D.m[i][j];
            if (ch == 0) {
                Lam[0].m[i][j] = x1;
                Lam[1].m[i][j] = x2;
                Lam[2].m[i][j] = x3;
            } else {
                Lam[5].m[i][j] = -(Lam[0].m[i][j] + x1);
                Lam[4].m[i][j] = Lam[1].m[i][j] + x2;
                Lam[3].m[i][j] = -(Lam[2].m[i][j] + x3);
                Lam[0].m[i][j] = Lam[0].m[i][j] - x1;
                Lam[1].m[i][j] = Lam[1].m[i][j] - x2;
                Lam[2].m[i][j] = Lam[2].m[i][j] - x3;
            }
        }
    }
#pragma unroll
    for (int pl = 0; pl < 6; pl++)
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const cpx<double> u = Lam[pl].m[k / 3][k % 3], v = Lam[pl].m[k % 3][k / 3];
            a.omega[((long)pl * 9 + k) * V + s] = make_double2(u.re + v.re, u.im - v.im);
        }
}

__device__ __forceinline__ M3c load_omega(const double2 *om, long V, int pl, long s)
{
    M3c r;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        double2 v = __ldg(om + ((long)pl * 9 + k) * V + s);
        r.m[k / 3][k % 3] = {v.x, v.y};
    }
    return r;
}

// Re tr(lambda_a M) (IM = false) or Im tr(lambda_a M), a = 1..8
template <bool IM> __device__ __forceinline__ void gell_mann_traces(const M3c &M, double *o)
{
    const double r3 = 0.57735026918962576;
    auto p = [](cpx<double> z) { return IM ? z.im : z.re; };
    auto pi = [](cpx<double> z) { return IM ? z.re : -z.im; };  // of i z
#pragma unroll
    for (int k = 0; k < 3; k++) {  // (i, j) = 01, 02, 12: lambda 1, 2; 4, 5; 6, 7
        const int i = k < 2 ? 0 : 1, j = k == 0 ? 1 : 2, n = k == 0 ? 0 : k == 1 ? 3 : 5;
        o[n] = p(M.m[i][j]) + p(M.m[j][i]);
        o[n + 1] = pi(M.m[i][j]) - pi(M.m[j][i]);
    }
    o[2] = p(M.m[0][0]) - p(M.m[1][1]);
    o[7] = r3 * (p(M.m[0][0]) + p(M.m[1][1]) - 2.0 * p(M.m[2][2]));
}

__device__ __forceinline__ long shifted(const int *x, const GeomDev &g, int mu, int dmu, int nu, int dnu, long (*index)(const GeomDev &, int, int, int, int))
{
    int c[4];
#pragma unroll
    for (int d = 0; d < 4; d++) {
        int v = x[d] + (d == mu ? dmu : 0) + (d == nu ? dnu : 0);
        c[d] = v < 0 ? v + g.L[d] : v >= g.L[d] ? v - g.L[d] : v;
    }
    return index(g, c[0], c[1], c[2], c[3]);
}

// The clover insertions of one plaquette loop W_0 W_1 W_2 W_3 = U_al(x) U_be(x+al) U_al(x+be)^dag U_be(x)^dag,
// Omega O_j at the corner before W_j, for its four links at once: with G_j = O_j W_j + W_j O_{j+1} and
// S_j = W_j W_{j+1},  E_k = G_{k+1} S_{k+2} + S_{k+1} G_{k+3}.  Thread row j forms G_j and S_j, shares
// them through shared memory, and then does E_j and the link's eight traces: 6 matrix products per link,
// against 10 when every link forms its six loops alone.  plaq[pl][j][a][x] = Im tr(lambda_a / 2 K).
template <int BL>
__global__ void __launch_bounds__(128) k_plaq(GeomDev g, ForceArgs a)
{
    __shared__ double2 sh[2][4][9][32];  // G, S
    const int j = threadIdx.y, t = threadIdx.x;
    const long s0 = (long)blockIdx.x * 32 + t;
    const long s = s0 < g.V ? s0 : g.V - 1;  // (V is a multiple of 16: a last half warp repeats a site)
    const int pl = blockIdx.y;
    const int al = pl < 3 ? 0 : pl < 5 ? 1 : 2, be = pl < 3 ? pl + 1 : pl < 5 ? pl - 1 : 3;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int *o = g.blk_org + st.blk * 4;
    const int x[4] = {o[0] + st.c[0], o[1] + st.c[1], o[2] + st.c[2], o[3] + st.c[3]};
    // corner j and the next one, the site and direction of link j
    const int j1 = (j + 1) & 3;
    const long cj = shifted(x, g, al, j == 1 || j == 2, be, j >= 2, internal_index<BL>);
    const long cn = shifted(x, g, al, j1 == 1 || j1 == 2, be, j1 >= 2, internal_index<BL>);
    const int dir = (j & 1) ? be : al;
    M3c W = load_link64(a.U64, g.V, dir, j < 2 ? cj : cn);
    if (j >= 2) W = m3_dag(W);
    {
        M3c G = m3_mul(load_omega(a.omega, g.V, pl, cj), W);
        m3_acc(G, m3_mul(W, load_omega(a.omega, g.V, pl, cn)), 1.0);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            sh[0][j][k][t] = make_double2(G.m[k / 3][k % 3].re, G.m[k / 3][k % 3].im);
            sh[1][j][k][t] = make_double2(W.m[k / 3][k % 3].re, W.m[k / 3][k % 3].im);
        }
    }
    auto get = [&](int f, int q) {
        M3c r;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const double2 v = sh[f][q & 3][k][t];
            r.m[k / 3][k % 3] = {v.x, v.y};
        }
        return r;
    };
    __syncthreads();
    const M3c S = m3_mul(W, get(1, j + 1));
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 9; k++) sh[1][j][k][t] = make_double2(S.m[k / 3][k % 3].re, S.m[k / 3][k % 3].im);
    __syncthreads();
    M3c E = m3_mul(get(0, j + 1), get(1, j + 2));
    m3_acc(E, m3_mul(get(1, j + 1), get(0, j + 3)), 1.0);
    // K = -f i U E (link held as U, j < 2) or +f i E U^dag (held as U^dag), f = csw / 8; Im tr(lambda/2 K)
    const M3c T = j < 2 ? m3_mul(W, E) : m3_mul(E, W);
    double tr[8];
    gell_mann_traces<false>(T, tr);
    const double f = 0.5 * a.csw / 8.0 * (j < 2 ? -1.0 : 1.0);
    if (s0 < g.V)
#pragma unroll
        for (int k = 0; k < 8; k++) a.plaq[pl][((long)j * 8 + k) * g.V + s] = f * tr[k];
}

// h = (1 + sg g_mu) psi restricted to its two independent spin components, psi_u + sg e_mu psi_d
__device__ __forceinline__ void load_projected(const double2 *f, long V, long s, int mu, double sg, cpx<double> (&h)[2][3])
{
    cpx<double> d[2][3];
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const double2 u = f[(long)k * V + s], v = f[(long)(6 + k) * V + s];
        h[k / 3][k % 3] = {u.x, u.y};
        d[k / 3][k % 3] = {v.x, v.y};
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cpx<double> e0, e1;  // e_mu psi_d
        switch (mu) {
        case 0: e0 = -d[0][c]; e1 = -d[1][c]; break;
        case 1: e0 = timesMinusI(d[1][c]); e1 = timesMinusI(d[0][c]); break;
        case 2: e0 = -d[1][c]; e1 = d[0][c]; break;
        default: e0 = timesMinusI(d[0][c]); e1 = timesI(d[1][c]); break;
        }
        h[0][c] = {fma(sg, e0.re, h[0][c].re), fma(sg, e0.im, h[0][c].im)};
        h[1][c] = {fma(sg, e1.re, h[1][c].re), fma(sg, e1.im, h[1][c].im)};
    }
}

// per link: K from the hopping bilinears, de_a = Im tr(T_a K), plus the traces of the six plaquettes that
// hold the link.  (1 -+ g_mu) = P^dag P with P psi the half spinor, so the spin sum of
// [(1 - g) R] L^dag has two outer products of half spinors.
template <int BL>
__global__ void __launch_bounds__(64) k_force(GeomDev g, ForceArgs a)
{
    const long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    const int mu = blockIdx.y;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    const int *o = g.blk_org + st.blk * 4;
    const int x[4] = {o[0] + st.c[0], o[1] + st.c[1], o[2] + st.c[2], o[3] + st.c[3]};
    bool cross;
    int ph;
    const long sf = neighbour<BL>(st, mu, +1, g, &cross, &ph);
    // Y = sum c [(1-g)R(x+mu)] L(x)^dag, Z = sum c [(1+g)R(x)] L(x+mu)^dag
    M3c Y = m3_zero(), Z = m3_zero();
#pragma unroll 1
    for (int r = 0; r < 2 * a.nrhs; r++) {
        const int rr = r >> 1;
        const double2 *L = ((r & 1) ? a.L2 : a.L1) + rr * a.rs, *R = ((r & 1) ? a.R2 : a.R1) + rr * a.rs;
        const double c = a.c[rr] * ph;
        cpx<double> l[2][3], q[2][3];
        load_projected(R, g.V, sf, mu, -1.0, q);
        load_projected(L, g.V, s, mu, -1.0, l);
#pragma unroll
        for (int sp = 0; sp < 2; sp++) {
#pragma unroll
            for (int k = 0; k < 3; k++) q[sp][k] = c * q[sp][k];
            outer_mac(Y, q[sp], l[sp]);
        }
        load_projected(R, g.V, s, mu, +1.0, q);
        load_projected(L, g.V, sf, mu, +1.0, l);
#pragma unroll
        for (int sp = 0; sp < 2; sp++) {
#pragma unroll
            for (int k = 0; k < 3; k++) q[sp][k] = c * q[sp][k];
            outer_mac(Z, q[sp], l[sp]);
        }
    }
    const M3c U = load_link64(a.U64, g.V, mu, s);
    M3c K = m3_mul(U, Y);
    m3_acc(K, m3_mul(Z, m3_dag(U)), -1.0);
    double de[8];
    gell_mann_traces<true>(K, de);
#pragma unroll
    for (int k = 0; k < 8; k++) de[k] *= 0.5;
    if (a.csw != 0.0)
        for (int nu = 0; nu < 4; nu++) {
            if (nu == mu) continue;
            const int al = mu < nu ? mu : nu, be = mu < nu ? nu : mu;
            const int pl = al == 0 ? be - 1 : al == 1 ? be + 1 : 5;
            // link 0 of the loop at x and 2 of the one at x - nu (mu = al), 3 at x and 1 at x - nu (mu = be)
            const long sn = shifted(x, g, nu, -1, mu, 0, internal_index<BL>);
            const double *p0 = a.plaq[pl] + (mu == al ? 0L : 3L) * 8 * g.V + s;
            const double *p1 = a.plaq[pl] + (mu == al ? 2L : 1L) * 8 * g.V + sn;
#pragma unroll
            for (int k = 0; k < 8; k++) de[k] += p0[(long)k * g.V] + p1[(long)k * g.V];
        }
    const long lx = (((long)x[0] * g.L[1] + x[1]) * g.L[2] + x[2]) * g.L[3] + x[3];
#pragma unroll
    for (int k = 0; k < 8; k++) a.out[(lx * 4 + mu) * 8 + k] = de[k];
}

// y = g5 x on every site (flip spins 2, 3)
__global__ void k_gamma5(long n12V, long V, int nrhs, long rs, const double2 *x, double2 *y)
{
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n12V * nrhs) return;
    long r = i / n12V, e = i - r * n12V;
    long k = e / V;
    double2 v = x[r * rs + e];
    y[r * rs + e] = k >= 6 ? make_double2(-v.x, -v.y) : v;
}

// z = P (y - g5 t) on supp P, zero elsewhere
template <int BL>
__global__ void k_zvec(GeomDev g, const double2 *y, const double2 *t, double2 *z, long rs)
{
    long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    Site<BL> st;
    decode_site<BL>(s, g, st);
    bool in = false;
    if (st.blk < g.nblk_c)
        for (int m = 0; m < 4; m++) in |= (st.c[m] == 0 || st.c[m] == BL - 1);
    long o = (long)blockIdx.y * rs + s;
    for (int k = 0; k < 12; k++) {
        double2 a = y[o + (long)k * g.V], b = t[o + (long)k * g.V];
        if (k >= 6) b = make_double2(-b.x, -b.y);
        z[o + (long)k * g.V] = in ? make_double2(a.x - b.x, a.y - b.y) : make_double2(0.0, 0.0);
    }
}

#define DISPATCH_BL(ctx, KERNEL, GRID, BLOCK, ...)                                                        \
    ++(ctx)->launches;                                                                                    \
    switch ((ctx)->l) {                                                                                   \
    case 2: KERNEL<2><<<GRID, BLOCK, 0, (ctx)->stream>>>(__VA_ARGS__); break;                             \
    case 4: KERNEL<4><<<GRID, BLOCK, 0, (ctx)->stream>>>(__VA_ARGS__); break;                             \
    case 6: KERNEL<6><<<GRID, BLOCK, 0, (ctx)->stream>>>(__VA_ARGS__); break;                             \
    default: KERNEL<8><<<GRID, BLOCK, 0, (ctx)->stream>>>(__VA_ARGS__); break;                            \
    }

void gamma5(ddrw_ctx *ctx, const double2 *x, double2 *y, int nrhs)
{
    long n = 12 * ctx->V;
    ++ctx->launches;
    k_gamma5<<<(unsigned)((n * nrhs + 255) / 256), 256, 0, ctx->stream>>>(n, ctx->V, nrhs, n, x, y);
}

}  // namespace

}  // namespace ddrw

using namespace ddrw;

extern "C" ddrw_status ddrw_force(ddrw_ctx *ctx, int nhit, uint64_t seed, uint64_t hit_offset, const double *eta_user,
                                  const double *weights, double *exponents, double *dU, double *dm2,
                                  ddrw_solve_info *info)
{
    if (!ctx || nhit <= 0) return set_error(ctx, DDRW_EINVAL, "bad argument");
    if (!ctx->have_gauge) return set_error(ctx, DDRW_ESTATE, "no gauge field loaded");
    cudaSetDevice(ctx->device);
    auto t0 = std::chrono::steady_clock::now();
    const long V = ctx->V, rs = 12 * V;
    const int R2 = 2 * nhit;
    const size_t f1 = sizeof(double2) * rs * nhit, f2 = sizeof(double2) * rs * R2;
    ddrw_status st;
    // fields: eta, delta (nhit) from the forward chain
    double2 *eta, *delta;
    if ((st = workspace(ctx, "frc_eta", f1, (void **)&eta))) return st;
    if ((st = workspace(ctx, "frc_delta", f1, (void **)&delta))) return st;
    std::vector<double> e(nhit);
    SolveStats stats;
    st = estimate_fields_for_force(ctx, nhit, seed, hit_offset, eta_user, eta, delta, e.data(), stats);
    ddrw_status conv = DDRW_OK;
    if (st == DDRW_ENOCONV) conv = st;
    else if (st) return st;
    if (exponents) std::copy(e.begin(), e.end(), exponents);

    double2 *F[8];
    const char *names[8] = {"frc_v2", "frc_a", "frc_q", "frc_zt", "frc_wt", "frc_t1", "frc_t2", "frc_z"};
    for (int k = 0; k < 8; k++)
        if ((st = workspace(ctx, names[k], f2, (void **)&F[k]))) return st;
    double2 *V2 = F[0], *A = F[1], *Q = F[2], *ZT = F[3], *WT = F[4], *T1 = F[5], *T2 = F[6], *Zf = F[7];
    // y = eta + delta into slot 1 of V2, eta into slot 0
    DDRW_CUDA_CHECK(cudaMemcpyAsync(V2, eta, f1, cudaMemcpyDeviceToDevice, ctx->stream));
    DDRW_CUDA_CHECK(cudaMemcpyAsync(V2 + rs * nhit, eta, f1, cudaMemcpyDeviceToDevice, ctx->stream));
    Blas<PrecD>::axpby(ctx, VecRange{V, 0, V, rs, nhit}, 1.0, delta, 1.0, V2 + rs * nhit);
    double2 *y = V2 + rs * nhit;

    MassSet m2s, m12;
    double mm[2] = {ctx->m1, ctx->m2};
    if ((st = make_massset(ctx, 1, &ctx->m2, &m2s))) return st;
    if ((st = make_massset(ctx, 2, mm, &m12))) return st;

    // z = y - P g5 D_bw u'_w, D(m2) u' = g5 y
    gamma5(ctx, y, T1, nhit);
    DDRW_CUDA_CHECK(cudaMemsetAsync(T2, 0, f1, ctx->stream));
    st = full_solve64(ctx, m2s, T1, T2, nhit, ctx->tol_outer, ctx->maxiter, ctx->prec, &stats);
    if (st == DDRW_ENOCONV) conv = st;
    else if (st) return st;
    DDRW_CUDA_CHECK(cudaMemsetAsync(T1, 0, f1, ctx->stream));
    hop_between64(ctx, DDRW_BLACK, T2, T1, nhit, -0.5);
    GeomDev g = geom_dev(ctx);
    {
        dim3 grid((unsigned)((V + 127) / 128), (unsigned)nhit);
        DISPATCH_BL(ctx, k_zvec, grid, 128, g, y, T1, Zf, rs);
    }
    // two mass slots (m1: v = eta, m2: v = y) of the four block solves
    auto bsolve = [&](int colour, const double2 *b, double2 *x) -> ddrw_status {
        DDRW_CUDA_CHECK(cudaMemsetAsync(x, 0, f2, ctx->stream));
        ddrw_status s2 = block_solve64(ctx, colour, m12, b, x, R2, ctx->tol_block, ctx->maxiter, ctx->prec, &stats,
                                       true);
        if (s2 == DDRW_ENOCONV) conv = s2;
        else if (s2) return s2;
        return DDRW_OK;
    };
    DDRW_CUDA_CHECK(cudaMemsetAsync(T1, 0, f2, ctx->stream));
    hop_between64(ctx, DDRW_WHITE, V2, T1, R2, -0.5);  // E v
    if ((st = bsolve(DDRW_WHITE, T1, A))) return st;  // a = W^-1 E v
    DDRW_CUDA_CHECK(cudaMemsetAsync(T1, 0, f2, ctx->stream));
    hop_between64(ctx, DDRW_BLACK, A, T1, R2, -0.5);  // C a
    if ((st = bsolve(DDRW_BLACK, T1, Q))) return st;  // q = B^-1 C a
    // g5 z in both slots
    gamma5(ctx, Zf, T1, nhit);
    DDRW_CUDA_CHECK(cudaMemcpyAsync(T1 + rs * nhit, T1, f1, cudaMemcpyDeviceToDevice, ctx->stream));
    if ((st = bsolve(DDRW_BLACK, T1, T2))) return st;  // B^-1 g5 z
    gamma5(ctx, T2, ZT, R2);                            // zt = g5 B^-1 g5 z
    DDRW_CUDA_CHECK(cudaMemsetAsync(T1, 0, f2, ctx->stream));
    hop_between64(ctx, DDRW_WHITE, T2, T1, R2, -0.5);  // E g5 zt
    if ((st = bsolve(DDRW_WHITE, T1, T2))) return st;
    gamma5(ctx, T2, WT, R2);  // wt = g5 W^-1 E g5 zt
    // rho = q - a (into Q), sigma = a - v (into A)
    Blas<PrecD>::axpby(ctx, VecRange{V, 0, V, rs, R2}, -1.0, A, 1.0, Q);
    Blas<PrecD>::axpby(ctx, VecRange{V, 0, V, rs, R2}, -1.0, V2, 1.0, A);

    // coefficients: +w (m1 slot), -w (m2 slot)
    std::vector<double> c(R2);
    for (int j = 0; j < nhit; j++) {
        double w = weights ? weights[j] : 1.0;
        c[j] = w;
        c[nhit + j] = -w;
    }
    double *cd, *red;
    if ((st = workspace(ctx, "frc_c", sizeof(double) * (R2 + 12 * R2), (void **)&cd))) return st;
    red = cd + R2;
    DDRW_CUDA_CHECK(cudaMemcpyAsync(cd, c.data(), sizeof(double) * R2, cudaMemcpyHostToDevice, ctx->stream));

    // de/dm2 = -2 Re[<zt_2, q_2> + <wt_2, a_2>] = -2 Re[<L1, rho> + <L2, sigma>] on the m2 slot
    if (dm2) {
        if ((st = Blas<PrecD>::norm_dot(ctx, VecRange{V, 0, V, rs, nhit}, ZT + rs * nhit, Q + rs * nhit, red))) return st;
        if ((st = Blas<PrecD>::norm_dot(ctx, VecRange{V, 0, V, rs, nhit}, WT + rs * nhit, A + rs * nhit, red + 3 * nhit)))
            return st;
        std::vector<double> h(6 * nhit);
        DDRW_CUDA_CHECK(cudaMemcpyAsync(h.data(), red, sizeof(double) * 6 * nhit, cudaMemcpyDeviceToHost, ctx->stream));
        DDRW_SYNC(ctx);
        for (int j = 0; j < nhit; j++) dm2[j] = -2.0 * (h[3 * j + 1] + h[3 * nhit + 3 * j + 1]);
    }
    if (dU) {
        double2 *omega;
        if ((st = workspace(ctx, "frc_omega", sizeof(double2) * 54 * V, (void **)&omega))) return st;
        // the plaquettes' traces, 256 bytes per site and plane, take the place of fields that are done with: four of
        // the chain's and two of the block solves', each at least 384 bytes per site
        double *plaq[6] = {(double *)V2, (double *)T1, (double *)T2, (double *)Zf};
        const size_t pb = sizeof(double) * 32 * V;
        if ((st = workspace(ctx, "blk_res64", pb, (void **)&plaq[4]))) return st;
        if ((st = workspace(ctx, ctx->prec == DDRW_FP64 ? "blk_e64" : "ds_split", pb, (void **)&plaq[5]))) return st;
        double *out;
        void *dout;
        bool host;
        size_t ob = sizeof(double) * 32 * V;
        if ((st = stage_out(ctx, dU, ob, "stage_force", &dout, &host))) return st;
        out = (double *)dout;
        ForceArgs fa{ZT, Q, WT, A, cd, R2, rs, ctx->U64, omega, {}, ctx->csw, out};
        std::copy(plaq, plaq + 6, fa.plaq);
        if (ctx->csw != 0.0) {
            ++ctx->launches;
            k_omega<<<(unsigned)((V + 63) / 64), 64, 0, ctx->stream>>>(V, fa);
            dim3 grid((unsigned)((V + 31) / 32), 6u);
            DISPATCH_BL(ctx, k_plaq, grid, dim3(32, 4), g, fa);
        }
        {
            dim3 grid((unsigned)((V + 63) / 64), 4u);
            DISPATCH_BL(ctx, k_force, grid, 64, g, fa);
        }
        if ((st = finish_out(ctx, dU, out, ob, host))) return st;
    }
    if ((st = sync(ctx))) return st;
    if (info) {
        info->iters_outer = stats.outer_iters;
        info->cycles = stats.outer_cycles;
        info->fp64_dslash_calls = stats.fp64_dslash_full;
        info->block_iters_max = stats.block_iters_max;
        info->iters_inner_total = (int)std::min<long>(stats.block_iters_total, 2147483647L);
        info->true_rel_residual = stats.outer_rel_residual;
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    return conv;
}
