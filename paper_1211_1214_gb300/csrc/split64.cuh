// split64.cuh -- the FP64 stencil of one site by eight lanes, for lattices too small to fill the chip
// with one thread per site.
//
// GB300 issues one FP64 warp instruction per 20 clocks and SM, and a thread's chain of about 1200 of them
// takes 40 us however small the lattice is.  Here lane u of a site first does hop u (direction u / 2,
// forward for even u): projection and link multiply, about 84 FP64 instructions.  The half spinors meet
// in shared memory; then lane (spin al = u & 3, half q = u >> 2) sums four of the hops and half of the
// clover row of its spin, and the two halves of a spin join by a shuffle: about 160 FP64 instructions per
// lane in place of 1164 per thread, for 12 % more in total.  Spin factors of the chiral basis are +-1 and
// +-i, so they are exchanges of real and imaginary part and flips of the sign bit, no FP64 operations.
#pragma once

#include "ddrw_internal.cuh"

namespace ddrw {

__device__ __forceinline__ double flip_sign(double a, bool n)
{
    return __hiloint2double(__double2hiint(a) ^ (n ? (int)0x80000000 : 0), __double2loint(a));
}

// e_mu (see project): row sp has its entry in column sp ^ swaps(mu); entry -1, -i, or +1, +i if positive
struct SpinFactor {
    bool imag, neg;
};
__device__ __forceinline__ SpinFactor e_factor(int mu, int sp)
{
    return {(mu & 1) != 0, !(sp == 1 && mu >= 2)};
}
__device__ __forceinline__ int e_swap(int mu) { return mu == 1 || mu == 2; }

// f z for f = (neg ? -1 : 1) (imag ? i : 1)
__device__ __forceinline__ cpx<double> times_factor(cpx<double> z, bool imag, bool neg)
{
    return {flip_sign(imag ? z.im : z.re, neg != imag), flip_sign(imag ? z.re : z.im, neg)};
}

// the half spinor of hop (mu, fwd): w = V (psi_u + s e_mu psi_d)(y), V = U_mu(x) and s = -1 forward,
// U_mu(y)^dag and +1 backward; spinor component k of the source at src[k * sk], link component k at lnk[k * V]
__device__ __forceinline__ void split_hop(const double2 *src, long sk, const double2 *__restrict__ lnk, long V, int mu,
                                          bool fwd, Half<double> &w)
{
    Half<double> h;
    const int sw = e_swap(mu);
#pragma unroll
    for (int sp = 0; sp < 2; sp++) {
        const SpinFactor f = e_factor(mu, sp);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 u = src[(3 * sp + c) * sk], d = src[(6 + 3 * (sp ^ sw) + c) * sk];
            const cpx<double> e = times_factor({d.x, d.y}, f.imag, f.neg != fwd);
            h.v[sp][c] = {u.x + e.re, u.y + e.im};
        }
    }
    Link<double> L;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 v = __ldg(lnk + (fwd ? 3 * a + c : 3 * c + a) * V);
            L.m[a][c] = {v.x, flip_sign(v.y, !fwd)};
        }
    link_mul(L, h, w);
}

// sum of hops 4 q .. 4 q + 3 on output spin al (3 colours), from the half spinors of the site's hops
// (component k = 3 spin + colour of hop u at w[u * 6 + k])
__device__ __forceinline__ void split_sum(const double2 *w, int al, int q, cpx<double> (&o)[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) o[c] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int u = 4 * q + k, mu = u >> 1;
        const bool fwd = (u & 1) == 0;
        // upper spins take w, lower spin r takes s conj(e_mu(sp)) w_sp with sp = r ^ swap
        const int sp = al < 2 ? al : (al & 1) ^ e_swap(mu);
        const SpinFactor f = e_factor(mu, sp);
        const bool lower = al >= 2;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 v = w[u * 6 + 3 * sp + c];
            // conj(e) is -e for the imaginary factors
            const cpx<double> z = times_factor({v.x, v.y}, lower && f.imag, lower && ((f.neg != f.imag) != fwd));
            o[c].re += z.re;
            o[c].im += z.im;
        }
    }
}

// half of a row block of the packed Hermitian 6x6 matrices (both chiralities, planes V apart, site offset
// applied): o_a = sum_b H(3 (al & 1) + a, 3 q + b) v_b of chirality al >> 1, diag added on the diagonal
__device__ __forceinline__ void split_herm(const double2 *__restrict__ H, long V, int al, int q, double diag,
                                           const cpx<double> (&v)[3], cpx<double> (&o)[3])
{
    const double2 *b = H + (long)(al >> 1) * 18 * V;
    const int i0 = 3 * (al & 1), j0 = 3 * q;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        o[a] = {0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int i = i0 + a, j = j0 + c, lo = min(i, j), hi = max(i, j);
            if (i == j) {
                const double2 t = __ldg(b + (long)(i >> 1) * V);
                const double d = diag + ((i & 1) ? t.y : t.x);
                o[a] = {fma(d, v[c].re, o[a].re), fma(d, v[c].im, o[a].im)};
            } else {
                const double2 t = __ldg(b + (long)(3 + herm_off(lo, hi)) * V);
                cmac(o[a], cpx<double>{t.x, flip_sign(t.y, i > j)}, v[c]);
            }
        }
    }
}

// the other half's terms: lanes u and u ^ 4
__device__ __forceinline__ void split_join(cpx<double> (&o)[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        o[c].re += __shfl_xor_sync(0xffffffffu, o[c].re, 4);
        o[c].im += __shfl_xor_sync(0xffffffffu, o[c].im, 4);
    }
}

// the three components of spin 2 (al >> 1) + q of the same site, held (like all of its spin) by lanes of
// that spin: the input half of split_herm
__device__ __forceinline__ void split_fetch(const cpx<double> (&o)[3], int al, int q, cpx<double> (&v)[3])
{
    const int src = (threadIdx.x & 24) + (al & 2) + q;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        v[c].re = __shfl_sync(0xffffffffu, o[c].re, src);
        v[c].im = __shfl_sync(0xffffffffu, o[c].im, src);
    }
}

}  // namespace ddrw
