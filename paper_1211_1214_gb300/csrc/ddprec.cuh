// ddprec.cuh -- double-single ("double-float") arithmetic for the defect-correction residuals of
// the mixed path.
//
// GB300 runs FP64 at 1/64 of its FP32 rate, so the FP64 stencil of the residual
// r = b - D x costs several FP32 stencils.  Here each real number is an unevaluated sum hi + lo of
// two FP32 numbers (|lo| <= ulp(hi)/2), about 44 significant bits, and the arithmetic uses the
// error-free transformations of Knuth's two-sum and the FMA-based two-product (Dekker's
// double-length arithmetic with a fused multiply-add).  Every operation is written with the
// round-to-nearest intrinsics, which the compiler never contracts or reassociates.
//
// Sums of products (link and clover multiplies) use accumulated pairs normalised once per result
// (dd2_acc below).
//
// Storage: a "split" field holds one complex number per 16-byte element (re.hi, im.hi, re.lo,
// im.lo: the register pairs of the packed arithmetic), the same bytes as an FP64 field; links (9 complex per
// direction) and the clover term (72 reals per site) are split once per configuration, the stencil input
// once per residual, and the result is written back as FP64 (hi + lo).
#pragma once

#include "ddrw_internal.cuh"

namespace ddrw {

struct dd {
    float hi, lo;
    __host__ __device__ dd() {}
    __host__ __device__ constexpr dd(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ dd(double x)
    {
        hi = (float)x;
        lo = (float)(x - (double)hi);
    }
    __host__ __device__ dd(int x) : dd((double)x) {}
};

// a + b with a two-sum of the leading parts (relative error ~2^-44 of |a| + |b|)
__device__ __forceinline__ dd operator+(dd a, dd b)
{
    float s = __fadd_rn(a.hi, b.hi);
    float v = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    float h = __fadd_rn(s, e);
    return dd(h, __fsub_rn(e, __fsub_rn(h, s)));
}
__device__ __forceinline__ dd operator-(dd a) { return dd(-a.hi, -a.lo); }
__device__ __forceinline__ dd operator-(dd a, dd b) { return a + (-b); }
// a * b with an FMA two-product of the leading parts
__device__ __forceinline__ dd operator*(dd a, dd b)
{
    float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    float h = __fadd_rn(p, e);
    return dd(h, __fsub_rn(e, __fsub_rn(h, p)));
}
__device__ __forceinline__ bool operator!=(dd a, dd b) { return a.hi != b.hi || a.lo != b.lo; }

// ---- complex numbers in packed form: the real and imaginary parts go through the same operations, so
// each step is one f32x2 instruction on (re, im).  The residual stencil is limited by instruction fetch and
// issue (about 8900 scalar FP32 instructions per site update, 28 % of the issue slots): the packed form
// has about half as many, in 168 registers (three CTAs of 128 threads per SM).  D on 16^4, 16 right-hand
// sides: 882 us scalar, 750 us packed with up to 255 registers, 648 us with 168 (682 with 128).
struct dd2 {
    f32x2 hi, lo;
};
__device__ __forceinline__ dd2 pack_dd(const cpx<dd> &z) { return {pack2(z.re.hi, z.im.hi), pack2(z.re.lo, z.im.lo)}; }
__device__ __forceinline__ dd2 pack_dd_swapped(const cpx<dd> &z) { return {pack2(z.im.hi, z.re.hi), pack2(z.im.lo, z.re.lo)}; }
__device__ __forceinline__ cpx<dd> unpack_dd(dd2 p)
{
    cpx<dd> z;
    unpack2(p.hi, z.re.hi, z.im.hi);
    unpack2(p.lo, z.re.lo, z.im.lo);
    return z;
}
// the operations of operator+(dd, dd) on both parts
__device__ __forceinline__ cpx<dd> operator+(cpx<dd> x, cpx<dd> y)
{
    const dd2 a = pack_dd(x), b = pack_dd(y);
    const f32x2 s = add2(a.hi, b.hi), v = sub2(s, a.hi);
    f32x2 e = add2(sub2(a.hi, sub2(s, v)), sub2(b.hi, v));
    e = add2(e, add2(a.lo, b.lo));
    const f32x2 h = add2(s, e);
    return unpack_dd({h, sub2(e, sub2(h, s))});
}

// A factor of an accumulated product: x and, for the error terms, -x (both parts may carry signs)
struct dd2_factor {
    f32x2 hi, nhi, nlo;
};
__device__ __forceinline__ dd2_factor both(dd x) { return {pack2(x.hi, x.hi), pack2(-x.hi, -x.hi), pack2(-x.lo, -x.lo)}; }
__device__ __forceinline__ dd2_factor minus_plus(dd x) { return {pack2(-x.hi, x.hi), pack2(x.hi, -x.hi), pack2(x.lo, -x.lo)}; }
__device__ __forceinline__ dd2_factor plus_minus(dd x) { return {pack2(x.hi, -x.hi), pack2(-x.hi, x.hi), pack2(-x.lo, x.lo)}; }

// ---- accumulated products.  A sum of products sum_k x_k y_k is kept as an unnormalised pair:
// each product's leading part enters the leading word through a two-sum, its rounding error and
// the two-sum's error collect in the trailing word, and the pair is normalised once at the end
// (12 FP32 operations per product instead of 18 for a normalised product plus a normalised sum).
struct dd2_acc {
    f32x2 hi = {0ull}, lo = {0ull};
    __device__ __forceinline__ void mac(dd2_factor x, dd2 y)  // += x y, part by part
    {
        const f32x2 p = mul2(x.hi, y.hi);
        f32x2 n = fma2(x.nhi, y.hi, p);  // minus the product's error
        n = fma2(x.nhi, y.lo, n);
        n = fma2(x.nlo, y.hi, n);
        const f32x2 s = add2(hi, p), v = sub2(s, hi);
        const f32x2 t = add2(sub2(hi, sub2(s, v)), sub2(p, v));
        hi = s;
        lo = add2(lo, sub2(t, n));
    }
    __device__ __forceinline__ cpx<dd> get() const
    {
        const f32x2 h = add2(hi, lo);
        return unpack_dd({h, sub2(lo, sub2(h, hi))});
    }
};

// w = U h (DAG: U^dag h) on the two spin components of a half spinor, in accumulated form:
// (re, im) += u.re (h.re, h.im) + (-u.im, u.im) (h.im, h.re)
template <bool DAG> __device__ __forceinline__ void link_mul_dd(const Link<dd> &U, const Half<dd> &h, Half<dd> &w)
{
    dd2 y[2][3], z[2][3];
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            y[s][b] = pack_dd(h.v[s][b]);
            z[s][b] = pack_dd_swapped(h.v[s][b]);
        }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        dd2_acc t[2];
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const cpx<dd> u = DAG ? U.m[b][a] : U.m[a][b];
            const dd2_factor fr = both(u.re), fi = DAG ? plus_minus(u.im) : minus_plus(u.im);
#pragma unroll
            for (int s = 0; s < 2; s++) {
                t[s].mac(fr, y[s][b]);
                t[s].mac(fi, z[s][b]);
            }
        }
#pragma unroll
        for (int s = 0; s < 2; s++) w.v[s][a] = t[s].get();
    }
}
template <> __device__ __forceinline__ void link_mul<dd>(const Link<dd> &U, const Half<dd> &h, Half<dd> &w)
{
    link_mul_dd<false>(U, h, w);
}
template <> __device__ __forceinline__ void link_dag_mul<dd>(const Link<dd> &U, const Half<dd> &h, Half<dd> &w)
{
    link_mul_dd<true>(U, h, w);
}

// out = (diag + H) v for a packed Hermitian 6x6 H (layout of herm6_mul), in accumulated form
template <> __device__ __forceinline__ void herm6_mul<dd>(const dd *c, dd diag, const cpx<dd> *v, cpx<dd> *out)
{
    dd2_acc t[6];
    dd2 y[6], z[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        y[i] = pack_dd(v[i]);
        z[i] = pack_dd_swapped(v[i]);
        t[i].mac(both(diag + c[i]), y[i]);
    }
#pragma unroll
    for (int i = 0; i < 6; i++)
#pragma unroll
        for (int j = i + 1; j < 6; j++) {
            const int o = 6 + 2 * herm_off(i, j);
            const dd2_factor hr = both(c[o]);
            // out_i += h_ij v_j ; out_j += conj(h_ij) v_i
            t[i].mac(hr, y[j]);
            t[i].mac(minus_plus(c[o + 1]), z[j]);
            t[j].mac(hr, y[i]);
            t[j].mac(plus_minus(c[o + 1]), z[i]);
        }
#pragma unroll
    for (int i = 0; i < 6; i++) out[i] = t[i].get();
}

// a power of two (alpha and beta of a double-single launch are): exact on both words
__device__ __forceinline__ cpx<dd> times_pow2(float a, cpx<dd> z)
{
    return {dd(a * z.re.hi, a * z.re.lo), dd(a * z.im.hi, a * z.im.lo)};
}

// Storage policy of the double-single stencil: split spinors, links and clover in, FP64 out.
struct PrecDD {
    using R = dd;
    using SElem = float4;  // one complex number (re.hi, im.hi, re.lo, im.lo)
    static constexpr int ID = 128;
    static constexpr double SBYTES = 192, UBYTES = 144, CBYTES = 576;
    static constexpr int SPLANES = 12;
    static constexpr int UPLANES = 9;
    static constexpr int CPLANES = 36;
    using UElem = float4;
    using CElem = float4;

    __device__ static __forceinline__ cpx<dd> unpack(float4 v) { return cpx<dd>{dd(v.x, v.z), dd(v.y, v.w)}; }

    __device__ static __forceinline__ void load_spinor(const SElem *__restrict__ f, int stride, int s, Spinor<R> &p)
    {
#pragma unroll
        for (int k = 0; k < 12; k++) p.v[k / 3][k % 3] = unpack(__ldg(f + (k * stride + s)));
    }
    __device__ static __forceinline__ void load_spinor_rw(const SElem *f, int stride, int s, Spinor<R> &p)
    {
#pragma unroll
        for (int k = 0; k < 12; k++) p.v[k / 3][k % 3] = unpack(f[k * stride + s]);
    }
    __device__ static __forceinline__ void load_chiral(const SElem *__restrict__ f, int stride, int s, int ch, cpx<R> *v)
    {
#pragma unroll
        for (int k = 0; k < 6; k++) v[k] = unpack(__ldg(f + ((6 * ch + k) * stride + s)));
    }
    __device__ static __forceinline__ void load_link(const UElem *__restrict__ U, int V, int mu, int s, Link<R> &L)
    {
        const UElem *b = U + (long)mu * 9 * V;
#pragma unroll
        for (int k = 0; k < 9; k++) L.m[k / 3][k % 3] = unpack(__ldg(b + (k * V + s)));
    }
    // 36 reals of chirality block ch, stored as 18 elements of two (hi, lo) reals each
    __device__ static __forceinline__ void load_clover(const CElem *__restrict__ Cl, int V, int s, int ch, R *c)
    {
        const CElem *b = Cl + (long)ch * 18 * V;
#pragma unroll
        for (int k = 0; k < 18; k++) {
            float4 v = __ldg(b + (k * V + s));
            c[2 * k] = dd(v.x, v.z);
            c[2 * k + 1] = dd(v.y, v.w);
        }
    }
};

}  // namespace ddrw
