// blas.cuh -- declarations of the vector kernels and reductions (blas.cu).
#pragma once

#include "../../include/ddrw.h"
#include "ddrw_internal.cuh"

namespace ddrw {

// Krylov scalars of one right-hand side, resident on the device.
struct KScal {
    double2 rho, alpha, omega, beta;
    double rr;      // ||r||^2 of the current iterate
    double thresh;  // stop when rr <= thresh (tol^2 ||b||^2)
    int active;     // 0 once converged, stalled or broken down
    int iters;
    int maxiter;
    int breakdown;  // 0 none, else the step that found a zero denominator or NaN
};

// sites [off, off + n) of every plane (plane stride V), nrhs right-hand sides rs elements apart
struct VecRange {
    long V, off, n, rs;
    int nrhs;
};

template <class P> struct Blas {
    using E = typename P::SElem;
    static ddrw_status bicg_init(ddrw_ctx *ctx, const VecRange &vr, E *r, E *rh, E *p, E *x, KScal *sc);
    static ddrw_status bicg_alpha(ddrw_ctx *ctx, const VecRange &vr, const E *rh, const E *v, KScal *sc);
    static void bicg_s(ddrw_ctx *ctx, const VecRange &vr, E *r, const E *v, const KScal *sc);
    static ddrw_status bicg_omega(ddrw_ctx *ctx, const VecRange &vr, const E *t, const E *r, const E *rh, KScal *sc);
    static ddrw_status bicg_xrp(ddrw_ctx *ctx, const VecRange &vr, E *x, E *p, E *r, const E *t, const E *v, const E *rh,
                                KScal *sc);
    static ddrw_status norm2(ddrw_ctx *ctx, const VecRange &vr, const E *f, double *out);
    static ddrw_status norm_dot(ddrw_ctx *ctx, const VecRange &vr, const E *d, const E *e, double *out);
    static void axpby(ddrw_ctx *ctx, const VecRange &vr, double a, const E *x, double b, E *y);
};

// ----------------------------------------------------------------------------- reductions
// (deterministic grid-wide sums shared by the vector kernels of blas.cu and sap.cu)

// A running sum: FP64 for FP64 fields; for FP32 arithmetic an unevaluated pair hi + lo (Knuth's
// two-sum, about 48 significant bits against the 24 of the terms, in the range of a float: sums of FP32
// products, whose vectors are scaled to unit right-hand sides).  GB300 adds FP64 at 1/64 of its FP32
// rate: with FP64 shuffle steps in every warp and FP64 sums over the warps, the reductions took longer
// than the fields' passes (bicg_omega on 12 x 65536 FP16 sites 43 us, against 14 us for the
// three passes of bicg_s, which does not reduce).
template <typename R> struct RunSum;
template <> struct RunSum<double> {
    using Raw = double;
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void join(Raw o) { s += o; }
    __device__ __forceinline__ Raw raw() const { return s; }
    __device__ __forceinline__ double value() const { return s; }
    template <int W> __device__ __forceinline__ void shuffle_sum()  // lane 0: the sum over lanes 0 .. W - 1
    {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
};
template <> struct RunSum<float> {
    using Raw = float2;
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void join(Raw o)
    {
        const float s = __fadd_rn(hi, o.x), v = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(o.y, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(o.x, v))));
        hi = s;
    }
    __device__ __forceinline__ void add(float x) { join(make_float2(x, 0.f)); }
    __device__ __forceinline__ Raw raw() const { return make_float2(hi, lo); }
    // an overflowed or NaN sum is reported as hi gives it (lo is then NaN)
    __device__ __forceinline__ double value() const { return (double)hi + (lo - lo == 0.f ? (double)lo : 0.0); }
    template <int W> __device__ __forceinline__ void shuffle_sum()
    {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) {
            Raw q;
            q.x = __shfl_down_sync(0xffffffffu, hi, o);
            q.y = __shfl_down_sync(0xffffffffu, lo, o);
            join(q);
        }
    }
};

// Sums of products over the components k = 0, 1, ... of a site (unrolled loops), in chains of four: a chain of
// all twelve, 24 terms deep, rounds 1.25 times as much as adding up |z|^2 or conj(a) b component by component,
// chains of four 0.8 times (rms error against 64 bits, 128 to 131072 sites), for one more addition per chain.
template <typename R> struct SiteNorm {
    R s = R(0), c = R(0);
    __device__ __forceinline__ void add(int k, cpx<R> z)  // += |z|^2
    {
        if (k > 0 && k % 4 == 0) s += c, c = R(0);
        c = fmad(z.re, z.re, fmad(z.im, z.im, c));
    }
    __device__ __forceinline__ R total() const { return s + c; }
};
template <typename R> struct SiteDot {
    cpx<R> s = {R(0), R(0)}, c = {R(0), R(0)};
    __device__ __forceinline__ void add(int k, cpx<R> a, cpx<R> b)  // += conj(a) b
    {
        if (k > 0 && k % 4 == 0) s = s + c, c = {R(0), R(0)};
        cmacc(c, a, b);
    }
    __device__ __forceinline__ cpx<R> total() const { return s + c; }
};

// Warp totals of K running sums at once: while several sums are left, each exchange step also halves the
// sums a lane keeps, so K = 7 takes 9 additions per lane instead of 35 (FP64 additions are what these
// reductions wait for).  Afterwards lane l holds the total of sum l >> SHIFT.
template <int K, typename R> struct WarpSums {
    static constexpr int M = K <= 1 ? 1 : K <= 2 ? 2 : K <= 4 ? 4 : 8;
    static constexpr int SHIFT = M == 1 ? 5 : M == 2 ? 4 : M == 4 ? 3 : 2;
    __device__ static __forceinline__ typename RunSum<R>::Raw xchg(typename RunSum<R>::Raw a, int o)
    {
        if constexpr (sizeof(R) == 8) {
            return __shfl_xor_sync(0xffffffffu, a, o);
        } else {
            a.x = __shfl_xor_sync(0xffffffffu, a.x, o);
            a.y = __shfl_xor_sync(0xffffffffu, a.y, o);
            return a;
        }
    }
    __device__ static __forceinline__ RunSum<R> total(const RunSum<R> (&v)[K])
    {
        RunSum<R> t[M];
#pragma unroll
        for (int k = 0; k < K; k++) t[k] = v[k];
#pragma unroll
        for (int o = 16, m = M; o > 0; o >>= 1) {
            if (m > 1) {
                m >>= 1;
                const bool up = (threadIdx.x & o) != 0;
#pragma unroll
                for (int k = 0; k < M / 2; k++)
                    if (k < m) {
                        const RunSum<R> keep = up ? t[k + m] : t[k], send = up ? t[k] : t[k + m];
                        t[k] = keep;
                        t[k].join(xchg(send.raw(), o));
                    }
            } else {
                t[0].join(xchg(t[0].raw(), o));
            }
        }
        return t[0];
    }
};

// CTA totals of v[0..K): sum k in out[k] (shared memory), complete after the caller's next __syncwarp of
// warp 0 (whose lanes write it) or a barrier; sm and out are used again only after a barrier
template <int K, int NT, typename R>
__device__ __forceinline__ void cta_sum_run(RunSum<R> (&v)[K], typename RunSum<R>::Raw (*sm)[K],
                                            typename RunSum<R>::Raw (&out)[K])
{
    using WS = WarpSums<K, R>;
    constexpr int NW = NT / 32;
    static_assert(NW == 8, "eight warps");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const RunSum<R> t = WS::total(v);
    const int k = lane >> WS::SHIFT;
    if ((lane & ((1 << WS::SHIFT) - 1)) == 0 && k < K) sm[w][k] = t.raw();
    __syncthreads();
    if (w == 0)
#pragma unroll
        for (int k0 = 0; k0 < K; k0 += 4) {  // four sums at a time, eight lanes each
            const int kk = k0 + (lane >> 3);
            RunSum<R> q;
            if (kk < K) q.join(sm[lane & 7][kk]);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) q.join(WS::xchg(q.raw(), o));
            if ((lane & 7) == 0 && kk < K) out[kk] = q.raw();
        }
}

// Sum v[0..K) over the grid's CTAs for right-hand side blockIdx.y.  Returns true in thread 0 of the
// last CTA, with the totals in out.  part: [nrhs][gridDim.x][K] 8-byte partial sums, ticket:
// [nrhs] zeroed.
template <int K, int NT, typename R>
__device__ bool grid_sum_run(RunSum<R> (&v)[K], double (&out)[K], double *part, unsigned *ticket)
{
    using Raw = typename RunSum<R>::Raw;
    __shared__ Raw sm[NT / 32][K], tot[K];
    __shared__ bool last;
    const int r = blockIdx.y, G = gridDim.x;
    Raw *pp = reinterpret_cast<Raw *>(part) + (long)r * G * K;
    cta_sum_run<K, NT, R>(v, sm, tot);
    if (threadIdx.x < 32) {
        __syncwarp();
        if (threadIdx.x < K) pp[(long)blockIdx.x * K + threadIdx.x] = tot[threadIdx.x];
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) {
            unsigned t = atomicAdd(ticket + r, 1u);
            last = (t == (unsigned)(G - 1));
        }
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < K; k++) v[k] = RunSum<R>();
    for (int i = threadIdx.x; i < G; i += NT)
#pragma unroll
        for (int k = 0; k < K; k++) v[k].join(__ldcg(pp + (long)i * K + k));
    cta_sum_run<K, NT, R>(v, sm, tot);
    if (threadIdx.x >= 32) return false;
    __syncwarp();
    if (threadIdx.x != 0) return false;
    RunSum<R> q;
#pragma unroll
    for (int k = 0; k < K; k++) {
        q = RunSum<R>();
        q.join(tot[k]);
        out[k] = q.value();
    }
    ticket[r] = 0;
    return true;
}

// the same from per-thread FP64 values, in place
template <int K, int NT> __device__ bool grid_sum(double (&v)[K], double *part, unsigned *ticket)
{
    RunSum<double> q[K];
#pragma unroll
    for (int k = 0; k < K; k++) q[k].s = v[k];
    return grid_sum_run<K, NT, double>(q, v, part, ticket);
}

// alpha (mode 1) or omega (mode 2) of the BiCGStab recurrence from the per-warp partial sums of a
// fused stencil epilogue (DslashCall::red), nwt times RED_PARTS 8-byte partial sums per right-hand side
void bicg_fin(ddrw_ctx *ctx, int mode, int nrhs, const double *part, long nwt, KScal *sc);

// partial-sum and ticket buffers of grid_sum for nrhs right-hand sides (at most 608 CTAs per
// right-hand side and 8 doubles per CTA)
ddrw_status reduce_ws(ddrw_ctx *ctx, int nrhs, double **part, unsigned **ticket);

// FP64 fields <-> storage precision P (FP32, FP16, BF16) over a range, with a per-right-hand-side
// scale (may be null); rsl is the field stride of the P fields
template <class P>
void to_low(ddrw_ctx *ctx, const VecRange &vr, long rsl, const double2 *in, typename P::SElem *out,
            const double *scale);
// x += scale e (first: x = scale e); xs, if given, receives the split copy of x (double-single residual)
template <class P>
void add_low(ddrw_ctx *ctx, const VecRange &vr, long rsl, const typename P::SElem *e, double2 *x, const double *scale,
             bool first = false, float4 *xs = nullptr);
// FP32 field (stride vr.rs) -> 16-bit field (stride rs16) over the range; and x32 += x16, x16 = 0
template <class P16>
void f32_to_16(ddrw_ctx *ctx, const VecRange &vr, long rs16, const float4 *in, typename P16::SElem *out);
template <class P16>
void fold_16_into_32(ddrw_ctx *ctx, const VecRange &vr, long rs16, typename P16::SElem *x16, float4 *x32);
// FP32 link / clover planes -> 16-bit planes of the same order (n float4 elements; bf: BF16, else FP16)
void f32_to_low(ddrw_ctx *ctx, const float4 *in, uint2 *out, long n, bool bf);

}  // namespace ddrw
