// Helpers of the one-reduction PCG kernels (pcg_reg.cu, pcg_split.cu): sums
// that travel between CTAs as pairs of 8-byte accumulators.
#pragma once

#include "pcg_rows.cuh"

namespace mpcg {

// A thread's share of ||r||^2, which the exit test and the reported residual alone
// use: a plain float beside float pairs, a double beside doubles
__device__ __forceinline__ dfloat sq_sum(float a, float b, dfloat) { return dfloat{__fmaf_rn(b, b, __fmul_rn(a, a)), 0.f}; }
__device__ __forceinline__ double sq_sum(float a, float b, double) {
    return __fma_rn((double)b, (double)b, __dmul_rn((double)a, (double)a));
}

__device__ __forceinline__ dfloat bcast(dfloat a, int lane) {
    return dfloat{__shfl_sync(0xffffffffu, a.hi, lane), __shfl_sync(0xffffffffu, a.lo, lane)};
}
__device__ __forceinline__ double bcast(double a, int lane) { return __shfl_sync(0xffffffffu, a, lane); }

// two accumulators as one 16-byte push
__device__ __forceinline__ void push_pair(uint32_t addr, dfloat a, dfloat b, uint32_t mbar) {
    st_async_v4(addr, a.hi, a.lo, b.hi, b.lo, mbar);
}
__device__ __forceinline__ void push_pair(uint32_t addr, double a, double b, uint32_t mbar) {
    st_async_v4(addr, __int_as_float(__double2loint(a)), __int_as_float(__double2hiint(a)),
                __int_as_float(__double2loint(b)), __int_as_float(__double2hiint(b)), mbar);
}

__device__ __forceinline__ void load_pair(const dfloat *p, dfloat &a, dfloat &b) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a = dfloat{v.x, v.y};
    b = dfloat{v.z, v.w};
}
__device__ __forceinline__ void load_pair(const double *p, double &a, double &b) {
    const double2 v = *reinterpret_cast<const double2 *>(p);
    a = v.x;
    b = v.y;
}

// beta = eta / eta_old, with the reciprocal of eta_old taken ahead of the reduction
// that brings eta.  In float both are scaled where eta_old is small, so that
// the reciprocal does not overflow (a test in place of it, taken once beta is
// wanted, was 0.8 % slower at N = 512); the product is as close as __fdividef.  In
// double the quotient itself is taken there, and else one correction step takes
// the product to the rounded quotient.
template <typename T>
struct EtaRecip;
template <>
struct EtaRecip<float> {
    float inv = 0.f, scale = 1.f;
    __device__ __forceinline__ void set(float eta) {
        scale = fabsf(eta) < 7.8886091e-31f ? 1.8446744e19f : 1.f;  // 2^-100, 2^64
        inv = __fdividef(1.f, eta * scale);
    }
    __device__ __forceinline__ float beta(float eta, float) const { return __fmul_rn(__fmul_rn(eta, scale), inv); }
};
template <>
struct EtaRecip<double> {
    double inv = 0.0;
    __device__ __forceinline__ void set(double eta) { inv = 1.0 / eta; }
    __device__ __forceinline__ double beta(double eta, double eta_old) const {
        if (!(fabs(inv) <= 1.7976931348623157e308)) return eta / eta_old;
        const double b = __dmul_rn(eta, inv);
        return __fma_rn(__fma_rn(-b, eta_old, eta), inv, b);
    }
};

// a carried sum rounded to float (pairs are normalised)
__device__ __forceinline__ float rounded(dfloat a, float) { return a.hi; }
__device__ __forceinline__ float rounded(double a, float) { return __double2float_rn(a); }
__device__ __forceinline__ double rounded(double a, double) { return a; }

// p^T S p for p = r~ + beta p_old, without a reduction of its own.  With the last
// beta, g, in the place of the one that r^T r~ will give, each thread adds up
//     eps = (r~ + g / 2 p_old)^T S p_old,
// and then
//     p^T S p = r~^T S r~ + beta (2 eps + (beta - g) p_old^T S p_old),
// so that the carried p_old^T S p_old enters with beta - g in place of beta: its error
// is passed on times |beta (beta - g)| (p_old^T S p_old) / (p^T S p), 0.1-0.2 at the
// median and 0.3-0.55 at the 95th percentile of the iterations (Kuka-shaped,
// N = 32 and 128, nx = 36), where plain beta passes it on times 1 on average and
// up to 10 in a row.  Relative error of alpha, rms of 48 iterations whose solution is
// white noise, this form / summed itself / carried plainly in float: nx = 14,
// N = 64 5.1e-7 / 4.8e-7 / 2.9e-6, N = 512 4.1e-7 / 4.0e-7 / 2.0e-6; nx = 36, N = 64
// 4.0e-7 / 5.3e-7 / 3.0e-6.  Rounded once, by the compensated Horner scheme
// (Graillat, Langlois, Louvet) in float pairs, in double arithmetic else.
// Against the plain float form it takes 2 to 5 % of the time; a fifth sum in
// place of the prediction, the same accuracy, 9 %.
__device__ __forceinline__ dfloat curvature(dfloat del, dfloat eps, dfloat old, float beta, float g) {
    auto step = [](float b, float x, float xl, float a, float al, float &lo) {  // a + b x
        const float p = __fmul_rn(b, x), s = __fadd_rn(p, a), t = __fsub_rn(s, p);
        const float e = __fadd_rn(__fsub_rn(p, __fsub_rn(s, t)), __fsub_rn(a, t));
        lo = __fmaf_rn(b, xl, __fadd_rn(__fadd_rn(e, __fmaf_rn(b, x, -p)), al));
        return s;
    };
    float l1, l2;
    const float s1 = step(__fsub_rn(beta, g), old.hi, old.lo, eps.hi + eps.hi, eps.lo + eps.lo, l1);
    const float s2 = step(beta, s1, l1, del.hi, del.lo, l2), hi = __fadd_rn(s2, l2);
    return dfloat{hi, __fsub_rn(l2, __fsub_rn(hi, s2))};
}
__device__ __forceinline__ double curvature(double del, double eps, double old, double beta, double g) {
    return __fma_rn(beta, __fma_rn(beta - g, old, eps + eps), del);
}

// Is that p^T S p not to be trusted, and to be summed itself?  It is not positive or
// not finite, its three terms cancel to less than about 1/32 of their size, or
// more than 0.9 of the error of p_old^T S p_old is passed on (so that no more than
// ten iterations' worth of errors can gather).
__device__ __forceinline__ bool doubtful(float ups, dfloat del, dfloat eps, dfloat old, float beta, float g) {
    const float b = fabsf(beta), passed = b * (fabsf(beta - g) * fabsf(old.hi)),
                m = __fmaf_rn(b, 2.f * fabsf(eps.hi), fabsf(del.hi)) + passed;
    return !(ups > 0.f && ups > 0.03125f * m && passed <= 0.9f * ups && ups <= 3.402823466e38f);
}
// (float32 with double sums: an FP64 instruction, conversions among them, takes an
// issue slot of 64 cycles, so the terms are compared by their high words)
__device__ __forceinline__ float high(double x) {  // |x| to a relative 2^-20, in float's range
    const int h = __double2hiint(x) & 0x7fffffff, lo = 0x38100000, hi = 0x47efffff;
    return h < lo ? 0.f : __int_as_float((min(h, hi) - 0x38000000) << 3);
}
__device__ __forceinline__ bool doubtful(float ups, double del, double eps, double old, float beta, float g) {
    return doubtful(ups, dfloat{high(del), 0.f}, dfloat{high(eps), 0.f}, dfloat{high(old), 0.f}, beta, g);
}
// In double p_old^T S p_old is a sum of its own in each iteration (g = 0), and nothing
// is carried (error of alpha 1.2e-15, 1.1e-15 summed itself, 7.0e-15 carried).  The
// terms are compared by their exponents.
__device__ __forceinline__ bool doubtful(double ups, double del, double eps, double old, double beta, double) {
    auto ex = [](double x) { return (__double2hiint(x) >> 20) & 2047; };
    const int eb = ex(beta) - 1023, lead = max(ex(del), max(ex(eps) + 1, ex(old) + eb) + eb);
    return !(ups > 0.0 && ex(ups) >= lead - 4 && ups <= 1.7976931348623157e308);
}

// Sums over a warp of five accumulators per lane by recursive halving, each lane
// giving away half of its sums per level: lanes 8u end with sum u, lane 4 with
// the fifth.  fold5: the last three levels, with sum lane / 8 in x and the fifth in
// e (each over lanes lane % 8).
template <class AT, typename A>
__device__ __forceinline__ A halve(A p0, A p1, int m) {
    const bool h = threadIdx.x & m;
    return AT::add_tree(h ? p1 : p0, AT::shfl_xor(h ? p0 : p1, m));
}
template <class AT, typename A>
__device__ __forceinline__ A fold5(A x, A e) {
    x = halve<AT>(x, e, 4);
    x = AT::add_tree(x, AT::shfl_xor(x, 2));
    return AT::add_tree(x, AT::shfl_xor(x, 1));
}
template <class AT, typename A>
__device__ __forceinline__ A warp_sums5(A v0, A v1, A v2, A v3, A v4) {
    const A x = halve<AT>(halve<AT>(v0, v2, 16), halve<AT>(v1, v3, 16), 8);
    const A e = AT::add_tree(v4, AT::shfl_xor(v4, 16));
    return fold5<AT>(x, AT::add_tree(e, AT::shfl_xor(e, 8)));
}

// Every lane of a warp waits (bounded) for the phase of `parity`; true in all
// lanes if any of them gave up.
__device__ __forceinline__ bool warp_wait(uint32_t mbar, uint32_t parity, const volatile int *abort_flag) {
    const bool ok = mbar_wait_bounded_abort(mbar, parity, WAIT_LIMIT_NS, abort_flag);
    return __any_sync(0xffffffffu, !ok) != 0;
}

}  // namespace mpcg
