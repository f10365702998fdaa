// Helpers of the one-reduction PCG kernels (pcg_reg.cu, pcg_split.cu): sums
// that travel between CTAs as pairs of 8-byte accumulators.
#pragma once

#include "pcg_rows.cuh"

namespace mpcg {

// ||r||^2 term in the accumulator's precision (the exit test alone uses it)
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

// beta = eta / eta_old, with the reciprocal inv of eta_old taken ahead of the
// reduction that brings eta; the quotient itself where the reciprocal overflows
// (eta_old subnormal).  In double one correction step takes the product to
// the rounded quotient; in float the product is as close as __fdividef.
__device__ __forceinline__ float beta_from(float eta, float inv, float eta_old) {
    return fabsf(inv) <= 3.402823466e38f ? __fmul_rn(eta, inv) : __fdiv_rn(eta, eta_old);
}
__device__ __forceinline__ double beta_from(double eta, double inv, double eta_old) {
    if (!(fabs(inv) <= 1.7976931348623157e308)) return eta / eta_old;
    const double b = __dmul_rn(eta, inv);
    return __fma_rn(__fma_rn(-b, eta_old, eta), inv, b);
}

// Every lane of a warp waits (bounded) for the phase of `parity`; true in all
// lanes if any of them gave up.
__device__ __forceinline__ bool warp_wait(uint32_t mbar, uint32_t parity, const volatile int *abort_flag) {
    const bool ok = mbar_wait_bounded_abort(mbar, parity, WAIT_LIMIT_NS, abort_flag);
    return __any_sync(0xffffffffu, !ok) != 0;
}

}  // namespace mpcg
