// The quantizer of the fully quantized transforms (Section 4.1): one code of Q(v / s) with
// s = amax / 127 in fp64, code = rint(v / s) (half to even), clipped to [-127, 127].  Deciding in
// fp64 makes every code a function of the values alone, not of an instruction order.
#pragma once

#include <cuda_runtime.h>

namespace wfq {

constexpr double kIntQmax = 127.0;

// Q(v / s) by fp64 division.
static __device__ __noinline__ int code_by_division(double v, double s)
{
    const double q = rint(__ddiv_rn(v, s));
    return (int)fmin(fmax(q, -kIntQmax), kIntQmax);
}
// The same code without the division in all but rare cases: a candidate from the reciprocal
// (rinv = 1 / s, one division per scale instead of one per element), its remainder v - q s by one
// fused multiply-add, a step to the neighbour if the remainder says so, and the division itself
// where the remainder is within 1e-9 s of half a step (there the rounding of the quotient
// decides, and the definition is the division).
__device__ __forceinline__ int code_of(double v, double s, double rinv)
{
    double q = rint(__dmul_rn(v, rinv));
    const double r = __fma_rn(-q, s, v);
    const double h = 0.5 * s, ar = fabs(r);
    if (fabs(ar - h) <= 1e-9 * s) return code_by_division(v, s);
    if (ar > h) q += r > 0.0 ? 1.0 : -1.0;
    return (int)fmin(fmax(q, -kIntQmax), kIntQmax);
}
static __device__ __noinline__ int code_exact(float v, float amax)
{
    if (!(amax > 0.f)) return 0;
    const double s = __ddiv_rn((double)amax, kIntQmax);
    return code_of((double)v, s, __ddiv_rn(1.0, s));
}
// The code of an fp32 value of a group with abs-max amax, rinv = fl32(127 / amax).  The fp32 product
// is within 127 * 2^-23 = 1.5e-5 of the quotient: unless that is near the middle between two integers
// (or not finite: amax zero or tiny, infinities, NaN) its nearest integer is the code, in five fp32
// operations instead of a dozen fp64 ones and two conversions.
__device__ __forceinline__ int code_of_float(float v, float amax, float rinv)
{
    const float t = __fmul_rn(v, rinv);
    const float r = __fadd_rn(t, 12582912.f);
    if (fabsf(__fsub_rn(t, __fsub_rn(r, 12582912.f))) < 0.4999f) return __float_as_int(r) - 0x4B400000;
    return code_exact(v, amax);
}

}  // namespace wfq
