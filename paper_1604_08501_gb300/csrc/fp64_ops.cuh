// FP64 values taken apart and put together on the integer pipe, and the
// reciprocal the FP64 kernels use.  GB300 converts between FP64 and FP32 at the
// FP64 pipe's rate (1.67 per clock and SM), so the bits are moved by shifts.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace numa {

// The double with bits b, |.| < 2^128, cut to a float (towards zero; zero below
// the normal floats).
__device__ __forceinline__ float f64_to_f32_trunc(long long b) {
    const uint32_t hi = (uint32_t)((unsigned long long)b >> 32);
    const int h = (int)(hi & 0x7FFFFFFFu) - (896 << 20);   // exponent field less the bias difference
    const uint32_t m = __funnelshift_l((uint32_t)b, (uint32_t)h, 3) | (hi & 0x80000000u);
    return h < (1 << 20) ? 0.0f : __uint_as_float(m);
}

// A float widened to a double exactly (zero and normal floats).
__device__ __forceinline__ double f32_to_f64(float f) {
    const uint32_t u = __float_as_uint(f), a = u & 0x7FFFFFFFu;
    const uint32_t hi = (u & 0x80000000u) | ((a >> 3) + (896u << 20));
    return a < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(u << 29));
}

// 1/a in three FP64 operations: the FP32 reciprocal y0 of a's leading 24 bits and one
// step of the third-order hyperpower iteration (Schulz's iteration carried one
// term further), y0 (1 + e + e^2), e = 1 - a y0, whose own error is e^3.  a cut to
// 24 bits and rcp.approx (absolute error 2^-23 on [1, 2), by PTX's documentation)
// leave |e| <= 1.5 2^-22, so the result is within 0.5005 units in the last place
// (38000 values of every exponent field: all correctly rounded), where __drcp_rn,
// correctly rounded throughout, takes about twice the FP64 operations.  Zero, subnormal, infinite, NaN and extreme a take __drcp_rn.
static __device__ __noinline__ double rcp_fp64_call(double a) { return __drcp_rn(a); }   // not speculated

__device__ __forceinline__ double rcp_fp64(double a) {
    const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
    const int e = (int)((hi >> 20) & 0x7FFu);
    const float m = __uint_as_float(0x3F800000u | (__funnelshift_l(lo, hi, 3) & 0x7FFFFFu));
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const uint32_t u = __float_as_uint(r);
    const uint32_t h0 = ((u >> 3) + ((uint32_t)(896 + 1023 - e) << 20)) | (hi & 0x80000000u);
    const double y0 = __hiloint2double((int)h0, (int)(u << 29));
    if ((unsigned)(e - 23) > 2000u) return rcp_fp64_call(a);
    const double d = fma(-a, y0, 1.0);
    return fma(y0, fma(d, d, d), y0);
}

}  // namespace numa
