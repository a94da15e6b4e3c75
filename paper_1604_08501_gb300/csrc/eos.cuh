// Pressure perturbation p' = p(Theta) - p(Theta_ref) for the native FP64 and
// the mixed-precision kernels (equation of state of Sec. 2:
// p = p0 (R Theta / p0)^gamma, gamma = cp / (cp - R)).
//
// Both evaluate p' = p_ref ((1 + x)^gamma - 1) with x = Theta'/Theta_ref,
// written A Theta' g(x) with A = p_ref / Theta_ref and
// g(x) = sum_k binom(gamma, k) x^(k-1).  That is the same quantity as the
// difference of two pressures, without its cancellation.
//
// FP64 has three forms, each accurate to a few ulps over its whole range:
// the series to 9 terms for |x| <= 1/64 (the last four in FP32 where they are
// below 2^-34 of the sum, as for any gamma near 1.4: FP32's error is then below
// 2^-58 of it) and to 15 terms for |x| <= 1/8
// (truncation below 2^-55 relative for gamma near 1.4), and
// p_ref expm1(gamma log1p(x)) for any x > -1.  A warp takes the widest form
// any of its lanes needs, so that a warp never runs several of them one after
// the other: states advanced over many stages drift past 1/64, and on fine
// meshes past 1/8.  Where Theta_ref = 0 (w and A not finite) or x <= -1 the
// definition, two evaluations of the equation of state, is used.
// FP32 likewise: 5 terms for |x| <= 1/64, 16 terms for |x| <= 1/2 (truncation
// below 2^-26), expm1f(gamma log1pf(x)) beyond, chosen per warp.
#pragma once

#include "fp64_ops.cuh"
#include "kernel_params.h"

namespace numa {

// p0 (R Theta / p0)^gamma, the equation of state of Sec. 2.  Not inlined:
// the rhs kernel calls it only where the series does not apply, and keeping
// pow out of line keeps its registers out of the kernel's budget.
static __device__ __noinline__ double eos_pressure(double Th, const EosConstants &c) {
    return __dmul_rn(c.p0, pow(__ddiv_rn(__dmul_rn(c.R, Th), c.p0), c.gamma));
}

// The active lanes of the calling lane's group of GROUP lanes.
template <int GROUP>
static __device__ __forceinline__ unsigned vote_mask() {
    unsigned lanes = __activemask();
    if constexpr (GROUP < 32) {
        unsigned lane;
        asm("mov.u32 %0, %%laneid;" : "=r"(lane));
        lanes &= ((1u << GROUP) - 1u) << (lane & ~(GROUP - 1u));
    }
    return lanes;
}

// p' of one point; the form is chosen per warp (see above), or per GROUP lanes.
// Every active lane of the group must call it together.
// Params: NativeParams or HighParams (the series coefficients c and eos).
template <int GROUP = 32, typename Params>
static __device__ __forceinline__ double pressure_perturbation(double Th, double th0, double w, double A,
                                                        const Params &P) {
    const double thp = Th - th0;              // Theta'
    const double x = thp * w;                 // Theta' / Theta_ref
    // |x| compared as bits, on the integer pipe (a NaN's are larger)
    const long long xb = __double_as_longlong(x);
    const unsigned long long ab = (unsigned long long)xb & 0x7FFFFFFFFFFFFFFFull;
    const double ax = fabs(x);
    const unsigned lanes = vote_mask<GROUP>();
    if (__all_sync(lanes, ab <= 0x3F90000000000000ull)) {   // 1/64
        double g;
        if (P.tail_f32) {   // uniform
            const float xf = f64_to_f32_trunc(xb);
            float t = P.ct[3];
#pragma unroll
            for (int k = 2; k >= 0; --k) t = fmaf(t, xf, P.ct[k]);
            g = f32_to_f64(t);
        } else {
            g = P.c[8];
#pragma unroll
            for (int k = 7; k >= 5; --k) g = fma(g, x, P.c[k]);
        }
#pragma unroll
        for (int k = 4; k >= 0; --k) g = fma(g, x, P.c[k]);   // sum_k c_{k+1} x^k
        return (A * thp) * g;
    }
    if (__all_sync(lanes, ab <= 0x3FC0000000000000ull)) {   // 1/8
        double g = P.c[14];
#pragma unroll
        for (int k = 13; k >= 0; --k) g = fma(g, x, P.c[k]);
        return (A * thp) * g;
    }
    // x > -1 and finite (a NaN fails the comparison, an infinite x fails < 2^1000)
    if (__all_sync(lanes, x > -1.0 && ax < 1e300))
        return (A * th0) * expm1(P.eos.gamma * log1p(x));
    return eos_pressure(Th, P.eos) - eos_pressure(th0, P.eos);
}

// FP32 form from the perturbation Theta' itself (mixed precision): the series
// (5 or 16 terms) or expm1f(gamma log1pf(x)), chosen per warp as in FP64 (N = 8..15:
// per point), all free of cancellation.
// A = K Theta_ref^(gamma - 1) with K = p0^(1 - gamma) R^gamma is recomputed
// from Theta_ref instead of being read from memory.  eos_reference_f32 forms
// the per-point factors (w = 1/Theta_ref and A), which a caller that keeps a
// point for many evaluations computes once.
struct EosRef32 {
    float w, A;
};

template <typename Params>
static __device__ __forceinline__ EosRef32 eos_reference_f32(float th0, const Params &P) {
    return EosRef32{__frcp_rn(th0), P.K * exp2f(P.gm1 * log2f(th0))};   // A = p(Theta_ref)/Theta_ref
}

// p' by the first TERMS terms of the series, sum_k c_{k+1} x^k.
template <int TERMS, typename Params>
static __device__ __forceinline__ float eos_series_f32(float thp, float x, float A, const Params &P) {
    float g = P.c[TERMS - 1];
#pragma unroll
    for (int k = TERMS - 2; k >= 0; --k) g = fmaf(g, x, P.c[k]);
    return (A * thp) * g;
}

// Params: MixedParams or HighParams32 (c, K, gm1, gamma).  GROUP = 1: each point its
// own form, for the kernels of N = 8..15, which share an element out to warps in
// two ways and give it the same result (a warp whose points all take the short
// series still runs nothing else; without that N = 15 took 108.4 us instead of 103.3).
template <int GROUP = 32, typename Params>
static __device__ __forceinline__ float pressure_perturbation_f32(float thp, float th0, EosRef32 r,
                                                           const Params &P) {
    const unsigned lanes = vote_mask<GROUP == 1 ? 32 : GROUP>();
    if (__all_sync(lanes, th0 > 0.0f)) {
        const float x = thp * r.w;
        const float ax = fabsf(x);
        if (__all_sync(lanes, ax <= 0.015625f)) return eos_series_f32<5>(thp, x, r.A, P);
        if constexpr (GROUP > 1) {
            if (__all_sync(lanes, ax <= 0.5f)) return eos_series_f32<16>(thp, x, r.A, P);
            if (__all_sync(lanes, x > -1.0f)) return (r.A * th0) * expm1f(P.gamma * log1pf(x));
        }
    }
    if constexpr (GROUP == 1) {
        const float x = thp * r.w;
        const float ax = fabsf(x);
        if (th0 > 0.0f && ax <= 0.015625f) return eos_series_f32<5>(thp, x, r.A, P);
        if (th0 > 0.0f && ax <= 0.5f) return eos_series_f32<16>(thp, x, r.A, P);
    }
    // Theta_ref = 0 (the paper's full-pressure form): p' = p(Theta'); and,
    // per lane, whatever the warp's common forms do not cover.
    if (th0 > 0.0f) return (r.A * th0) * expm1f(P.gamma * log1pf(thp * r.w));
    return P.K * powf(thp, P.gamma);
}

template <int GROUP = 32, typename Params>
static __device__ __forceinline__ float pressure_perturbation_f32(float thp, float th0,
                                                           const Params &P) {
    if (th0 > 0.0f) return pressure_perturbation_f32<GROUP>(thp, th0, eos_reference_f32(th0, P), P);
    return P.K * powf(thp, P.gamma);
}

}  // namespace numa
