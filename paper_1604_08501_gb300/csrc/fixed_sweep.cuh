// The D sweep of one line of FP64 fluxes in 64-bit fixed point.
//
// GB300 issues 1.67 DFMA per clock and SM (measured) but about 30 multiply-adds of
// 32 x 32 + 64 bits and 60 other integer operations, and an even-odd sweep in
// FP64 (element_sweep.cuh) is 90 of the volume term's 157 FP64 operations per
// point at Nq = 8.  Here the sums run on the integer pipes, beside the FP64
// pipe, and are more accurate than in FP64:
//
//  * The thread of a line takes the largest exponent field e of its Nq fluxes
//    and writes each as an integer X with F = X 2^(e - 1080), |X| < 2^58: the 53
//    significant bits of the largest flux, and 5 bits below.
//  * E_m = X_m + X_{N-m} and O_m = X_m - X_{N-m} are exact, below 2^59.
//  * D is an integer too, D 2^s rounded to nearest, s such that the largest sum
//    of |D[i][n]| over a row is at most 2^58.  Both are cut at bit 28 into
//    32-bit words, E = Eh 2^28 + El (0 <= El < 2^28) and D = Dh 2^28 + Dl
//    (|Dl| <= 2^27), and
//      sum D E / 2^56 = sum Eh Dh + (sum (Eh Dl + El Dh)) / 2^28 + (sum El Dl) / 2^56.
//    The first sum is exact (below 2^60), the second too (at most 9 terms below
//    2^59 each) and its quotient is rounded down; the third, below 4.5, is
//    dropped.  Three multiply-adds per product.
//  * S_i = a_i + b_i and S_{N-i} = b_i - a_i, |S| <= 2^60, replace the line's
//    fluxes; the value is S 2^(e - 1024 - s).  Phase 3 adds a point's three sums
//    as integers at the largest of their exponents (|sum| <= 3 2^60), multiplies
//    them by J^-1 as integers and rounds once to FP64 (fixed_sums).
//
// Measured: vol_rhs_fp64_kernel at N = 7, 32768 elements, 4.949 -> 1.881 ms; the
// FP64 batch 2.07 times as fast.  (Rounded before an FP64 multiply by J^-1, one
// test for each field; all fields' integer chains side by side: see vol_fp64.cu.)
//
// Error: at most 1 in each X and 2^-1 in each integer D entry, so at most
// 2^-55 (largest |D| row sum) (largest flux of the line), as a bound; the
// rounding errors of the FP64 sweep of such a line are 2^-53 of its partial
// sums.  tests/test_fixed_sweep_host.py holds it to that bound and to at most
// the FP64 sweep's error, over random, smooth and graded lines of every Nq.
//
// Nq = 2 keeps the FP64 sweep: its D is +-1/2, so that FP64 rounds only sums and
// differences, and the fixed-point sum of three directions, cut at 2^-58 of the
// largest line, was less exact (6.0e-18 against 8.7e-19 of the line's scale on
// smooth lines, where the sums are far smaller than the fluxes).
//
// Lines whose largest exponent field is outside [kFixMinExp, kFixMaxExp]
// (infinities, NaN, values that could overflow, lines of tiny values) take the
// FP64 sweep: their exponent is kFixNone and the slots hold doubles.  A line
// of zeros is a line of integer zeros.
#pragma once

#include <cstdint>
#include <cstring>

#include "element_sweep.cuh"
#include "kernel_params.h"

namespace numa {

constexpr int kFixMinExp = 200, kFixMaxExp = 1900;
constexpr int kFixNone = -1;      // exponent of a line left in FP64

// Orders whose lines are swept in fixed point.
template <int NQ>
__host__ __device__ constexpr bool fixed_point() {
    return NQ > 2;
}

__host__ __device__ __forceinline__ long long fix_bits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    std::memcpy(&b, &x, sizeof b);
    return b;
#endif
}

__host__ __device__ __forceinline__ double fix_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    std::memcpy(&x, &b, sizeof x);
    return x;
#endif
}

// x >> n for any n >= 0 (n >= 64: all sign bits).
__host__ __device__ __forceinline__ long long fix_shr(long long x, int n) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));   // clamps n
    return r;
#else
    return x >> (n > 63 ? 63 : n);
#endif
}

__host__ __device__ __forceinline__ int fix_clz(unsigned long long x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// X of the double with bits b, in a line of largest exponent field e: its
// mantissa with the hidden bit at bit 57, shifted down by the difference of
// the exponents (towards zero), with its sign.  Zeros and subnormals shift out.
__host__ __device__ __forceinline__ long long fix_from_bits(long long b, int e) {
    const uint32_t hi = (uint32_t)((unsigned long long)b >> 32);
    const int d = e - (int)((hi >> 20) & 0x7FFu);
    const long long m =
        (long long)((((unsigned long long)((hi & 0xFFFFFu) | 0x100000u)) << 32 | (uint32_t)b)
                    << (kFixBits - 53));
    const long long a = fix_shr(m, d), s = b >> 63;
    return (a ^ s) - s;
}

// The integer R, |R| < 2^63, times 2^(e - 1024 - s), rounded to nearest (ties
// away from zero).  kFixMinExp and kFixMaxExp keep the result normal.
__host__ __device__ __forceinline__ double fix_to_double(long long R, int e, int shift) {
    const long long s = R >> 63;
    const unsigned long long a = (unsigned long long)((R ^ s) - s);
    const int lz = fix_clz(a);
    const unsigned long long m = a << (lz & 63);   // leading bit at 63
    // exponent field of 2^(63 - lz) 2^(e - 1024 - s), less the hidden bit's one
    const int E = e - shift + 61 - lz;
    const unsigned long long v = ((unsigned long long)(uint32_t)E << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return a == 0ull ? 0.0 : fix_double((long long)(v | ((unsigned long long)s & (1ull << 63))));
}

__host__ __device__ __forceinline__ unsigned long long fix_mulhi(unsigned long long a,
                                                                 unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}

// -y R 2^(e - 1024 - s), rounded once (to nearest, ties away from zero): the
// integer's leading 64 bits times the 53 of y (exponent field ey), a multiply
// on the integer pipes.  ok is cleared where the product is not a normal number.
__host__ __device__ __forceinline__ double fix_scale(long long R, int e, int shift, double y, int ey,
                                                     bool &ok) {
    const long long yb = fix_bits(y);
    const long long s = R >> 63;
    const unsigned long long a = (unsigned long long)((R ^ s) - s);
    const int lz = fix_clz(a);
    // y's mantissa with its hidden bit at 63; the product in [2^62, 2^64)
    const unsigned long long my = ((unsigned long long)yb << 11) | (1ull << 63);
    unsigned long long p = fix_mulhi(a << (lz & 63), my);
    const int up = (long long)p < 0 ? 0 : 1;
    p <<= up;
    // exponent field of 2^(63 - lz) 2^(e - 1024 - s) y, less the hidden bit's one
    const int E = e - shift + 61 - lz + ey - 1023 + 1 - up;
    const unsigned long long v = ((unsigned long long)(uint32_t)E << 52) + (p >> 11) + ((p >> 10) & 1ull);
    ok = ok && (a == 0ull || (unsigned)(E - 1) < 2044u);
    return a == 0ull ? 0.0
                     : fix_double((long long)(v | ((unsigned long long)(~(s ^ yb)) & (1ull << 63))));
}
__host__ __device__ __forceinline__ int fix_exponent(double y) {
    return (int)((unsigned long long)fix_bits(y) >> 52) & 0x7FF;
}

// The FP64 sweep, for the lines that cannot be fixed point.  Out of line: its
// registers stay out of the kernels' budget.
template <int NQ, typename Tab>
__host__ __device__ __attribute__((noinline)) void sweep_line_fp64_call(double *buf, int line, const Tab &tab) {
    sweep_line<NQ>(buf, line, tab);
}

// One product of a sum: acc_h += Eh Dh, acc_m += Eh Dl + El Dh.
struct FixedSum {
    long long h, m;
};
// x y + z, 32 x 32 + 64 bits.  In C the compiler loses sight of the operands' 32
// bits (an E cut by a mask is a 64-bit value to it) and multiplies 64 by 64:
// 256 multiplies a line at Nq = 8 instead of 96.
__host__ __device__ __forceinline__ long long fix_mad_wide(int x, int y, long long z) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(x), "r"(y), "l"(z));
    return r;
#else
    return (long long)x * y + z;
#endif
}
__host__ __device__ __forceinline__ void fix_mad(FixedSum &a, int Eh, int El, int Dh, int Dl) {
    a.h = fix_mad_wide(Eh, Dh, a.h);
    a.m = fix_mad_wide(Eh, Dl, a.m);
    a.m = fix_mad_wide(El, Dh, a.m);
}
__host__ __device__ __forceinline__ long long fix_value(FixedSum a) {
    return a.h + (a.m >> kFixLow);
}

// The sums S of the line's integers X[0..NQ), each given to put(n, S) as it is formed.
template <int NQ, typename FT, typename Put>
__host__ __device__ __forceinline__ void sweep_fixed(const long long *X, const FT &ft, Put put) {
    constexpr int HALF = NQ / 2;
    constexpr bool ODD = (NQ & 1) != 0;
    constexpr int C = NQ / 2;
    constexpr long long MASK = (1ll << kFixLow) - 1;
    int Eh[HALF], El[HALF], Oh[HALF], Ol[HALF];
#pragma unroll
    for (int m = 0; m < HALF; ++m) {
        const long long E = X[m] + X[NQ - 1 - m], O = X[m] - X[NQ - 1 - m];
        Eh[m] = (int)(E >> kFixLow);
        El[m] = (int)(E & MASK);
        Oh[m] = (int)(O >> kFixLow);
        Ol[m] = (int)(O & MASK);
    }
    int Ch = 0, Cl = 0;
    if constexpr (ODD) {
        Ch = (int)(X[C] >> kFixLow);
        Cl = (int)(X[C] & MASK);
    }
#pragma unroll
    for (int r = 0; r < HALF; ++r) {
        FixedSum a{0, 0}, b{0, 0};
        if constexpr (ODD) fix_mad(a, Ch, Cl, ft.Dch[r], ft.Dcl[r]);
#pragma unroll
        for (int m = 0; m < HALF; ++m) {
            fix_mad(a, Eh[m], El[m], ft.Deh[r * HALF + m], ft.Del[r * HALF + m]);
            fix_mad(b, Oh[m], Ol[m], ft.Doh[r * HALF + m], ft.Dol[r * HALF + m]);
        }
        const long long A = fix_value(a), B = fix_value(b);
        put(r, B + A);
        put(NQ - 1 - r, B - A);
    }
    if constexpr (ODD) {
        FixedSum c{0, 0};
#pragma unroll
        for (int m = 0; m < HALF; ++m) fix_mad(c, Oh[m], Ol[m], ft.Dcrh[m], ft.Dcrl[m]);
        put(C, fix_value(c));
    }
}

// Sweep line `line` of buf in place: fluxes (doubles) in, integer sums out,
// and the line's exponent returned (kFixNone: the sums are doubles).
template <int NQ, typename Tab, typename FT>
__host__ __device__ __forceinline__ int sweep_line_fixed(double *buf, int line, const Tab &tab, const FT &ft) {
    if constexpr (!fixed_point<NQ>()) {
        sweep_line<NQ>(buf, line, tab);
        return kFixNone;
    }
    long long X[NQ];
    double F[NQ];
    load_line<NQ, double>(buf, line, F);
    uint32_t top = 0, any = 0;
#pragma unroll
    for (int n = 0; n < NQ; ++n) {
        X[n] = fix_bits(F[n]);
        const uint32_t h = (uint32_t)((unsigned long long)X[n] >> 32) & 0x7FFFFFFFu;
        top = h > top ? h : top;
        any |= (uint32_t)X[n];
    }
    int e = (int)(top >> 20);
    if (e < kFixMinExp || e > kFixMaxExp) {
        if ((top | any) != 0u) {
            sweep_line_fp64_call<NQ>(buf, line, tab);
            return kFixNone;
        }
        e = kFixMinExp;   // zeros of either sign: X = 0
    }
#pragma unroll
    for (int n = 0; n < NQ; ++n) X[n] = fix_from_bits(X[n], e);
    if constexpr (line_vector<NQ, double>() > 1) {
        sweep_fixed<NQ>(X, ft, [&](int n, long long S) { F[n] = fix_double(S); });
        store_line<NQ, double>(buf, line, F);
    } else {
        sweep_fixed<NQ>(X, ft, [&](int n, long long S) { buf[slot<NQ, double>(line, n)] = fix_double(S); });
    }
    return e;
}

// -y times the sum of a point's three directions where a line is in FP64, or
// the integer multiply does not take y (rare).
static __host__ __device__ __attribute__((noinline)) double fixed_sum3_slow(double r, int er, double s,
                                                                            int es, double t, int et,
                                                                            int shift, double y) {
    const double R = er < 0 ? r : fix_to_double(fix_bits(r), er, shift);
    const double S = es < 0 ? s : fix_to_double(fix_bits(s), es, shift);
    const double T = et < 0 ? t : fix_to_double(fix_bits(t), et, shift);
    return -y * (R + S + T);
}

// v[b] = -y times the sum of a point's three directions, b < NB: at(d, b) gives
// the slot's bits and ex(d, b) the line's exponent.  One test for all of them,
// after the integer operations, so that their chains run side by side.
template <int NQ, int NB, typename At, typename Ex>
__host__ __device__ __forceinline__ void fixed_sums(double (&v)[NB], int shift, double y, At at, Ex ex) {
    if constexpr (!fixed_point<NQ>()) {
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = -y * (at(0, b) + at(1, b) + at(2, b));
        return;
    }
    const int ey = fix_exponent(y);
    bool ok = (unsigned)(ey - 1) < 2046u;   // not zero, subnormal, infinite or NaN
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int e0 = ex(0, b), e1 = ex(1, b), e2 = ex(2, b);
        ok = ok && (e0 | e1 | e2) >= 0;
        const int m = e0 > e1 ? e0 : e1, e = m > e2 ? m : e2;
        const long long R = fix_shr(fix_bits(at(0, b)), e - e0) + fix_shr(fix_bits(at(1, b)), e - e1) +
                            fix_shr(fix_bits(at(2, b)), e - e2);
        v[b] = fix_scale(R, e, shift, y, ey, ok);
    }
    if (!ok) {
#pragma unroll
        for (int b = 0; b < NB; ++b)
            v[b] = fixed_sum3_slow(at(0, b), ex(0, b), at(1, b), ex(1, b), at(2, b), ex(2, b), shift, y);
    }
}

}  // namespace numa
