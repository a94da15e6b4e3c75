// The D sweep of one line of FP64 fluxes in 64-bit fixed point.
//
// GB300 issues 1.67 DFMA per clock and SM (measured) but about 30 multiply-adds of
// 32 x 32 + 64 bits and 60 other integer operations, and an even-odd sweep in
// FP64 (element_sweep.cuh) is 90 of the volume term's 157 FP64 operations per
// point at Nq = 8.  Here the sums run on the integer pipes, beside the FP64 pipe:
//
//  * The thread of a line takes the largest exponent field e of its Nq fluxes
//    and writes each as an integer X with F = X 2^(e - 1082), |X| < 2^60: the 53
//    significant bits of the largest flux, and 7 bits below (cut towards zero).
//  * E_m = X_m + X_{N-m} and O_m = X_m - X_{N-m} are exact, below 2^61.
//  * Each row of D is an integer row of its own scale, D[i][n] 2^s_i rounded to
//    nearest, s_i such that the row's sum of |D[i][n]| lies in [2^60, 2^61) (rows
//    i and N-i share it): the inner rows' entries are many times smaller than
//    those of the first and last row.  E is cut at bit 31 and D at bit 30 into
//    32-bit words, E = Eh 2^31 + El (0 <= El < 2^31) and D = Dh 2^30 + Dl / 2
//    (|Dl| <= 2^30, even), and
//      sum D E / 2^61 = sum Eh Dh + (sum (Eh Dl + El Dh)) / 2^31 + (sum El Dl) / 2^62.
//    The first sum is exact, the second too (below 2^63 for the tables of every
//    Nq: tests/test_fixed_sweep_rows.py) and its quotient is rounded to nearest;
//    the third, at most half a unit a product, is dropped.  Three multiply-adds
//    per product.
//  * S_i = a_i + b_i and S_{N-i} = b_i - a_i, |S| <= 2^60, replace the line's
//    fluxes; the value is S 2^(e - 1021 - s_i).  Phase 3 adds a point's three sums
//    as integers at the largest of their exponents (|sum| <= 3 2^60), multiplies
//    them by J^-1 as integers and rounds once to FP64 (fixed_sums).
//  * The centre row of odd Nq does not use the centre flux and, D being
//    centro-antisymmetric, is a sum over the differences O_m alone.  Those can be
//    far smaller than the line's largest flux (a spike at the centre; a smooth or
//    nearly uniform line), so they are shifted up to 61 bits first and the centre
//    sum has an exponent of its own.  Where fluxes beside the centre lost bits to
//    the line's scale and the differences are small (below 2^56), the row is
//    summed in FP64.  At Nq = 3, whose D is +-1/2, 1, 3/2 and 2, every sum is
//    exact, and the outer rows are shifted up in the same way.
//
//  * From Nq = 10, lines in which one or two values exceed all others 16 times
//    or more stay in FP64: inner rows hardly use such a value, and FP64 rounds
//    relative to what a row uses.
//
// Measured: vol_rhs_fp64_kernel at N = 7, 32768 elements, 4.949 -> 1.535 ms with the
// steps named in vol_fp64.cu; the FP64 batch 75.5 -> 30.2 ms.  One scale for the
// whole line and all rows, 58 bits and sums cut instead of rounded were 0 to 3 %
// faster (3.5 million points, us, then and so: N = 2 743 755, N = 4 330 334, N = 6 386
// 397, N = 7 338 338, N = 8 587 606, N = 11 543 551, N = 15 673 693; 512 elements of
// N = 4 13.9 14.4), but less exact than FP64 in the centre row of odd Nq (1e-14 to
// 1e-7 of the row's value on the lines above) and in inner rows of Nq >= 8.
//
// Error of S_i, in units of S: at most 1 from the X, 1/2 (Nq/2 pairs) and 1/4 (the
// centre column) from the integer D, as much again twice over from the dropped
// third sums, 1 from the rounding of a and b: below 1.5 (Nq/2) + 3.  A unit is
// at most 2^-58 of (the row's sum of |D[i][n]|) x (largest flux of the line), so the
// bound is 2^-54.8 of that at Nq = 8 and 2^-54.1 at Nq = 16.  That is a bound for
// a row and a line as a whole, where FP64 rounds each term relative to itself; row by
// row the root mean square error was at most the FP64 sweep's on random, smooth,
// nearly uniform, graded and nearly even lines and on lines with spikes of any size
// at the centre, an end, beside an end or at several points
// (tests/test_fixed_sweep_rows.py).
//
// Nq = 2 keeps the FP64 sweep: its D is +-1/2, so that FP64 rounds only sums and
// differences.
//
// Lines whose largest exponent field is outside [kFixMinExp, kFixMaxExp]
// (infinities, NaN, values that could overflow, lines of tiny values) take the
// FP64 sweep as well: their exponent is kFixNone and the slots hold doubles.  A line
// of zeros is a line of integer zeros.
#pragma once

#include <cstdint>
#include <cstring>

#include "element_sweep.cuh"
#include "kernel_params.h"

namespace numa {

constexpr int kFixMinExp = 200, kFixMaxExp = 1900;
constexpr int kFixNone = -1;      // exponent of a line left in FP64
constexpr int kFixMinCentre = 64; // least exponent field of a centre row summed in FP64
constexpr int kFixDominated = 10; // Nq from which lines of one or two dominant values stay in FP64:
constexpr uint32_t kFixNear = 4;  // those with no third value within this many binades of the largest

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
// mantissa with the hidden bit at bit 59, shifted down by the difference of
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

// The integer R, |R| < 2^63, times 2^(e - 1024), rounded to nearest (ties away from
// zero).  kFixMinExp and kFixMaxExp keep the result normal.
__host__ __device__ __forceinline__ double fix_to_double(long long R, int e) {
    const long long s = R >> 63;
    const unsigned long long a = (unsigned long long)((R ^ s) - s);
    const int lz = fix_clz(a);
    const unsigned long long m = a << (lz & 63);   // leading bit at 63
    // exponent field of 2^(63 - lz) 2^(e - 1024), less the hidden bit's one
    const int E = e + 61 - lz;
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

// -y R 2^(e - 1024), rounded once (to nearest, ties away from zero): the
// integer's leading 64 bits times the 53 of y (exponent field ey), a multiply
// on the integer pipes.  ok is cleared where the product is not a normal number.
__host__ __device__ __forceinline__ double fix_scale(long long R, int e, double y, int ey, bool &ok) {
    const long long yb = fix_bits(y);
    const long long s = R >> 63;
    const unsigned long long a = (unsigned long long)((R ^ s) - s);
    const int lz = fix_clz(a);
    // y's mantissa with its hidden bit at 63; the product in [2^62, 2^64)
    const unsigned long long my = ((unsigned long long)yb << 11) | (1ull << 63);
    unsigned long long p = fix_mulhi(a << (lz & 63), my);
    const int up = (long long)p < 0 ? 0 : 1;
    p <<= up;
    // exponent field of 2^(63 - lz) 2^(e - 1024) y, less the hidden bit's one
    const int E = e + 61 - lz + ey - 1023 + 1 - up;
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

// The centre row of a line in FP64 (odd Nq), out of line too.
template <int NQ, typename Tab>
__host__ __device__ __attribute__((noinline)) double centre_fp64_call(const double *buf, int line, const Tab &tab) {
    double c = 0.0;
    for (int m = 0; m < NQ / 2; ++m)
        c = fma(tab.Dcr[m], buf[slot<NQ, double>(line, m)] - buf[slot<NQ, double>(line, NQ - 1 - m)], c);
    return c;
}

// A sum of products: h = sum Eh Dh, m = sum (Eh Dl + El Dh) and half a unit of the
// quotient, which is so rounded to nearest.
struct FixedSum {
    long long h = 0, m = 1ll << (kFixLow - 1);
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

// Shift that brings integers below 2^61 in magnitude to 61 bits; mag: the "or" of
// their x ^ (x >> 63).  61 for zeros.
__host__ __device__ __forceinline__ int fix_headroom(long long mag) {
    return fix_clz((unsigned long long)mag) - 3;
}
__host__ __device__ __forceinline__ long long fix_magnitude(long long x) { return x ^ (x >> 63); }
__host__ __device__ __forceinline__ long long fix_shl(long long x, int n) {
    return (long long)((unsigned long long)x << n);
}

// The sums S of the line's integers X[0..NQ), each given to put(n, S) as it is
// formed; the centre row of odd Nq with its differences shifted up by `up`.
template <int NQ, typename FT, typename Put>
__host__ __device__ __forceinline__ void sweep_fixed(const long long *X, const FT &ft, int up, Put put) {
    constexpr int HALF = NQ / 2;
    constexpr bool ODD = (NQ & 1) != 0;
    constexpr int C = NQ / 2;
    constexpr int MASK = (int)((1u << kFixLow) - 1);
    if constexpr (ODD) {
        FixedSum c;
#pragma unroll
        for (int m = 0; m < HALF; ++m) {
            const long long O = fix_shl(X[m] - X[NQ - 1 - m], up);
            fix_mad(c, (int)(O >> kFixLow), (int)O & MASK, ft.Dcrh[m], ft.Dcrl[m]);
        }
        put(C, fix_value(c));
    }
    int Eh[HALF], El[HALF], Oh[HALF], Ol[HALF];
#pragma unroll
    for (int m = 0; m < HALF; ++m) {
        const long long E = X[m] + X[NQ - 1 - m], O = X[m] - X[NQ - 1 - m];
        Eh[m] = (int)(E >> kFixLow);
        El[m] = (int)E & MASK;
        Oh[m] = (int)(O >> kFixLow);
        Ol[m] = (int)O & MASK;
    }
    int Ch = 0, Cl = 0;
    if constexpr (ODD) {
        Ch = (int)(X[C] >> kFixLow);
        Cl = (int)X[C] & MASK;
    }
#pragma unroll
    for (int r = 0; r < HALF; ++r) {
        FixedSum a, b;
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
}

template <typename FT>
__host__ __device__ __forceinline__ int row_shift(const FT &ft, int n) {
    return (int)(ft.rows >> (4 * n)) & 15;
}

// Sweep line `line` of buf in place: fluxes (doubles) in, integer sums out, each at
// its row's scale: row n is S 2^(e - 1024 - ft.shift - row_shift(ft, n)).  The line's
// exponent e is returned (kFixNone: the sums are doubles); centre: the exponent of
// the centre row (odd Nq).  DOMINATED: lines of one or two dominant values too.
template <int NQ, bool DOMINATED = false, typename Tab, typename FT>
__host__ __device__ __forceinline__ int sweep_line_rows(double *buf, int line, const Tab &tab, const FT &ft,
                                                        int &centre) {
    constexpr bool ODD = (NQ & 1) != 0;
    constexpr int C = NQ / 2;
    centre = kFixNone;
    if constexpr (!fixed_point<NQ>()) {
        sweep_line<NQ>(buf, line, tab);
        return kFixNone;
    }
    long long X[NQ];
    double F[NQ];
    load_line<NQ, double>(buf, line, F);
    uint32_t top = 0, any = 0, low = ~0u;   // low: the smallest beside the centre
#pragma unroll
    for (int n = 0; n < NQ; ++n) {
        X[n] = fix_bits(F[n]);
        const uint32_t h = (uint32_t)((unsigned long long)X[n] >> 32) & 0x7FFFFFFFu;
        top = h > top ? h : top;
        any |= (uint32_t)X[n];
        if (ODD && n != C) low = h < low ? h : low;
    }
    int e = (int)(top >> 20);
    bool fixed = e >= kFixMinExp && e <= kFixMaxExp;
    if constexpr (!DOMINATED && NQ >= kFixDominated) {
        int near = 0;
#pragma unroll
        for (int n = 0; n < NQ; ++n)
            near += ((uint32_t)((unsigned long long)X[n] >> 32) & 0x7FFFFFFFu) + (kFixNear << 20) >= top ? 1 : 0;
        fixed = fixed && near > 2;
    }
    if (!fixed) {
        if ((top | any) != 0u) {
            sweep_line_fp64_call<NQ>(buf, line, tab);
            return kFixNone;
        }
        e = kFixMinExp;   // zeros of either sign: X = 0
        low = (uint32_t)kFixMinExp << 20;
    }
#pragma unroll
    for (int n = 0; n < NQ; ++n) X[n] = fix_from_bits(X[n], e);
    int up = 0;
    bool centre_fp64 = false;
    double c64 = 0.0;
    if constexpr (ODD) {
        long long mag = 0;
#pragma unroll
        for (int m = 0; m < C; ++m) mag |= fix_magnitude(X[m] - X[NQ - 1 - m]);
        up = fix_headroom(mag);
        centre = e - up;
        // an X lost bits where it lies more than kFixBits - 53 binades below the
        // line's largest, less than 2^-55 of differences that reach 2^56
        centre_fp64 = e - (int)(low >> 20) > kFixBits - 53 && up > 4;
        if (centre_fp64) c64 = centre_fp64_call<NQ>(buf, line, tab);
    }
    if constexpr (line_vector<NQ, double>() > 1 || NQ == 3) {
        sweep_fixed<NQ>(X, ft, up, [&](int n, long long S) { F[n] = fix_double(S); });
        if constexpr (NQ == 3) {   // exact sums: the outer rows shifted up as well
            const long long S0 = fix_bits(F[0]), S2 = fix_bits(F[2]);
            const int u = fix_headroom(fix_magnitude(S0) | fix_magnitude(S2));
            F[0] = fix_double(fix_shl(S0, u));
            F[2] = fix_double(fix_shl(S2, u));
            e -= u;
        }
        store_line<NQ, double>(buf, line, F);
    } else {
        sweep_fixed<NQ>(X, ft, up, [&](int n, long long S) { buf[slot<NQ, double>(line, n)] = fix_double(S); });
    }
    if (ODD && centre_fp64) {   // the FP64 sum's mantissa, and its exponent as the centre row's
        const long long b = fix_bits(c64);
        int ec = (int)((unsigned long long)b >> 52) & 0x7FF;
        ec = ec < kFixMinCentre ? kFixMinCentre : ec;
        buf[slot<NQ, double>(line, C)] = fix_double(fix_from_bits(b, ec));
        centre = ec + 1024 - (1022 + kFixBits) + ft.shift + row_shift(ft, C);
    }
    return e;
}

// The same with every row at the line's exponent, S 2^(e - 1024 - ft.shift): for
// host checks that add lines slot by slot.
template <int NQ, typename Tab, typename FT>
__host__ __device__ __forceinline__ int sweep_line_fixed(double *buf, int line, const Tab &tab, const FT &ft) {
    int c;
    const int e = sweep_line_rows<NQ, true>(buf, line, tab, ft, c);
    if (e == kFixNone) return e;
    const int top = (NQ & 1) && c > e ? c : e;
    for (int n = 0; n < NQ; ++n) {
        double &x = buf[slot<NQ, double>(line, n)];
        const int en = (NQ & 1) && n == NQ / 2 ? c : e;
        x = fix_double(fix_shr(fix_bits(x), top - en + row_shift(ft, n)));
    }
    return top;
}

// The sweep, its exponents to E[0] and, for the centre row of odd Nq, E[lines].
template <int NQ, typename Tab, typename FT>
__host__ __device__ __forceinline__ void sweep_line_to(double *buf, int line, const Tab &tab, const FT &ft,
                                                       short *E, int lines) {
    int c;
    E[0] = (short)sweep_line_rows<NQ>(buf, line, tab, ft, c);
    if constexpr (NQ & 1) E[lines] = (short)c;
}

// Where a point finds its line's exponent and its row's scale: `at` entries into the
// exponents of a block's lines (the centre rows' follow those of all lines, by
// `lines`), and the row's shift.
struct FixedRow {
    int at, shift;
};
template <int NQ, typename FT>
__host__ __device__ __forceinline__ FixedRow fixed_row(const FT &ft, int line, int n, int lines) {
    return FixedRow{(NQ & 1) && n == NQ / 2 ? line + lines : line, ft.shift + row_shift(ft, n)};
}
// Exponents per line in shared memory.
template <int NQ>
__host__ __device__ constexpr int line_exponents() {
    return 1 + (NQ & 1);
}

// -y times the sum of a point's three directions where a line is in FP64, or
// the integer multiply does not take y (rare); er, es, et: the exponents less the
// rows' shifts, or kFixDouble.
constexpr int kFixDouble = -(1 << 20);
static __host__ __device__ __attribute__((noinline)) double fixed_sum3_slow(double r, int er, double s,
                                                                            int es, double t, int et,
                                                                            double y) {
    const double R = er == kFixDouble ? r : fix_to_double(fix_bits(r), er);
    const double S = es == kFixDouble ? s : fix_to_double(fix_bits(s), es);
    const double T = et == kFixDouble ? t : fix_to_double(fix_bits(t), et);
    return -y * (R + S + T);
}

// v[b] = -y times the sum of a point's three directions, b < NB: at(d, b) gives
// the slot's bits, ex(d, b) the exponent of its line (or centre row) and sh[d] the
// shift of the point's row in direction d.  One test for all of them, after the
// integer operations, so that their chains run side by side.
template <int NQ, int NB, typename At, typename Ex>
__host__ __device__ __forceinline__ void fixed_sums(double (&v)[NB], const int (&sh)[3], double y, At at,
                                                    Ex ex) {
    if constexpr (!fixed_point<NQ>()) {
#pragma unroll
        for (int b = 0; b < NB; ++b) v[b] = -y * (at(0, b) + at(1, b) + at(2, b));
        return;
    }
    const int ey = fix_exponent(y);
    bool ok = (unsigned)(ey - 1) < 2046u;   // not zero, subnormal, infinite or NaN
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int x0 = ex(0, b), x1 = ex(1, b), x2 = ex(2, b);
        ok = ok && (x0 | x1 | x2) >= 0;
        const int e0 = x0 - sh[0], e1 = x1 - sh[1], e2 = x2 - sh[2];
        const int m = e0 > e1 ? e0 : e1, e = m > e2 ? m : e2;
        const long long R = fix_shr(fix_bits(at(0, b)), e - e0) + fix_shr(fix_bits(at(1, b)), e - e1) +
                            fix_shr(fix_bits(at(2, b)), e - e2);
        v[b] = fix_scale(R, e, y, ey, ok);
    }
    if (!ok) {
        auto e = [&](int d, int b) { return ex(d, b) < 0 ? kFixDouble : ex(d, b) - sh[d]; };
#pragma unroll
        for (int b = 0; b < NB; ++b)
            v[b] = fixed_sum3_slow(at(0, b), e(0, b), at(1, b), e(1, b), at(2, b), e(2, b), y);
    }
}
// One shift for every row (sweep_line_fixed).
template <int NQ, int NB, typename At, typename Ex>
__host__ __device__ __forceinline__ void fixed_sums(double (&v)[NB], int shift, double y, At at, Ex ex) {
    const int sh[3] = {shift, shift, shift};
    fixed_sums<NQ>(v, sh, y, at, ex);
}

}  // namespace numa
