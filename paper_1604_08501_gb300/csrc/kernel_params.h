// Parameters and per-point array descriptors that the volume-term kernels take
// by value: what a kernel's device code depends on besides its own source.
// (The launchers, the batch and engine structures and the handle are in
// numa_internal.h.)
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace numa {

constexpr int kFields = 5;      // rho, U1, U2, U3, Theta
constexpr int kMaxFields = 8;   // with three passive tracers

// Elements [e0, e0 + count) of a mesh whose per-point planes hold M values.
struct ElemRange {
    int64_t e0, count, M;
};

// Device-side geometry of one handle. Every per-point array has M entries,
// padded so that each starts on a 256-byte boundary.
struct DeviceGeometry {
    const double *g[9];      // metric terms g[3*d + a]
    const double *Jinv;      // 1 / J
    const double *rho_ref;   // reference density
    const double *theta_ref; // reference Theta
    const double *w;         // 1 / Theta_ref
    const double *A;         // p(Theta_ref) / Theta_ref
    const double *D;         // (N+1)^2, row-major D[i*Nq + n]
};

struct EosConstants {
    double p0, R, gamma, grav;
};

// Even-odd tables of D as (high, low) integer words for the fixed-point sweep of
// the FP64 kernels (fixed_sweep.cuh), row n times 2^s, s = shift + row_shift + 3; T: entries of De
// and Do, H: of the centre column and row (odd Nq).
constexpr int kFixBits = 60;   // line values are integers below 2^60
constexpr int kFixLow = 31;    // bits of their sums' low words
constexpr int kFixD = 61;      // the sum of a row's |D| 2^s is below 2^61
constexpr int kFixDLow = 30;   // bits of D's low words, which hold twice the value
template <int T, int H>
struct FixedTables {
    int Deh[T], Del[T], Doh[T], Dol[T], Dch[H], Dcl[H], Dcrh[H], Dcrl[H];
    int shift;            // the shift of the row with the largest sum of |D|, less 3
    unsigned long long rows;   // a row's shift beyond it, below 16: four bits each
};

// Parameters of the native kernel: EOS constants, c[k] = binom(gamma, k+1)
// (k = 0..14, the coefficients of the p' series), and the even-odd pieces of D
// for r, m < Nq/2: De = (D[r][m] + D[r][N-m])/2, Do = (D[r][m] - D[r][N-m])/2,
// Dc[r] = D[r][c] and Dcr[m] = D[c][m] (centre column and row, odd Nq).  (The
// integer tables go beside it: a batch keeps a NativeParams per instance.)
// Uniform across threads, so the kernel reads them as constant-bank operands.
struct NativeParams {
    EosConstants eos;
    double c[15];
    float ct[4];     // c[5..8] in FP32
    int tail_f32;    // their share of the series is small enough for FP32
    double De[16], Do[16], Dc[4], Dcr[4];
};

// Parameters of the native kernel for orders N = 8..15 (Nq = 9..16): the same
// quantities as NativeParams with even-odd tables up to (Nq/2)^2 = 64 entries.
struct HighParams {
    EosConstants eos;
    double c[15];
    float ct[4];     // c[5..8] in FP32
    int tail_f32;    // their share of the series is small enough for FP32
    double De[64], Do[64], Dc[8], Dcr[8];
    FixedTables<64, 8> fix;
};

// The same for the mixed-precision mode at N = 8..15: FP32 tables and the FP32
// EOS constants of MixedParams (c[k] = binom(gamma, k+1)).
struct HighParams32 {
    float De[64], Do[64], Dc[8], Dcr[8];
    float c[16];
    float K, gm1, gamma, grav;
};

// Per-point arrays of the double-float path (N = 1..7): float2 (h, l) pairs, and
// the reference state in FP64, so that rho - rho_ref and Theta - Theta_ref are
// exact FP64 differences before they are split.
struct DfGeometry {
    const float2 *g[9];      // metric terms
    const float2 *Jinv;      // 1 / J
    const double *rho_ref;   // reference density
    const double *theta_ref; // reference Theta
    const float2 *w;         // 1 / Theta_ref
    const float2 *A;         // p(Theta_ref) / Theta_ref
};

// Per-point arrays of the mixed-precision path, FP32.
struct MixedGeometry {
    const float *g[9];
    const float *Jinv;
    const float *rho_ref;
    const float *theta_ref;
};

// Parameters of the mixed-precision kernel: even-odd pieces of D (as in
// NativeParams), c[k] = binom(gamma, k+1) for k = 0..15, K = p0^(1-gamma) R^gamma
// (so p(Theta) = K Theta^gamma), gamma - 1, gamma and gravity.
struct MixedParams {
    float De[16], Do[16], Dc[4], Dcr[4];
    float c[16];
    float K, gm1, gamma, grav;
};

// Double-float value: the unevaluated sum h + l of two floats.
struct df {
    float h, l;
};

struct DfParams {
    df De[4][4];       // (D[i][m] + D[i][N-m]) / 2, i, m < Nq/2
    df Do[4][4];       // (D[i][m] - D[i][N-m]) / 2
    df Dc[4];          // D[i][c], the centre column (odd Nq), i < Nq/2
    df Dcr[4];         // D[c][m], the centre row (odd Nq), m < Nq/2
    df c1, c2, c3;     // binom(gamma, k), k = 1..3
    float ct[6];       // binom(gamma, k), k = 4..9
    df grav_df;        // gravity
    double grav, p0, R, gamma;
    double D[64];      // D, row-major D[i Nq + n], for the native fallback
};

}  // namespace numa
