// Native FP64 element volume term on sm_103a, orders N = 1..7 (N = 8..15:
// vol_fp64_high.cu), with or without passive tracers.
//
// Computes, per element and point, the pressure perturbation from the Theta
// equation of state, the contravariant fluxes of the five fields in the three
// reference directions, the three D sweeps, the Jinv scaling and the gravity
// source (Sec. 2, Eq. (2); sign and flux form of the paper's r/s subroutines,
// Sec. 3).  State, geometry, pressure, fluxes and rhs are FP64; the D sweeps
// run in 64-bit fixed point (fixed_sweep.cuh: its bound, and its error beside the
// FP64 sweep's).
//
// On GB300 the FP64 pipe (1.67 DFMA per clock and SM, 0.53 T/s) binds this
// kernel, so the design minimises FP64 instructions per point:
//  * p' = p(Theta) - p(Theta_ref) is evaluated as p_ref ((1+x)^gamma - 1) by
//    its binomial series in x = (Theta - Theta_ref)/Theta_ref (12 FP64
//    operations for |x| <= 1/64, and no cancellation); eos.cuh has the wider
//    forms.
//  * 1/rho is formed once; u_d = (g_d . U) * (1/rho).
//  * The fluxes are computed once per point into shared memory (the paper's
//    flux precompute, Sec. 3, opt. level 5).
//  * Each line of each (direction, field) is swept by one thread with the
//    even-odd split of the GLL D (D[N-i][N-n] = -D[i][n]), half the multiplies
//    of the direct sweep, on the integer pipes: no FP64 operation.  The sweeps
//    and the sums over the directions were 100 of 157 FP64 operations per point
//    at Nq = 8.  The integer work of one CTA runs beside the FP64 work of the
//    others on its SM.  Measured at N = 7, 32768 elements, with two CTAs of 512
//    threads: 4.949 ms with FP64 sweeps, 1.881 ms (59 FP64 operations' time per
//    point) in fixed point.
//  * Jinv is applied once to the sum of the three sweeps (opt. level 8), as an
//    integer multiply before the one rounding to FP64; the last terms of the
//    pressure series are FP32 and 1/rho starts from an FP32 reciprocal
//    (fp64_ops.cuh).  That leaves 47 of 59 FP64 operations per point; N = 7 needed
//    smaller CTAs as well (vol_rhs_fp64_kernel<8, TwoPoints>).  With these, fix_mad_wide
//    and the sums in two groups of fields: N = 7 1.881 -> 1.535 ms, 3.5 million
//    points of N = 3 383 -> 318 us, N = 4 397 -> 334 us, N = 5 394 -> 330 us, 512
//    elements of N = 4 22.5 us with FP64 sweeps, 14.4 us so.
//
// One CTA of Nq^3 threads per element (several elements from Nq = 6 down, so
// that a CTA has a few hundred threads: cta_elements), in three phases: fluxes by point,
// sweeps by line (in place), combination by point.
#include <cuda_runtime.h>

#include "element_sweep.cuh"
#include "eos.cuh"
#include "fixed_sweep.cuh"
#include "numa_internal.h"

namespace numa {

namespace {

// Resident CTAs per SM the register budget is sized for: 1024 threads per SM,
// at most 32 CTAs.
template <int NQ>
constexpr int min_ctas() {
    constexpr int n = 1024 / (cta_threads<NQ>());
    return n < 1 ? 1 : (n > 32 ? 32 : n);
}

// Fluxes of one point: put(d, b, F) takes F_d[b].  Called by every active lane of
// a vote group together (the form of the equation of state).
template <int NQ, bool TRACERS, typename Put>
__device__ __forceinline__ void point_fluxes(const DeviceGeometry &geo, const NativeParams &P,
                                             const double *__restrict__ q, int64_t M, int64_t node,
                                             int nf, Put put) {
    const double rho = q[node];
    const double U[3] = {q[M + node], q[2 * M + node], q[3 * M + node]};
    const double Th = q[4 * M + node];
    const double pp = pressure_perturbation<vote_lanes<NQ>()>(Th, geo.theta_ref[node], geo.w[node],
                                                              geo.A[node], P);
    const double rinv = rcp_fp64(rho);
    double Q[kMaxFields - kFields];
    if constexpr (TRACERS) {
#pragma unroll
        for (int t = 0; t < kMaxFields - kFields; ++t)
            Q[t] = kFields + t < nf ? q[(kFields + t) * M + node] : 0.0;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double g1 = geo.g[3 * d][node], g2 = geo.g[3 * d + 1][node], g3 = geo.g[3 * d + 2][node];
        const double v = fma(g3, U[2], fma(g2, U[1], g1 * U[0]));
        const double u = v * rinv;
        put(d, 0, v);
        put(d, 1, fma(U[0], u, g1 * pp));
        put(d, 2, fma(U[1], u, g2 * pp));
        put(d, 3, fma(U[2], u, g3 * pp));
        put(d, 4, Th * u);
        if constexpr (TRACERS) {
#pragma unroll
            for (int t = 0; t < kMaxFields - kFields; ++t)
                if (kFields + t < nf) put(d, kFields + t, Q[t] * u);
        }
    }
}

// Line of point (i, j, k) in direction d (the numbering of dir_slot).
template <int NQ>
__device__ __forceinline__ int dir_line(int d, int i, int j, int k) {
    return d == 0 ? NQ * k + j : d == 1 ? NQ * k + i : NQ * j + i;
}

// TRACERS: nf = 5 + tracers fields (up to 8) at run time; the tracers follow
// Theta with flux Q u_d and no source.  Without tracers nf is 5.
template <int NQ, bool TRACERS>
__global__ void __launch_bounds__((cta_threads<NQ>()), min_ctas<NQ>())
vol_rhs_fp64_kernel(DeviceGeometry geo, const __grid_constant__ NativeParams P,
                    const __grid_constant__ FixedTables<16, 4> fix, const double *__restrict__ q,
                    double *__restrict__ rhs, int64_t M, int64_t e0, int64_t e_end, int nf_run) {
    constexpr int N3 = NQ * NQ * NQ;
    constexpr int NL = NQ * NQ;               // lines per (direction, field)
    const int nf = TRACERS ? nf_run : kFields;
    constexpr int EPC = cta_elements<NQ>();
    constexpr int TE = element_threads<NQ>(), NT = cta_threads<NQ>();
    constexpr int EW = EPC * N3;              // one (direction, field) block
    constexpr int EL = EPC * NL;              // lines of a block
    extern __shared__ __align__(16) double sF[];   // [direction*nf + field][element][slot]
    short *sE = reinterpret_cast<short *>(sF + 3 * nf * EW);   // [direction*nf + field][element][line]

    const int l = threadIdx.x;
    const int el = l / TE, p = l % TE;
    const int i = p % NQ, j = (p / NQ) % NQ, k = p / (NQ * NQ);
    const int64_t e = e0 + blockIdx.x * (int64_t)EPC + el;
    // threads with a point: not the padding of an element, nor past the last one
    const bool active = EPC == 1 || (p < N3 && e < e_end);
    const int64_t node = e * N3 + p;

    // ---- phase 1: p', fluxes ----------------------------------------
    if (active) {
        int sl[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) sl[d] = d * nf * EW + el * N3 + dir_slot<NQ, double>(d, i, j, k);
        point_fluxes<NQ, TRACERS>(geo, P, q, M, node, nf,
                                  [&](int d, int b, double F) { sF[sl[d] + b * EW] = F; });
    }
    __syncthreads();

    // ---- phase 2: even-odd sweeps, one line per task, in place --------
    for (int item = l; item < 3 * nf * EL; item += NT)   // a block's lines are contiguous
        sweep_line_to<NQ>(sF + (item / EL) * EW, item % EL, P, fix, sE + item, 3 * nf * EL);
    __syncthreads();
    if (!active) return;

    // ---- phase 3: combine, scale, gravity, store ----------------------
    const double Jinv = geo.Jinv[node];
    const double drho = q[node] - geo.rho_ref[node];
    int sl[3], ln[3], sh[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const FixedRow row = fixed_row<NQ>(fix, d * nf * EL + el * NL + dir_line<NQ>(d, i, j, k),
                                           d == 0 ? i : d == 1 ? j : k, 3 * nf * EL);
        sl[d] = d * nf * EW + el * N3 + dir_slot<NQ, double>(d, i, j, k);
        ln[d] = row.at;
        sh[d] = row.shift;
    }
    auto store = [&](auto &v, int b0) {   // fields b0 ..
        constexpr int NB = sizeof(v) / sizeof(double);
        fixed_sums<NQ>(v, sh, Jinv, [&](int d, int b) { return sF[sl[d] + (b0 + b) * EW]; },
                       [&](int d, int b) { return (int)sE[ln[d] + (b0 + b) * EL]; });
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (b0 + b == 3) v[b] = fma(-drho, P.eos.grav, v[b]);
            rhs[(b0 + b) * M + node] = v[b];
        }
    };
    // two groups: five fields' integer chains side by side spill at 64 registers
    double v3[3], v2[2];
    store(v3, 0);
    store(v2, 3);
    if constexpr (TRACERS) {
#pragma unroll
        for (int b = kFields; b < kMaxFields; ++b) {
            if (b >= nf) break;
            double w[1];
            fixed_sums<NQ>(w, sh, Jinv, [&](int d, int) { return sF[sl[d] + b * EW]; },
                           [&](int d, int) { return (int)sE[ln[d] + b * EL]; });
            rhs[b * M + node] = w[0];
        }
    }
}

// N = 7 without tracers: 256 threads per element, two points each, so that four
// CTAs share an SM and more phases mix (two of 512 threads left the FP64 pipe
// idle a third of the time once the integer phases had become as long as the
// FP64 one).  Four CTAs leave 57 KB of shared memory each, 13 of an element's
// 15 flux blocks: the t fluxes of rho and Theta wait in their own outputs' place
// in rhs, which nothing else reads or writes meanwhile, until the sums of the
// momenta are done; they then take two of the momenta's blocks.  Measured, 6912
// elements: two CTAs of 512 threads 425 us, three of 256 405 us, three of 320
// 441 us (registers), this 365 us.  The operations are those of
// vol_rhs_fp64_kernel<8>, so the results are the same bit for bit; that kernel
// takes the launches of fewer than six elements per SM, whose time is that of a
// few elements one after the other (us, 512 threads and these: 125 elements 16.3
// 18.5, 280 24.6 27.3, 800 55.6 56.5, 1728 103.6 100.1, 4352 237 220).
constexpr int kEight = 8, kEightThreads = 256, kEightBlocks = 13;
constexpr size_t kEightSmem = kEightBlocks * (sizeof(double) * 512 + sizeof(short) * 64);

// Block of direction d and field b: 5 d + b for r and s; t: the momenta's 10, 11, 12.
__device__ __forceinline__ constexpr int eight_block(int d, int b) { return d < 2 ? 5 * d + b : 9 + b; }

struct TwoPoints {};   // the form's name: vol_rhs_fp64_kernel<8, TwoPoints>
template <int NQ, typename Form>
__global__ void __launch_bounds__(kEightThreads, 4)
vol_rhs_fp64_kernel(DeviceGeometry geo, const __grid_constant__ NativeParams P,
                          const __grid_constant__ FixedTables<16, 4> fix, const double *__restrict__ q, double *rhs,
                          int64_t M, int64_t e0) {
    static_assert(NQ == kEight, "two points a thread: 512 points");
    constexpr int N3 = 512, NL = 64, NT = kEightThreads;
    extern __shared__ __align__(16) double sF[];                       // [block][slot]
    short *sE = reinterpret_cast<short *>(sF + kEightBlocks * N3);     // [block][line]
    const int l = threadIdx.x;
    const int i = l % NQ, j = (l / NQ) % NQ, k0 = l / NL;   // points (i, j, k0) and (i, j, k0 + 4)
    const int64_t node0 = (e0 + blockIdx.x) * N3 + l;

    // ---- phase 1: p', fluxes ----------------------------------------
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int k = k0 + 4 * x;
        const int64_t node = node0 + x * NT;
        int sl[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) sl[d] = dir_slot<NQ, double>(d, i, j, k);
        point_fluxes<NQ, false>(geo, P, q, M, node, kFields, [&](int d, int b, double F) {
            if (d == 2 && (b == 0 || b == 4)) rhs[b * M + node] = F;
            else sF[eight_block(d, b) * N3 + sl[d]] = F;
        });
    }
    __syncthreads();
    // ---- phase 2: the sweeps of the 13 blocks, one line per task -----------
#pragma unroll 1
    for (int item = l; item < kEightBlocks * NL; item += NT)
        sweep_line_to<NQ>(sF + (item / NL) * N3, item % NL, P, fix, sE + item, 0);
    __syncthreads();
    // ---- phase 3: the momenta; the waiting fluxes into blocks 10 and 11, whose
    // slots of these points this thread alone has read
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int k = k0 + 4 * x;
        const int64_t node = node0 + x * NT;
        int sl[3], ln[3], sh[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const FixedRow row = fixed_row<NQ>(fix, dir_line<NQ>(d, i, j, k), d == 0 ? i : d == 1 ? j : k, 0);
            sl[d] = dir_slot<NQ, double>(d, i, j, k);
            ln[d] = row.at;
            sh[d] = row.shift;
        }
        const double f0 = rhs[node], f4 = rhs[4 * M + node];
        const double drho = q[node] - geo.rho_ref[node];
        double v[3];
        fixed_sums<NQ>(v, sh, geo.Jinv[node],
                       [&](int d, int b) { return sF[eight_block(d, b + 1) * N3 + sl[d]]; },
                       [&](int d, int b) { return (int)sE[eight_block(d, b + 1) * NL + ln[d]]; });
        rhs[M + node] = v[0];
        rhs[2 * M + node] = v[1];
        rhs[3 * M + node] = fma(-drho, P.eos.grav, v[2]);
        sF[10 * N3 + sl[2]] = f0;
        sF[11 * N3 + sl[2]] = f4;
    }
    __syncthreads();
    if (l < 2 * NL)
        sweep_line_to<NQ>(sF + (10 + l / NL) * N3, l % NL, P, fix, sE + 10 * NL + l, 0);
    __syncthreads();
    // ---- rho and Theta
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int k = k0 + 4 * x;
        const int64_t node = node0 + x * NT;
        int sl[3], ln[3], sh[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const FixedRow row = fixed_row<NQ>(fix, dir_line<NQ>(d, i, j, k), d == 0 ? i : d == 1 ? j : k, 0);
            sl[d] = dir_slot<NQ, double>(d, i, j, k);
            ln[d] = row.at;
            sh[d] = row.shift;
        }
        double v[2];
        fixed_sums<NQ>(v, sh, geo.Jinv[node],
                       [&](int d, int b) { return sF[(d < 2 ? 5 * d + 4 * b : 10 + b) * N3 + sl[d]]; },
                       [&](int d, int b) { return (int)sE[(d < 2 ? 5 * d + 4 * b : 10 + b) * NL + ln[d]]; });
        rhs[node] = v[0];
        rhs[4 * M + node] = v[1];
    }
}

template <int NQ, bool TRACERS>
cudaError_t launch_kernel(ElemRange r, int nf, const DeviceGeometry &geo, const NativeParams &P,
                          const FixedTables<16, 4> &fix, const double *q, double *rhs, cudaStream_t s) {
    constexpr int EPC = cta_elements<NQ>(), NT = cta_threads<NQ>();
    const size_t smem =
        (sizeof(double) * NQ + sizeof(short) * line_exponents<NQ>()) * EPC * NQ * NQ * nf * 3;
    // The opt-in above 48 KB is per device; setting it on every launch keeps
    // multi-device processes correct and costs about a microsecond.
    cudaError_t e = cudaFuncSetAttribute(vol_rhs_fp64_kernel<NQ, TRACERS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    vol_rhs_fp64_kernel<NQ, TRACERS><<<(unsigned)((r.count + EPC - 1) / EPC), NT, smem, s>>>(
        geo, P, fix, q, rhs, r.M, r.e0, r.e0 + r.count, nf);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t launch_nq(ElemRange r, int nf, const DeviceGeometry &geo, const NativeParams &P,
                      const FixedTables<16, 4> &fix, const double *q, double *rhs, int num_sms,
                      cudaStream_t s) {
    if (nf == kFields) {
        if constexpr (NQ == kEight) {
            if (r.count >= 6 * (int64_t)num_sms) {
                const cudaError_t e = cudaFuncSetAttribute(vol_rhs_fp64_kernel<kEight, TwoPoints>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)kEightSmem);
                if (e != cudaSuccess) return e;
                vol_rhs_fp64_kernel<kEight, TwoPoints><<<(unsigned)r.count, kEightThreads, kEightSmem, s>>>(
                    geo, P, fix, q, rhs, r.M, r.e0);
                return cudaGetLastError();
            }
        }
        return launch_kernel<NQ, false>(r, nf, geo, P, fix, q, rhs, s);
    }
    return launch_kernel<NQ, true>(r, nf, geo, P, fix, q, rhs, s);
}

// w = 1/Theta_ref and A = p(Theta_ref)/Theta_ref, in place of a copy of Theta_ref.
__global__ void reference_eos_kernel(const double *__restrict__ theta_ref, double *__restrict__ w,
                                     double *__restrict__ A, int64_t M, EosConstants c) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
         m += (int64_t)gridDim.x * blockDim.x) {
        const double th = theta_ref[m];
        w[m] = 1.0 / th;
        A[m] = eos_pressure(th, c) / th;
    }
}

}  // namespace

cudaError_t launch_reference_eos(const double *theta_ref, double *w, double *A, int64_t M,
                                 EosConstants c, cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    reference_eos_kernel<<<1216, 256, 0, s>>>(theta_ref, w, A, M, c);
    return cudaGetLastError();
}

cudaError_t launch_vol_rhs_fp64(int N, int nf, ElemRange r, const DeviceGeometry &geo,
                                const NativeParams &P, const FixedTables<16, 4> &fix,
                                const double *q, double *rhs, int num_sms, cudaStream_t s) {
    if (r.count <= 0) return cudaSuccess;
    if (nf < kFields || nf > kMaxFields) return cudaErrorInvalidValue;
    switch (N) {
        case 1: return launch_nq<2>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 2: return launch_nq<3>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 3: return launch_nq<4>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 4: return launch_nq<5>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 5: return launch_nq<6>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 6: return launch_nq<7>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        case 7: return launch_nq<8>(r, nf, geo, P, fix, q, rhs, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace numa
