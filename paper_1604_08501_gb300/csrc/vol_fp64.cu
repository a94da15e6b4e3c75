// Native FP64 element volume term on sm_103a, orders N = 1..7 (N = 8..15:
// vol_fp64_high.cu), with or without passive tracers.
//
// Computes, per element and point, the pressure perturbation from the Theta
// equation of state, the contravariant fluxes of the five fields in the three
// reference directions, the three D sweeps, the Jinv scaling and the gravity
// source (Sec. 2, Eq. (2); sign and flux form of the paper's r/s subroutines,
// Sec. 3).  State, geometry, pressure, fluxes and rhs are FP64; the D sweeps
// run in 64-bit fixed point (fixed_sweep.cuh), whose error is below the FP64
// sweeps'.
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
//    at Nq = 8.  One thread's integers take 64 registers, as two CTAs of 512
//    threads allow, and the integer work of one CTA runs beside the FP64 work
//    of the other.  Measured at N = 7, 32768 elements: 4.949 ms with FP64
//    sweeps, 1.881 ms (59 FP64 operations' time per point) in fixed point;
//    N = 4, 512 elements, a call among others: 22.5 and 14.3 us.
//  * Jinv is applied once to the sum of the three sweeps (opt. level 8).
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

// TRACERS: nf = 5 + tracers fields (up to 8) at run time; the tracers follow
// Theta with flux Q u_d and no source.  Without tracers nf is 5.
template <int NQ, bool TRACERS>
__global__ void __launch_bounds__((cta_threads<NQ>()), min_ctas<NQ>())
vol_rhs_fp64_kernel(DeviceGeometry geo, const __grid_constant__ NativeParams P,
                    FixedTables<16, 4> fix, const double *__restrict__ q, double *__restrict__ rhs, int64_t M, int64_t e0,
                    int64_t e_end, int nf_run) {
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
    double rho = 1.0;
    if (active) {
        rho = q[node];
        const double U[3] = {q[M + node], q[2 * M + node], q[3 * M + node]};
        const double Th = q[4 * M + node];
        const double pp = pressure_perturbation<vote_lanes<NQ>()>(Th, geo.theta_ref[node], geo.w[node],
                                                                  geo.A[node], P);
        const double rinv = __drcp_rn(rho);
        double Q[kMaxFields - kFields];
        if constexpr (TRACERS) {
#pragma unroll
            for (int t = 0; t < kMaxFields - kFields; ++t)
                Q[t] = kFields + t < nf ? q[(kFields + t) * M + node] : 0.0;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double g1 = geo.g[3 * d][node], g2 = geo.g[3 * d + 1][node],
                         g3 = geo.g[3 * d + 2][node];
            const double v = fma(g3, U[2], fma(g2, U[1], g1 * U[0]));
            const double u = v * rinv;
            double *F = sF + d * nf * EW + el * N3 + dir_slot<NQ, double>(d, i, j, k);
            F[0 * EW] = v;
            F[1 * EW] = fma(U[0], u, g1 * pp);
            F[2 * EW] = fma(U[1], u, g2 * pp);
            F[3 * EW] = fma(U[2], u, g3 * pp);
            F[4 * EW] = Th * u;
            if constexpr (TRACERS) {
#pragma unroll
                for (int t = 0; t < kMaxFields - kFields; ++t)
                    if (kFields + t < nf) F[(kFields + t) * EW] = Q[t] * u;
            }
        }
    }
    __syncthreads();

    // ---- phase 2: even-odd sweeps, one line per task, in place --------
    for (int item = l; item < 3 * nf * EL; item += NT)   // a block's lines are contiguous
        sE[item] = (short)sweep_line_fixed<NQ>(sF + (item / EL) * EW, item % EL, P, fix);
    __syncthreads();
    if (!active) return;

    // ---- phase 3: combine, scale, gravity, store ----------------------
    const double Jinv = geo.Jinv[node];
    const double drho = rho - geo.rho_ref[node];
    const double *sFe = sF + el * N3;
    const short *sEe = sE + el * NL;
#pragma unroll
    for (int b = 0; b < (TRACERS ? kMaxFields : kFields); ++b) {
        if (TRACERS && b >= nf) break;
        const double R = fixed_sum3<NQ>(sFe[(0 * nf + b) * EW + dir_slot<NQ, double>(0, i, j, k)],
                                    sEe[(0 * nf + b) * EL + NQ * k + j],
                                    sFe[(1 * nf + b) * EW + dir_slot<NQ, double>(1, i, j, k)],
                                    sEe[(1 * nf + b) * EL + NQ * k + i],
                                    sFe[(2 * nf + b) * EW + dir_slot<NQ, double>(2, i, j, k)],
                                    sEe[(2 * nf + b) * EL + NQ * j + i], fix.shift);
        double v = -Jinv * R;
        if (b == 3) v = fma(-drho, P.eos.grav, v);
        rhs[b * M + node] = v;
    }
}

template <int NQ, bool TRACERS>
cudaError_t launch_kernel(ElemRange r, int nf, const DeviceGeometry &geo, const NativeParams &P,
                          const FixedTables<16, 4> &fix, const double *q, double *rhs, cudaStream_t s) {
    constexpr int EPC = cta_elements<NQ>(), NT = cta_threads<NQ>();
    const size_t smem = (sizeof(double) * NQ + sizeof(short)) * EPC * NQ * NQ * nf * 3;
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
                      const FixedTables<16, 4> &fix, const double *q, double *rhs, cudaStream_t s) {
    if (nf == kFields) return launch_kernel<NQ, false>(r, nf, geo, P, fix, q, rhs, s);
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
                                const double *q, double *rhs, cudaStream_t s) {
    if (r.count <= 0) return cudaSuccess;
    if (nf < kFields || nf > kMaxFields) return cudaErrorInvalidValue;
    switch (N) {
        case 1: return launch_nq<2>(r, nf, geo, P, fix, q, rhs, s);
        case 2: return launch_nq<3>(r, nf, geo, P, fix, q, rhs, s);
        case 3: return launch_nq<4>(r, nf, geo, P, fix, q, rhs, s);
        case 4: return launch_nq<5>(r, nf, geo, P, fix, q, rhs, s);
        case 5: return launch_nq<6>(r, nf, geo, P, fix, q, rhs, s);
        case 6: return launch_nq<7>(r, nf, geo, P, fix, q, rhs, s);
        case 7: return launch_nq<8>(r, nf, geo, P, fix, q, rhs, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace numa
