// Mixed-precision element volume term (NUMA_MIXED), orders N = 1..7 (N = 8..15:
// vol_mixed_high.cu, and vol_fp64_high.cu for small meshes and some forms), with or
// without passive tracers.
//
// The operation of Sec. 2, Eq. (2) (sign and flux form of the paper's r/s
// subroutines, Sec. 3) on FP32 data:
//   state   (rho', U1, U2, U3, Theta'), the perturbations rho' = rho - rho_ref and
//           Theta' = Theta - Theta_ref, so no significant bits go to the large
//           hydrostatic part;
//   geometry and reference state in FP32 (rounded once at create time);
//   fluxes, sweeps and rhs in FP32.
// p' = p(Theta) - p(Theta_ref) = p_ref ((1 + x)^gamma - 1), x = Theta'/Theta_ref,
// is evaluated from Theta' directly (binomial series for |x| <= 1/64,
// expm1(gamma log1p(x)) beyond), so it has no cancellation and FP32 suffices:
// relative error ~1e-7.  p_ref/Theta_ref = K Theta_ref^(gamma - 1) with
// K = p0^(1 - gamma) R^gamma is recomputed per point instead of being stored,
// which keeps the traffic at the algorithmic 88 bytes per point
// (5 + 9 + 1 + 2 arrays read, 5 written, 4 bytes each).  The kernel is bound by
// HBM bandwidth, and the extra arithmetic is free.
//
// Structure as in vol_fp64.cu: fluxes by point into shared memory, even-odd D
// sweeps by line in place, combination by point; one CTA of Nq^3 threads per
// element (several elements up to Nq = 4: cta_elements), four CTAs of 512 threads per SM at Nq = 8 (32 registers, 35 KB of
// shared memory each).  Thread 0 of every few CTAs (prefetch_group) prefetches
// to L2 (cp.async.bulk.prefetch.L2) the arrays of as many CTAs' elements a
// quarter of a wave of resident CTAs ahead (one CTA per SM at Nq = 8), so those
// CTAs' loads hit L2 rather than DRAM.  An odd Nq's elements are not whole
// 16-byte units: their range is rounded to the units that hold it
// (prefetch_l2_units; 3.5 million points without and with it: N = 4 63.5 and
// 53.4 us, N = 6 65.9 and 55.0 us).  Measured at N = 7 (GDOF/s): no prefetch 72.8, 1/8 of a
// wave 74.2, 1/4 74.7, 3/8 74.7, 1/2 74.2, 3/4 72.4, one wave 69.7, 3/2 55.0,
// two 48.3: a longer distance lets L2 evict the lines before their CTA
// starts.  At N = 7 the prefetch
// replaced a persistent kernel that staged each element's arrays in shared
// memory with cp.async.bulk on an mbarrier: the staging buffer limited that
// kernel to three CTAs per SM, and it ran at 0.271 against 0.254 ms here
// (0.242 ms with the line numbering of dir_slot at Nq = 8).
#include <cuda_runtime.h>

#include "bulk_copy.cuh"
#include "element_sweep.cuh"
#include "eos.cuh"
#include "numa_internal.h"

namespace numa {

namespace {

template <int NQ>
constexpr int mixed_min_ctas() {
    constexpr int n = 2048 / cta_threads<NQ>();
    return n < 1 ? 1 : (n > 32 ? 32 : n);
}

// Starts the arrays of points [off, off + n) toward L2; ODD: not whole 16-byte
// units.
template <bool ODD>
__device__ __forceinline__ void prefetch_points(const MixedGeometry &geo, const float *q, int64_t M,
                                                int nf, int64_t off, uint32_t n) {
    auto start = [&](const float *p) {
        if constexpr (ODD) prefetch_l2_units(p + off, n * 4);
        else prefetch_l2(p + off, n * 4);
    };
    for (int b = 0; b < nf; ++b) start(q + b * M);
#pragma unroll
    for (int a = 0; a < 9; ++a) start(geo.g[a]);
    start(geo.Jinv);
    start(geo.rho_ref);
    start(geo.theta_ref);
}

// Consecutive CTAs whose elements one of them prefetches: about 4 KB an array.
// One range a CTA, where an element is small, costs its first warp more than it
// saves (3.5 million points, us, one CTA's range and these groups: N = 4 53.8
// and 53.4, N = 5 52.2 and 51.5, N = 6 55.3 and 55.0; an array a lane instead
// of one lane for all was slower: N = 7 59.4 against 53.2).
template <int NQ>
__host__ __device__ constexpr int prefetch_group() {
    return NQ == 5 ? 8 : NQ == 6 || NQ == 7 ? 4 : NQ == 8 ? 1 : 2;
}

// TRACERS: nf = 5 + tracers fields at run time (tracers Q in FP32 as they are,
// flux Q u_d, no source).  Without tracers nf is 5.
template <int NQ, bool TRACERS>
__global__ void __launch_bounds__((cta_threads<NQ>()), mixed_min_ctas<NQ>())
vol_rhs_mixed_kernel(MixedGeometry geo, MixedParams P, const float *__restrict__ q,
                     float *__restrict__ rhs, int64_t M, int64_t e0, int nf_run, int64_t e_end,
                     int64_t ahead) {
    constexpr int N3 = NQ * NQ * NQ;
    constexpr int NL = NQ * NQ;
    constexpr int EPC = cta_elements<NQ>();
    constexpr int TE = element_threads<NQ>(), NT = cta_threads<NQ>();
    constexpr int EW = EPC * block_words<NQ, float>();   // one (direction, field) block
    const int nf = TRACERS ? nf_run : kFields;
    extern __shared__ __align__(16) float sFm[];   // [direction*nf + field][element][slot]

    const int l = threadIdx.x;
    const int el = l / TE, p = l % TE;
    const int i = p % NQ, j = (p / NQ) % NQ, k = p / (NQ * NQ);
    const int64_t eb = e0 + blockIdx.x * (int64_t)EPC;   // the CTA's first element
    // threads with a point: not the padding of an element, nor past the last one
    const bool active = EPC == 1 || (p < N3 && eb + el < e_end);
    const int64_t node = (eb + el) * N3 + p;
    constexpr int PG = prefetch_group<NQ>();
    if (l == 0 && blockIdx.x % PG == 0) {
        const int64_t pe = eb + ahead * EPC;
        if (pe < e_end) {
            const int n = e_end - pe < PG * EPC ? (int)(e_end - pe) : PG * EPC;
            prefetch_points<(N3 * 4) % 16 != 0>(geo, q, M, nf, pe * N3, (uint32_t)n * N3);
        }
    }

    // ---- phase 1: p', fluxes ----------------------------------------
    float rp = 0.f, Jinv = 0.f;
    if (active) {
        rp = q[node];
        const float U[3] = {q[M + node], q[2 * M + node], q[3 * M + node]};
        const float thp = q[4 * M + node];
        const float th0 = geo.theta_ref[node];
        const float rho = geo.rho_ref[node] + rp;
        const float Th = th0 + thp;
        const float pp = pressure_perturbation_f32<vote_lanes<NQ>()>(thp, th0, P);
        const float rinv = __frcp_rn(rho);   // correctly rounded, as 1.0f / rho
        // J^-1 with the other loads (loaded after phase 2 instead: 68.6 against
        // 69.5 GDOF/s at N = 7)
        Jinv = geo.Jinv[node];
        float Q[kMaxFields - kFields];
        if constexpr (TRACERS) {
#pragma unroll
            for (int t = 0; t < kMaxFields - kFields; ++t)
                Q[t] = kFields + t < nf ? q[(kFields + t) * M + node] : 0.f;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float g1 = geo.g[3 * d][node], g2 = geo.g[3 * d + 1][node],
                        g3 = geo.g[3 * d + 2][node];
            const float v = fmaf(g3, U[2], fmaf(g2, U[1], g1 * U[0]));
            const float u = v * rinv;
            float *F = sFm + d * nf * EW + el * block_words<NQ, float>() +
                       dir_slot<NQ, float>(d, i, j, k);
            F[0 * EW] = v;
            F[1 * EW] = fmaf(U[0], u, g1 * pp);
            F[2 * EW] = fmaf(U[1], u, g2 * pp);
            F[3 * EW] = fmaf(U[2], u, g3 * pp);
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
    for (int item = l; item < 3 * nf * EPC * NL; item += NT)   // a block's lines are contiguous
        sweep_line<NQ>(sFm + (item / (EPC * NL)) * EW, item % (EPC * NL), P);
    __syncthreads();
    if (!active) return;

    // ---- phase 3: combine, scale, gravity, store ----------------------
    const float *sFe = sFm + el * block_words<NQ, float>();
#pragma unroll
    for (int b = 0; b < (TRACERS ? kMaxFields : kFields); ++b) {
        if (TRACERS && b >= nf) break;
        const float R = sFe[(0 * nf + b) * EW + dir_slot<NQ, float>(0, i, j, k)] +
                        sFe[(1 * nf + b) * EW + dir_slot<NQ, float>(1, i, j, k)] +
                        sFe[(2 * nf + b) * EW + dir_slot<NQ, float>(2, i, j, k)];
        float v = -Jinv * R;
        if (b == 3) v = fmaf(-rp, P.grav, v);
        rhs[b * M + node] = v;
    }
}

template <int NQ, bool TRACERS>
cudaError_t launch_kernel(ElemRange r, int nf, const MixedGeometry &geo, const MixedParams &P,
                          const float *q, float *rhs, int num_sms, cudaStream_t s) {
    constexpr int EPC = cta_elements<NQ>(), NT = cta_threads<NQ>();
    const size_t smem = sizeof(float) * nf * 3 * EPC * block_words<NQ, float>();
    cudaError_t e = cudaFuncSetAttribute(vol_rhs_mixed_kernel<NQ, TRACERS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, vol_rhs_mixed_kernel<NQ, TRACERS>,
                                                      NT, smem);
    if (e != cudaSuccess) return e;
    const int64_t wave = (int64_t)num_sms * (per_sm > 0 ? per_sm : 1);
    const int64_t ahead = wave / 4 > 0 ? wave / 4 : 1;   // a quarter of a wave
    vol_rhs_mixed_kernel<NQ, TRACERS><<<(unsigned)((r.count + EPC - 1) / EPC), NT, smem, s>>>(
        geo, P, q, rhs, r.M, r.e0, nf, r.e0 + r.count, ahead);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t launch_nq(ElemRange r, int nf, const MixedGeometry &geo, const MixedParams &P,
                      const float *q, float *rhs, int num_sms, cudaStream_t s) {
    if (nf == kFields) return launch_kernel<NQ, false>(r, nf, geo, P, q, rhs, num_sms, s);
    return launch_kernel<NQ, true>(r, nf, geo, P, q, rhs, num_sms, s);
}

__global__ void to_f32_kernel(const double *__restrict__ src, float *__restrict__ dst, int64_t M) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
         m += (int64_t)gridDim.x * blockDim.x)
        dst[m] = __double2float_rn(src[m]);
}

}  // namespace

cudaError_t launch_to_f32(const double *src, float *dst, int64_t M, cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    to_f32_kernel<<<1216, 256, 0, s>>>(src, dst, M);
    return cudaGetLastError();
}

cudaError_t launch_vol_rhs_mixed(int N, int nf, ElemRange r, const MixedGeometry &geo,
                                 const MixedParams &P, const float *q, float *rhs, int num_sms,
                                 cudaStream_t s) {
    if (r.count <= 0) return cudaSuccess;
    if (nf < kFields || nf > kMaxFields) return cudaErrorInvalidValue;
    switch (N) {
        case 1: return launch_nq<2>(r, nf, geo, P, q, rhs, num_sms, s);
        case 2: return launch_nq<3>(r, nf, geo, P, q, rhs, num_sms, s);
        case 3: return launch_nq<4>(r, nf, geo, P, q, rhs, num_sms, s);
        case 4: return launch_nq<5>(r, nf, geo, P, q, rhs, num_sms, s);
        case 5: return launch_nq<6>(r, nf, geo, P, q, rhs, num_sms, s);
        case 6: return launch_nq<7>(r, nf, geo, P, q, rhs, num_sms, s);
        case 7: return launch_nq<8>(r, nf, geo, P, q, rhs, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace numa
