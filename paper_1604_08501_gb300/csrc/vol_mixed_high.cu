// Mixed-precision element volume term (NUMA_MIXED) for orders N = 8..15
// (Nq = 9..16), with or without passive tracers.
//
// The operation and the FP32 arithmetic of vol_mixed.cu (Sec. 2, Eq. (2); sign
// and flux form of the paper's r/s subroutines, Sec. 3), in the order of the
// paper's own kernels: one thread owns an (i, j) column of the element and
// walks the k-planes (Sec. 3), two at a time.
//  * The r and s derivatives of a plane need that plane alone: its r and s
//    fluxes go to shared memory (2 planes x 2 directions x fields x Nq lines of
//    an odd number of slots), the lines are swept in place by the even-odd
//    split and each thread keeps the sum of its point's two sweeps.
//  * The t derivative runs along the thread's own column: its fluxes wait in
//    the thread's lane of tensor memory and are swept in registers after the
//    last plane, with no shared memory and no barrier.
// A CTA so holds 104 KB at Nq = 16 (five fields) instead of an element's fifteen
// flux arrays (two CTAs of 256 threads per SM instead of one of 1024), and one
// CTA's loads run beside the other's sweeps.  The next planes' loads are issued
// before the sweeps of the current ones, and the element one wave of resident
// CTAs ahead is prefetched to L2 (even Nq: whole 16-byte units).
#include <cuda_runtime.h>

#include "bulk_copy.cuh"
#include "element_sweep.cuh"
#include "eos.cuh"
#include "numa_internal.h"
#include "tcgen05.cuh"

namespace numa {

namespace {

// NF = 5 (five fields) or 8 (six to eight: tracers).
template <int NQ, int NF>
struct Plane {
    static constexpr int NL = NQ * NQ;                    // columns
    static constexpr int N3 = NQ * NL;
    static constexpr int NT = (NL + 31) / 32 * 32;        // threads: whole warps
    static constexpr int LS = NQ | 1;                     // slots of a line
    static constexpr int FLUX = 2 * 2 * NF * NQ * LS;     // words: [plane][r, s][field][line][slot]
    // Columns of tensor memory: NF Nq fluxes a lane, the warps of one lane
    // quarter side by side, a power of two.
    static constexpr int WCOLS = NF * NQ;
    static constexpr int NEED = (NT / 32 + 3) / 4 * WCOLS;
    static constexpr int COLS = NEED <= 64 ? 64 : NEED <= 128 ? 128 : NEED <= 256 ? 256 : 512;
    static constexpr int TM_CTAS = 512 / COLS < 6 ? 512 / COLS : 6;
    // The sums of the r and s sweeps wait in shared memory, or, where that would
    // leave an SM fewer CTAs than tensor memory does, in the thread's places of
    // rhs, which nothing else touches before its results.
    static constexpr bool X_SMEM =
        TM_CTAS * (sizeof(float) * (FLUX + NF * N3) + 1024) <= 227 * 1024;
    static constexpr size_t USED = sizeof(float) * (FLUX + (X_SMEM ? NF * N3 : 0));
    // CTAs per SM: what tensor memory, shared memory and 96 registers allow.
    static constexpr int BY_SMEM = 227 * 1024 / (USED + 1024);
    static constexpr int BY_REGS = 65536 / (NT * 96);
    static constexpr int BY_MEM = TM_CTAS < BY_SMEM ? TM_CTAS : BY_SMEM;
    static constexpr int CTAS = BY_MEM < BY_REGS ? BY_MEM : BY_REGS;
    // at least a share of shared memory that keeps more than 512 / COLS CTAs off an SM
    static constexpr size_t FLOOR = 228 * 1024 / (512 / COLS + 1) + 1024;
    static constexpr size_t SMEM = USED > FLOOR ? USED : FLOOR;
    static_assert(CTAS >= 1 && CTAS * (SMEM + 1024) <= 228 * 1024, "shared memory of the CTAs of one SM");
};

// Forms that the whole-element kernel (vol_fp64_high.cu, T = float) runs faster.
// Measured at 3.5 million points, us, whole element and planes: five fields
// N = 8 102 93, 9 111 88, 10 165 94, 11 100 92, 12 119 114, 13 149 112, 14 143 101,
// 15 103 110; three tracers 8 209 156, 9 219 135, 10 167 139, 11 130 167, 12 208
// 166, 13 164 183, 14 165 150, 15 172 142.  (At Nq = 12 and 14 with tracers a
// CTA of 160 or 224 threads takes half of tensor memory, and 10 or 14 warps an
// SM do not hide its loads; at Nq = 16 with five fields the element's 32 warps,
// with no thread idle in the sweeps, are as good.)
template <int NQ, int NF>
constexpr bool element_kernel() {
    return NF == kFields ? NQ == 16 : NQ == 12 || NQ == 14;
}

// State and geometry of one point (the FP32 perturbation form).
template <int NF>
struct PointLoads {
    float q[NF], g[9], rho_ref, theta_ref;
};

struct Planes {};   // the form's name: vol_rhs_high_kernel<Nq, float, NF, Planes>
template <int NQ, typename T, int NF, typename Form>
__global__ void __launch_bounds__((Plane<NQ, NF>::NT), (Plane<NQ, NF>::CTAS))
vol_rhs_high_kernel(MixedGeometry geo, HighParams32 P, const float *__restrict__ q, float *rhs,
                    int64_t M, int64_t e0, int nf, int64_t e_end, int64_t ahead) {
    using S = Plane<NQ, NF>;
    constexpr int NL = S::NL, N3 = S::N3, NT = S::NT, LS = S::LS, HALF = NQ / 2;
    constexpr bool ODD = (NQ & 1) != 0;
    extern __shared__ __align__(16) float sF[];   // fluxes of two planes; r + s sums
    float *sX = sF + S::FLUX;                     // [field][k][column]
    __shared__ uint32_t s_tmem;
    const int c = threadIdx.x;
    const bool active = NT == NL || c < NL;
    const int i = c % NQ, j = c / NQ;
    const int64_t node0 = (e0 + blockIdx.x) * N3 + c;   // point (i, j, 0); + k NL
    if (NF == kFields) nf = kFields;

    if (c < 32) tc::tmem_alloc(&s_tmem, S::COLS);
    auto prefetch = [&](int64_t d) {   // element e0 + blockIdx.x + d toward L2 (even Nq)
        if constexpr ((N3 * 4) % 16 == 0) {
            const int64_t off = (e0 + blockIdx.x + d) * N3;
            constexpr uint32_t B = N3 * 4;
            for (int b = 0; b < nf; ++b) prefetch_l2(q + b * M + off, B);
#pragma unroll
            for (int a = 0; a < 9; ++a) prefetch_l2(geo.g[a] + off, B);
            prefetch_l2(geo.Jinv + off, B);
            prefetch_l2(geo.rho_ref + off, B);
            prefetch_l2(geo.theta_ref + off, B);
        }
    };
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const int w = c >> 5;
    const uint32_t park = s_tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * S::WCOLS);

    PointLoads<NF> pt[2];
    auto load = [&](int k0) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (!active || k0 + p >= NQ) continue;
            const int64_t node = node0 + (k0 + p) * NL;
#pragma unroll
            for (int b = 0; b < NF; ++b)
                if (b < nf) pt[p].q[b] = q[b * M + node];
#pragma unroll
            for (int a = 0; a < 9; ++a) pt[p].g[a] = geo.g[a][node];
            pt[p].rho_ref = geo.rho_ref[node];
            pt[p].theta_ref = geo.theta_ref[node];
        }
    };
    load(0);

    // slot of this thread's point in the r and s lines of field 0, plane 0
    const int sr = j * LS + i, ss = (NF * NQ + i) * LS + j;
    constexpr int FB = NQ * LS, PB = 2 * NF * FB;   // a field's lines; a plane's
#pragma unroll 1
    for (int k0 = 0; k0 < NQ; k0 += 2) {
        // ---- fluxes of planes k0 and k0 + 1 -----------------------------
        float Ft[2][NF];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (active && k0 + p < NQ) {
                const PointLoads<NF> &x = pt[p];
                const float U[3] = {x.q[1], x.q[2], x.q[3]};
                const float Th = x.theta_ref + x.q[4];
                const float pp = pressure_perturbation_f32<1>(x.q[4], x.theta_ref, P);
                const float rinv = __frcp_rn(x.rho_ref + x.q[0]);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const float v = fmaf(x.g[3 * d + 2], U[2], fmaf(x.g[3 * d + 1], U[1], x.g[3 * d] * U[0]));
                    const float u = v * rinv;
#pragma unroll
                    for (int b = 0; b < NF; ++b) {
                        if (b >= nf) break;
                        const float F = b == 0   ? v
                                        : b < 4  ? fmaf(U[b > 0 && b < 4 ? b - 1 : 0], u,
                                                        x.g[3 * d + (b > 0 && b < 4 ? b - 1 : 0)] * pp)
                                        : b == 4 ? Th * u
                                                 : x.q[b] * u;
                        if (d == 2) Ft[p][b] = F;
                        else sF[(d == 0 ? sr : ss) + p * PB + b * FB] = F;
                    }
                }
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {   // every lane: the stores are warp-wide
            if (k0 + p >= NQ) break;
#pragma unroll
            for (int b = 0; b < NF; ++b) {
                if (b >= nf) break;
                tc::tmem_st1(park + b * NQ + k0 + p, __float_as_uint(active ? Ft[p][b] : 0.f));
            }
        }
        if (k0 + 2 < NQ) load(k0 + 2);   // their latency passes under the sweeps
        __syncthreads();
        if (k0 == 0 && c == 0 && ahead > 0 && e0 + blockIdx.x + ahead < e_end) prefetch(ahead);
        // ---- the r and s sweeps of the planes' lines ---------------------
        const int lines = (k0 + 1 < NQ ? 2 : 1) * 2 * NF * NQ;
#pragma unroll 1
        for (int L = c; L < lines; L += NT)
            if (NF == kFields || (L / NQ) % NF < nf) sweep_line<NQ>(sF, L, P);
        __syncthreads();
        // ---- their sums at this thread's points.  (The next planes' fluxes
        // overwrite only slots that this thread has read: no barrier.)
        if (active) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (k0 + p >= NQ) break;
#pragma unroll
                for (int b = 0; b < NF; ++b) {
                    if (b >= nf) break;
                    const float X = sF[sr + p * PB + b * FB] + sF[ss + p * PB + b * FB];
                    if constexpr (S::X_SMEM) sX[(b * NQ + k0 + p) * NL + c] = X;
                    else rhs[b * M + node0 + (k0 + p) * NL] = X;
                }
            }
        }
    }
    // ---- the t sweep of each field along the column, and the rhs -----------
    tc::tmem_st_wait();
    float jinv[NQ];
    if (active) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) jinv[k] = geo.Jinv[node0 + k * NL];
    }
#pragma unroll 1
    for (int b = 0; b < nf; ++b) {
        float X[NQ];
        if (active) {
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                if constexpr (S::X_SMEM) X[k] = sX[(b * NQ + k) * NL + c];
                else X[k] = rhs[b * M + node0 + k * NL];
            }
        }
        uint32_t f[16];
        if constexpr (NQ == 16) {
            tc::tmem_ld16(park + b * NQ, f);
            tc::tmem_ld_wait16(f);
        } else {
            uint32_t lo[8];
            tc::tmem_ld8(park + b * NQ, lo);
#pragma unroll
            for (int n = 8; n < NQ; ++n) f[n] = tc::tmem_ld1(park + b * NQ + n);
            tc::tmem_ld_wait(lo);
#pragma unroll
            for (int n = 0; n < NQ; ++n) f[n] = n < 8 ? lo[n] : tc::after_wait(f[n]);
        }
        if (active) {
            float rp[NQ];
            if (b == 3) {
#pragma unroll
                for (int k = 0; k < NQ; ++k) rp[k] = q[node0 + k * NL];
            }
            auto out = [&](int k, float T) {
                float v = -jinv[k] * (X[k] + T);
                if (b == 3) v = fmaf(-rp[k], P.grav, v);
                rhs[b * M + node0 + k * NL] = v;
            };
            float E[HALF], O[HALF];
#pragma unroll
            for (int m = 0; m < HALF; ++m) {
                const float x = __uint_as_float(f[m]), y = __uint_as_float(f[NQ - 1 - m]);
                E[m] = x + y;
                O[m] = x - y;
            }
#pragma unroll
            for (int r = 0; r < HALF; ++r) {
                float a = ODD ? P.Dc[r] * __uint_as_float(f[HALF]) : 0.f, o = 0.f;
#pragma unroll
                for (int m = 0; m < HALF; ++m) {
                    a = fmaf(P.De[r * HALF + m], E[m], a);
                    o = fmaf(P.Do[r * HALF + m], O[m], o);
                }
                out(r, o + a);
                out(NQ - 1 - r, o - a);
            }
            if constexpr (ODD) {
                float s = 0.f;
#pragma unroll
                for (int m = 0; m < HALF; ++m) s = fmaf(P.Dcr[m], O[m], s);
                out(HALF, s);
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (c < 32) {
        tc::fence_after_sync();
        tc::tmem_dealloc(s_tmem, S::COLS);
    }
}

template <int NQ, int NF>
cudaError_t launch_plane(ElemRange r, int nf, const MixedGeometry &geo, const HighParams32 &P,
                         const float *q, float *rhs, int num_sms, cudaStream_t s) {
    using S = Plane<NQ, NF>;
    const cudaError_t e = cudaFuncSetAttribute(vol_rhs_high_kernel<NQ, float, NF, Planes>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t ahead = (int64_t)num_sms * S::CTAS;   // one wave
    vol_rhs_high_kernel<NQ, float, NF, Planes><<<(unsigned)r.count, S::NT, S::SMEM, s>>>(
        geo, P, q, rhs, r.M, r.e0, nf, r.e0 + r.count, ahead);
    return cudaGetLastError();
}

// Meshes below two elements per SM take the whole-element kernel: walking the
// planes with one thread per column, a lone element takes longer (us, whole
// element and planes: 4 elements of N = 8 9.1 and 10.6, N = 14 14.5 and 20.5; 150
// elements of N = 8 9.5 and 12.4, N = 14 24.0 and 26.2; 504 elements of N = 8 18.1
// and 17.4, N = 14 81.9 and 57.4).  The line is drawn by the mesh, not by the
// launch; both kernels give an element the same bits
// (tests/test_gpu_high_mesh_size.py).
template <int NQ>
cudaError_t launch_nq(ElemRange r, int nf, const MixedGeometry &geo, const HighParams32 &P,
                      const float *q, float *rhs, int num_sms, cudaStream_t s) {
    if (r.M / (NQ * NQ * NQ) >= 2 * (int64_t)num_sms) {
        if (nf == kFields) {
            if constexpr (!element_kernel<NQ, kFields>())
                return launch_plane<NQ, kFields>(r, nf, geo, P, q, rhs, num_sms, s);
        } else {
            if constexpr (!element_kernel<NQ, kMaxFields>())
                return launch_plane<NQ, kMaxFields>(r, nf, geo, P, q, rhs, num_sms, s);
        }
    }
    return launch_vol_rhs_mixed_element(NQ - 1, nf, r, geo, P, q, rhs, num_sms, s);
}

}  // namespace

cudaError_t launch_vol_rhs_mixed_high(int N, int nf, ElemRange r, const MixedGeometry &geo,
                                      const HighParams32 &P, const float *q, float *rhs,
                                      int num_sms, cudaStream_t s) {
    if (r.count <= 0) return cudaSuccess;
    if (nf < kFields || nf > kMaxFields) return cudaErrorInvalidValue;
    switch (N) {
        case 8: return launch_nq<9>(r, nf, geo, P, q, rhs, num_sms, s);
        case 9: return launch_nq<10>(r, nf, geo, P, q, rhs, num_sms, s);
        case 10: return launch_nq<11>(r, nf, geo, P, q, rhs, num_sms, s);
        case 11: return launch_nq<12>(r, nf, geo, P, q, rhs, num_sms, s);
        case 12: return launch_nq<13>(r, nf, geo, P, q, rhs, num_sms, s);
        case 13: return launch_nq<14>(r, nf, geo, P, q, rhs, num_sms, s);
        case 14: return launch_nq<15>(r, nf, geo, P, q, rhs, num_sms, s);
        case 15: return launch_nq<16>(r, nf, geo, P, q, rhs, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace numa
