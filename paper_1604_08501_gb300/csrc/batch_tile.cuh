// Per-tile device code of the batched low-storage Runge-Kutta integrator:
// one CTA of 512 threads takes `count` elements of one instance through all
// 5 * nsteps stages (see batch_lsrk.cu for the scheme and the design).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "element_sweep.cuh"
#include "eos.cuh"
#include "fixed_sweep.cuh"
#include "numa_internal.h"

namespace numa {

namespace {

constexpr int kThreads = 512;

// Shared memory of one CTA and CTAs per SM.  FP64: the fluxes (15 values per
// thread), q and dq (10 values); the D sweeps run on the integer pipes
// (fixed_sweep.cuh), so two CTAs of 64 registers share an SM and one's sweeps
// run beside the other's FP64 phases (the FP64 pipe binds, about 62 operations
// per point and stage).  Measured on 6 instances, 4.6 million points, ten steps
// (50 stages): 75.5 ms with FP64 sweeps, q and dq in registers and one CTA per SM,
// 30.2 ms so.  The tracer form keeps the base fields' q and dq in registers
// (98 KB of fluxes: one CTA per SM).  Mixed: the fluxes, q and dq (10 values) and the point's geometry
// (g and Jinv, 10 values) in shared memory, so that the kernel fits 64
// registers and two CTAs share an SM, twice the warps to hide latency.
// Flux words of one pass: 3 x NF blocks of EPP elements; the largest over the
// orders sizes the flux region (4-byte values at Nq = 8: lines of 9 slots).
// NF = 5, or 8 in the tiles' tracer forms (TR), whose tracers' q and dq also
// live in shared memory in FP64 (3 + 3 values per thread after the fluxes).
template <typename T, int NQ, int NF = kFields>
__host__ __device__ constexpr int pass_flux_words() {
    return 3 * NF * (kThreads / (NQ * NQ * NQ)) * block_words<NQ, T>();
}
template <typename T, int NF = kFields>
__host__ __device__ constexpr int tile_flux_words() {
    constexpr int w[] = {pass_flux_words<T, 2, NF>(), pass_flux_words<T, 3, NF>(),
                         pass_flux_words<T, 4, NF>(), pass_flux_words<T, 5, NF>(),
                         pass_flux_words<T, 6, NF>(), pass_flux_words<T, 7, NF>(),
                         pass_flux_words<T, 8, NF>()};
    int m = 0;
    for (int x : w) m = x > m ? x : m;
    return m;
}
constexpr int kMixedFluxWords = tile_flux_words<float>();
constexpr int kMixedSmemWords = kMixedFluxWords + (2 * 5 + 10) * kThreads;
// FP64: the exponents of the lines' fixed-point sums (fixed_sweep.cuh) follow.
template <int NF>
__host__ __device__ constexpr int tile_exponents() {   // of the lines of one pass: the largest over the orders
    int m = 0;
    for (int nq = 2; nq <= 8; ++nq) {
        const int x = 3 * NF * (kThreads / (nq * nq * nq)) * nq * nq * (1 + (nq & 1));
        m = x > m ? x : m;
    }
    return m;
}
// State words per thread in shared memory in FP64: q and dq of every field, or
// of the tracers alone in the tracer form.
template <bool TR>
__host__ __device__ constexpr int fp64_state_words() {
    return TR ? 2 * (kMaxFields - kFields) : 2 * kFields;
}
template <bool MIXED, bool TR = false>
constexpr size_t tile_smem_bytes() {
    constexpr int NF = TR ? kMaxFields : kFields;
    return MIXED ? sizeof(float) * (tile_flux_words<float, NF>() + (2 * NF + 10) * kThreads)
                 : sizeof(double) * (tile_flux_words<double, NF>() + fp64_state_words<TR>() * kThreads) +
                       sizeof(short) * tile_exponents<NF>();
}
template <bool MIXED, bool TR = false>
constexpr int tile_ctas_per_sm() {
    return MIXED || !TR ? 2 : 1;
}

// Sweep tables per Nq (index Nq; 2..8 used).  They depend only on the order:
// every handle's D is the library's GLL D.  In constant memory, every
// coefficient of a sweep is a constant-bank operand of its FMA, as in the
// single-evaluation kernels, where the tables are kernel parameters.
template <typename T>
struct SweepTables {
    T De[16], Do[16], Dc[4], Dcr[4];
};
__constant__ SweepTables<double> c_sweep64[9];
__constant__ SweepTables<float> c_sweep32[9];
__constant__ FixedTables<16, 4> c_fixed[9];

// Fills this translation unit's tables on the current device (synchronous).
inline cudaError_t upload_sweep_tables() {
    SweepTables<double> t64[9] = {};
    SweepTables<float> t32[9] = {};
    FixedTables<16, 4> tf[9] = {};
    for (int N = 1; N <= 7; ++N) {
        double D[64];
        gll_diff_matrix(N, D);
        SweepTables<double> &a = t64[N + 1];
        sweep_tables(N, D, a.De, a.Do, a.Dc, a.Dcr);
        fixed_tables(N, D, &tf[N + 1]);
        SweepTables<float> &b = t32[N + 1];
        for (int t = 0; t < 16; ++t) {
            b.De[t] = static_cast<float>(a.De[t]);
            b.Do[t] = static_cast<float>(a.Do[t]);
        }
        for (int t = 0; t < 4; ++t) {
            b.Dc[t] = static_cast<float>(a.Dc[t]);
            b.Dcr[t] = static_cast<float>(a.Dcr[t]);
        }
    }
    cudaError_t e = cudaMemcpyToSymbol(c_sweep64, t64, sizeof(t64));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_sweep32, t32, sizeof(t32));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_fixed, tf, sizeof(tf));
    return e;
}

// Stage coefficients of the scheme in the tile's arithmetic type: A[s] at
// [s], B[s] at [5 + s].  The kernels keep them in shared memory.
template <bool MIXED>
using tile_t = typename std::conditional<MIXED, float, double>::type;

template <bool MIXED>
__device__ __forceinline__ void load_stage_coefficients(const LsrkCoef &co, tile_t<MIXED> *sco) {
    if (threadIdx.x == 0) {   // constant indices: the parameter is read in place
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            sco[s] = static_cast<tile_t<MIXED>>(co.A[s]);
            sco[5 + s] = static_cast<tile_t<MIXED>>(co.B[s]);
        }
    }
}

// TR: the tracer form (instances of 5..8 fields, I.nf): flux blocks laid out
// for 8 fields, the tracers' q and dq in shared memory in both precisions.
template <int NQ, bool MIXED, bool TR = false>
__device__ void run_tile(const BatchInstance &I, int64_t e0, int64_t count,
                         const tile_t<MIXED> *sco, int nsteps, double dt, void *smem) {
    using T = tile_t<MIXED>;
    constexpr int N3 = NQ * NQ * NQ;
    constexpr int NL = NQ * NQ;
    constexpr int NF = TR ? kMaxFields : kFields;   // flux blocks per direction
    constexpr int NTR = kMaxFields - kFields;       // tracers at most
    constexpr int EPP = kThreads / N3;          // elements per pass
    constexpr int EW = block_words<NQ, T>();    // one element's (direction, field) block
    constexpr int BLK = EPP * EW;               // one (direction, field) block of sF
    constexpr int TASKS = 3 * NF * EPP * NL;    // lines per stage (TR: some blocks unused)
    constexpr bool SMEM_STATE = MIXED || !TR;   // the base fields' q and dq
    const int nf = TR ? I.nf : kFields;
    T *sF = static_cast<T *>(smem);             // [(d*NF + b)*EPP + el][slot]
    // FP64: the lines' exponents, [((d*NF + b)*EPP + el)*NL + line]
    short *sE = reinterpret_cast<short *>(sF + tile_flux_words<T, NF>() +
                                          fp64_state_words<TR>() * kThreads);
    const int l = threadIdx.x;
    const int el = l / N3, p = l % N3;
    const int i = p % NQ, j = (p / NQ) % NQ, k = p / NL;
    // this thread's flux slot of field b in direction d: f[d] + b * BLK
    int f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d] = d * NF * BLK + el * EW + dir_slot<NQ, T>(d, i, j, k);
    const int64_t M = I.M;
    T *qv = static_cast<T *>(I.q);
    const T dtt = static_cast<T>(dt);
    T grav;
    if constexpr (MIXED)
        grav = I.mp.grav;
    else
        grav = I.np.eos.grav;

    for (int64_t base = e0; base < e0 + count; base += EPP) {
        const int npass = (int)((e0 + count - base) < EPP ? (e0 + count - base) : EPP);
        const bool active = el < npass;
        const int64_t node = (base + (active ? el : 0)) * N3 + p;
        // q and the scheme's dq of this thread's point (registers in FP64,
        // shared memory in the mixed mode), and the mixed mode's per-point
        // constants, kept for all stages
        T qr[kFields], dqr[kFields];
        T *sQ = sF + tile_flux_words<T, NF>() + l;   // [b * kThreads], every field
        T *sD = sQ + NF * kThreads;                  // (FP64, TR: the tracers alone)
        T *sG = sD + NF * kThreads;                  // g (9), Jinv; mixed only
        // the tracers' q and dq (TR): shared memory in both precisions
        auto QT = [&](int t) -> T & {
            if constexpr (MIXED) return sQ[(kFields + t) * kThreads];
            else return sF[tile_flux_words<T, NF>() + t * kThreads + l];
        };
        auto DQT = [&](int t) -> T & {
            if constexpr (MIXED) return sD[(kFields + t) * kThreads];
            else return sF[tile_flux_words<T, NF>() + (NTR + t) * kThreads + l];
        };
        auto Q = [&](int b) -> T & {
            if constexpr (SMEM_STATE) return sQ[b * kThreads]; else return qr[b];
        };
        auto DQ = [&](int b) -> T & {
            if constexpr (SMEM_STATE) return sD[b * kThreads]; else return dqr[b];
        };
#pragma unroll
        for (int b = 0; b < kFields; ++b) {
            Q(b) = active ? qv[b * M + node] : T(0);
            DQ(b) = T(0);
        }
        if (!active) Q(0) = MIXED ? T(0) : T(1);   // idle threads hold a harmless state
        if constexpr (TR) {
#pragma unroll
            for (int t = 0; t < NTR; ++t) {
                QT(t) = active && kFields + t < nf ? qv[(kFields + t) * M + node] : T(0);
                DQT(t) = T(0);
            }
        }
        float th0 = 0.f, rho0 = 0.f;
        EosRef32 er{0.f, 0.f};
        if constexpr (MIXED) {
            if (active) {
                th0 = __ldg(I.mgeo.theta_ref + node);
                rho0 = __ldg(I.mgeo.rho_ref + node);
                if (th0 > 0.f) er = eos_reference_f32(th0, I.mp);
#pragma unroll
                for (int s2 = 0; s2 < 9; ++s2) sG[s2 * kThreads] = __ldg(I.mgeo.g[s2] + node);
                sG[9 * kThreads] = __ldg(I.mgeo.Jinv + node);
            }
        }

        for (int step = 0; step < nsteps; ++step) {
#pragma unroll 1
            for (int st = 0; st < 5; ++st) {
                // Phase 3 reads and phase 1 writes only the thread's own
                // point's flux slots (and its own state words), so within a
                // pass the next stage's phase 1 needs no barrier after phase 3.
                // The first stage of a pass takes one: the previous pass or
                // work item (possibly another order) gave its slots to other
                // threads.
                if (step == 0 && st == 0) __syncthreads();
                // ---- phase 1: p', fluxes ------------------------------
                if (active) {
                    T q[kFields];
#pragma unroll
                    for (int b = 0; b < kFields; ++b) q[b] = Q(b);
                    T rho, Th, pp, g[9];
                    if constexpr (MIXED) {
#pragma unroll
                        for (int s2 = 0; s2 < 9; ++s2) g[s2] = sG[s2 * kThreads];
                        rho = rho0 + q[0];
                        Th = th0 + q[4];
                        pp = pressure_perturbation_f32(q[4], th0, er, I.mp);
                    } else {
#pragma unroll
                        for (int s2 = 0; s2 < 9; ++s2) g[s2] = __ldg(I.geo.g[s2] + node);
                        rho = q[0];
                        Th = q[4];
                        pp = pressure_perturbation(Th, __ldg(I.geo.theta_ref + node),
                                                   __ldg(I.geo.w + node), __ldg(I.geo.A + node), I.np);
                    }
                    T rinv;
                    if constexpr (MIXED)
                        rinv = __frcp_rn(rho);   // the correctly rounded 1/rho, as 1.0f / rho
                    else
                        rinv = rcp_fp64(rho);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const T g1 = g[3 * d], g2 = g[3 * d + 1], g3 = g[3 * d + 2];
                        const T v = fma(g3, q[3], fma(g2, q[2], g1 * q[1]));
                        const T u = v * rinv;
                        T *F = sF + f[d];
                        F[0 * BLK] = v;
                        F[1 * BLK] = fma(q[1], u, g1 * pp);
                        F[2 * BLK] = fma(q[2], u, g2 * pp);
                        F[3 * BLK] = fma(q[3], u, g3 * pp);
                        F[4 * BLK] = Th * u;
                        if constexpr (TR) {
#pragma unroll
                            for (int t = 0; t < NTR; ++t)
                                if (kFields + t < nf) F[(kFields + t) * BLK] = QT(t) * u;   // Q u_d
                        }
                    }
                }
                __syncthreads();
                // ---- phase 2: sweeps, one line per task ------------------
#pragma unroll 1
                for (int t = l; t < TASKS; t += kThreads) {
                    const int bd = t / (EPP * NL), rem = t % (EPP * NL);
                    const int e = rem / NL, line = rem % NL;
                    if (e < npass && (!TR || bd % NF < nf)) {
                        if constexpr (MIXED)
                            sweep_line<NQ>(sF + bd * BLK + e * EW, line, c_sweep32[NQ]);
                        else
                            sweep_line_to<NQ>(sF + bd * BLK + e * EW, line, c_sweep64[NQ], c_fixed[NQ],
                                              sE + t, TASKS);
                    }
                }
                // FP64: J^-1 and rho_ref loaded before the barrier, so that
                // their latency passes while the last sweeps finish
                T jinv_g = T(0), rho_ref_g = T(0);
                if constexpr (!MIXED) {
                    if (active) {
                        jinv_g = __ldg(I.geo.Jinv + node);
                        rho_ref_g = __ldg(I.geo.rho_ref + node);
                    }
                }
                __syncthreads();
                // ---- phase 3: rhs, stage update ------------------------
                // -J^-1 times the sums of fields b0 .. of the three sweeps at the
                // thread's point
                auto sums = [&](auto &v, int b0, T jinv) {
                    constexpr int NB = sizeof(v) / sizeof(T);
                    if constexpr (MIXED) {
#pragma unroll
                        for (int b = 0; b < NB; ++b) {
                            const int o = (b0 + b) * BLK;
                            v[b] = -jinv * (sF[f[0] + o] + sF[f[1] + o] + sF[f[2] + o]);
                        }
                    } else {
                        constexpr int EB = EPP * NL;   // lines of one (direction, field)
                        const short *E = sE + b0 * EB + el * NL;
                        const FixedRow row[3] = {fixed_row<NQ>(c_fixed[NQ], NQ * k + j, i, TASKS),
                                                 fixed_row<NQ>(c_fixed[NQ], NQ * k + i, j, TASKS),
                                                 fixed_row<NQ>(c_fixed[NQ], NQ * j + i, k, TASKS)};
                        const int sh[3] = {row[0].shift, row[1].shift, row[2].shift};
                        fixed_sums<NQ>(
                            v, sh, jinv, [&](int d, int b) { return sF[f[d] + (b0 + b) * BLK]; },
                            [&](int d, int b) { return (int)E[(d * NF + b) * EB + row[d].at]; });
                    }
                };
                if (active) {
                    const T a = sco[st], bcoef = sco[5 + st];
                    T jinv, drho;   // drho: rho - rho_ref of this stage's state, before the update
                    if constexpr (MIXED) {
                        jinv = sG[9 * kThreads];
                        drho = Q(0);
                    } else {
                        jinv = jinv_g;
                        drho = Q(0) - rho_ref_g;
                    }
                    // dq and q of fields b0 .. from dt times their rhs
                    auto update = [&](auto &v, int b0) {
                        constexpr int NB = sizeof(v) / sizeof(T);
                        sums(v, b0, jinv);
#pragma unroll
                        for (int b = b0; b < b0 + NB; ++b) {
                            T rhs = v[b - b0];
                            if (b == 3) rhs = fma(-drho, grav, rhs);
                            const T d = fma(a, DQ(b), dtt * rhs);
                            DQ(b) = d;
                            Q(b) = fma(bcoef, d, Q(b));
                        }
                    };
                    // in two groups: the integer chains of all five fields side by
                    // side spill at 64 registers (FP64: 32.9 ms in one group,
                    // 29.7 in two, 30.1 in three, on the 6 instances above)
                    T v3[3], v2[2];
                    update(v3, 0);
                    update(v2, 3);
                    if constexpr (TR) {
#pragma unroll
                        for (int t = 0; t < NTR; ++t) {
                            if (kFields + t >= nf) break;
                            const int b = kFields + t;
                            T w[1];
                            sums(w, b, jinv);
                            const T d = fma(a, DQT(t), dtt * w[0]);
                            DQT(t) = d;
                            QT(t) = fma(bcoef, d, QT(t));
                        }
                    }
                }
            }
        }
        if (active) {
#pragma unroll
            for (int b = 0; b < kFields; ++b) qv[b * M + node] = Q(b);
            if constexpr (TR) {
#pragma unroll
                for (int t = 0; t < NTR; ++t)
                    if (kFields + t < nf) qv[(kFields + t) * M + node] = QT(t);
            }
        }
    }
}

// A function of its own per order (not inlined): each tile is then
// register-allocated by itself (inlined together the FP64 tiles spill).
template <int NQ, bool MIXED, bool TR>
__device__ __noinline__ void run_tile_call(const BatchInstance &I, int64_t e0, int64_t count,
                                           const tile_t<MIXED> *sco, int nsteps, double dt,
                                           void *smem) {
    run_tile<NQ, MIXED, TR>(I, e0, count, sco, nsteps, dt, smem);
}
template <int NQ, bool MIXED, bool TR>
__device__ __forceinline__ void run_tile_either_way(const BatchInstance &I, int64_t e0,
                                                    int64_t count, const tile_t<MIXED> *sco,
                                                    int nsteps, double dt, void *smem) {
    if constexpr (MIXED) run_tile<NQ, MIXED, TR>(I, e0, count, sco, nsteps, dt, smem);
    else run_tile_call<NQ, MIXED, TR>(I, e0, count, sco, nsteps, dt, smem);
}

}  // namespace

}  // namespace numa
