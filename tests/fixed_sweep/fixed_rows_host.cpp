// The fixed-point D sums (csrc/fixed_sweep.cuh) on the host, row by row, as the kernels
// form them: errors of a sum of three lines' sweeps, in fixed point and in FP64, against
// 113-bit arithmetic; and the integer tables.
#include <cfloat>
#include <cmath>
#include <cstring>

#include "fixed_sweep.cuh"
#include "numa_internal.h"

#if LDBL_MANT_DIG >= 113
typedef long double quad;
#else
typedef __float128 quad;
#endif

using namespace numa;

namespace {

// in: n triples of lines of NQ values; row r of a triple adds rows r, r + off1 and r + off2
// (mod NQ) of its lines.  err_fixed, err_fp64: [triple][row]; exps: [triple][3].
template <int NQ>
void run(int n, int off1, int off2, const double *in, double *err_fixed, double *err_fp64, int *exps) {
    constexpr int T = NQ > 8 ? 64 : 16, H = NQ > 8 ? 8 : 4, W = block_words<NQ, double>();
    double D[16 * 16];
    gll_diff_matrix(NQ - 1, D);
    struct {
        double De[T], Do[T], Dc[H], Dcr[H];
    } t{};
    for (int r = 0; r < NQ / 2; ++r) {
        for (int m = 0; m < NQ / 2; ++m) {
            const long double a = D[r * NQ + m], b = D[r * NQ + NQ - 1 - m];
            t.De[r * (NQ / 2) + m] = (double)((a + b) / 2);
            t.Do[r * (NQ / 2) + m] = (double)((a - b) / 2);
        }
        if (NQ & 1) {
            t.Dc[r] = D[r * NQ + NQ / 2];
            t.Dcr[r] = D[(NQ / 2) * NQ + r];
        }
    }
    FixedTables<T, H> fix;
    fixed_tables(NQ - 1, D, &fix);
    alignas(16) double a[3][W], b[3][W];
    for (int k = 0; k < n; ++k) {
        const double *x = in + (size_t)k * 3 * NQ;
        int e[3][2];
        for (int d = 0; d < 3; ++d) {
            for (int m = 0; m < NQ; ++m) a[d][slot<NQ, double>(0, m)] = b[d][slot<NQ, double>(0, m)] = x[d * NQ + m];
            e[d][0] = sweep_line_rows<NQ>(a[d], 0, t, fix, e[d][1]);
            sweep_line<NQ>(b[d], 0, t);
            exps[3 * k + d] = e[d][0];
        }
        for (int r = 0; r < NQ; ++r) {
            const int row[3] = {r, (r + off1) % NQ, (r + off2) % NQ};
            int sh[3], at[3];
            quad ref = 0;
            double s[3];
            for (int d = 0; d < 3; ++d) {
                const FixedRow f = fixed_row<NQ>(fix, 0, row[d], 1);
                sh[d] = f.shift;
                at[d] = f.at;
                s[d] = b[d][slot<NQ, double>(0, row[d])];
                for (int m = 0; m < NQ; ++m) ref += (quad)D[row[d] * NQ + m] * (quad)x[d * NQ + m];
            }
            double v[1];
            fixed_sums<NQ>(v, sh, -1.0, [&](int d, int) { return a[d][slot<NQ, double>(0, row[d])]; },
                           [&](int d, int) { return e[d][at[d]]; });
            err_fixed[k * NQ + r] = (double)((quad)v[0] - ref);
            err_fp64[k * NQ + r] = (double)((quad)(s[0] + s[1] + s[2]) - ref);
        }
    }
}

template <int NQ>
void tables(int *out) {   // Deh, Del, Doh, Dol (HALF^2 each), Dch, Dcl, Dcrh, Dcrl (HALF each), shift, row
    constexpr int T = NQ > 8 ? 64 : 16, H = NQ > 8 ? 8 : 4, S = (NQ / 2) * (NQ / 2), C = NQ / 2;
    double D[16 * 16];
    gll_diff_matrix(NQ - 1, D);
    FixedTables<T, H> f;
    fixed_tables(NQ - 1, D, &f);
    for (const int *p : {f.Deh, f.Del, f.Doh, f.Dol}) out = (int *)std::memcpy(out, p, S * sizeof(int)) + S;
    for (const int *p : {f.Dch, f.Dcl, f.Dcrh, f.Dcrl}) out = (int *)std::memcpy(out, p, C * sizeof(int)) + C;
    *out++ = f.shift;
    for (int n = 0; n < NQ; ++n) out[n] = row_shift(f, n);
}

}  // namespace

#define EACH_NQ(call)                                                                              \
    switch (nq) {                                                                                  \
        case 2: call(2); break; case 3: call(3); break; case 4: call(4); break;                    \
        case 5: call(5); break; case 6: call(6); break; case 7: call(7); break;                    \
        case 8: call(8); break; case 9: call(9); break; case 10: call(10); break;                  \
        case 11: call(11); break; case 12: call(12); break; case 13: call(13); break;              \
        case 14: call(14); break; case 15: call(15); break; case 16: call(16); break;              \
    }

extern "C" void rows_case(int nq, int n, int off1, int off2, const double *in, double *err_fixed,
                          double *err_fp64, int *exps) {
#define CALL(NQ) run<NQ>(n, off1, off2, in, err_fixed, err_fp64, exps)
    EACH_NQ(CALL)
#undef CALL
}

extern "C" void tables_case(int nq, int *out) {
#define CALL(NQ) tables<NQ>(out)
    EACH_NQ(CALL)
#undef CALL
}
