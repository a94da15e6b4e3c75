// The fixed-point D sweep (csrc/fixed_sweep.cuh) on the host, beside the FP64 sweep
// and a long-double one: sweep_case() takes the lines of a block of Nq^2 lines, sums
// a "point's" three directions over line triples, and returns both results.
#include <cmath>
#include <vector>

#include "fixed_sweep.cuh"
#include "numa_internal.h"

using namespace numa;

namespace {

template <int NQ, int T, int H>
struct Tables {
    double De[T], Do[T], Dc[H], Dcr[H];
    FixedTables<T, H> fix;
};

// in: 3 blocks of NQ^2 lines of NQ values (a line's values side by side); fixed,
// fp64, ref: the sums of the three blocks' sweeps, slot for slot; exps: the lines' exponents.
template <int NQ>
void run(const double *in, double *fixed, double *fp64, double *ref, int *exps) {
    constexpr int NL = NQ * NQ, W = block_words<NQ, double>(), T = NQ > 8 ? 64 : 16, H = NQ > 8 ? 8 : 4;
    double D[16 * 16];
    gll_diff_matrix(NQ - 1, D);
    Tables<NQ, T, H> t{};
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
    fixed_tables(NQ - 1, D, &t.fix);
    std::vector<double> a(3 * W), b(3 * W);
    for (int d = 0; d < 3; ++d)
        for (int line = 0; line < NL; ++line) {
            for (int n = 0; n < NQ; ++n)
                a[d * W + slot<NQ, double>(line, n)] = b[d * W + slot<NQ, double>(line, n)] =
                    in[(d * NL + line) * NQ + n];
            exps[d * NL + line] = sweep_line_fixed<NQ>(a.data() + d * W, line, t, t.fix);
            sweep_line<NQ>(b.data() + d * W, line, t);
        }
    for (int line = 0; line < NL; ++line)
        for (int n = 0; n < NQ; ++n) {
            const int s = slot<NQ, double>(line, n), o = line * NQ + n;
            double v[1];
            fixed_sums<NQ>(v, t.fix.shift, -1.0, [&](int d, int) { return a[d * W + s]; },
                           [&](int d, int) { return exps[d * NL + line]; });
            fixed[o] = v[0];
            fp64[o] = b[s] + b[W + s] + b[2 * W + s];
            long double x = 0;
            for (int d = 0; d < 3; ++d)
                for (int m = 0; m < NQ; ++m)
                    x += (long double)D[n * NQ + m] * in[(d * NL + line) * NQ + m];
            ref[o] = (double)x;
        }
}

}  // namespace

extern "C" void sweep_case(int nq, const double *in, double *fixed, double *fp64, double *ref,
                           int *exps) {
    switch (nq) {
        case 2: return run<2>(in, fixed, fp64, ref, exps);
        case 3: return run<3>(in, fixed, fp64, ref, exps);
        case 4: return run<4>(in, fixed, fp64, ref, exps);
        case 5: return run<5>(in, fixed, fp64, ref, exps);
        case 6: return run<6>(in, fixed, fp64, ref, exps);
        case 7: return run<7>(in, fixed, fp64, ref, exps);
        case 8: return run<8>(in, fixed, fp64, ref, exps);
        case 9: return run<9>(in, fixed, fp64, ref, exps);
        case 10: return run<10>(in, fixed, fp64, ref, exps);
        case 11: return run<11>(in, fixed, fp64, ref, exps);
        case 12: return run<12>(in, fixed, fp64, ref, exps);
        case 13: return run<13>(in, fixed, fp64, ref, exps);
        case 14: return run<14>(in, fixed, fp64, ref, exps);
        case 15: return run<15>(in, fixed, fp64, ref, exps);
        case 16: return run<16>(in, fixed, fp64, ref, exps);
    }
}

// n values of -y R 2^(e - 1024 - shift) by the integer multiply.
extern "C" void scale_case(int n, const long long *R, int e, int shift, const double *y, double *out) {
    for (int k = 0; k < n; ++k) {   // one line's sum, the other directions zero
        double v[1];
        const double z = fix_double(R[k]);
        fixed_sums<8>(v, shift, y[k], [&](int d, int) { return d ? 0.0 : z; }, [&](int, int) { return e; });
        out[k] = v[0];
    }
}
