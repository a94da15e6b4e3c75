"""The fixed-point D sweep of the FP64 kernels (csrc/fixed_sweep.cuh), compiled for the
host, against the FP64 sweep it stands for and a long-double one, at every Nq."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1604_08501_gb300", "csrc")
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = next((d for d in ("/usr/local/cuda/include", os.path.join(os.path.dirname(os.path.dirname(
        shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")) if os.path.isdir(d)), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_sweep.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "fixed_sweep", "fixed_sweep_host.cpp"),
                    os.path.join(CSRC, "gll.cpp"), "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", cuda], check=True, capture_output=True, text=True)
    return C.CDLL(so)


def sweep(lib, nq, lines):
    lines = np.ascontiguousarray(lines, dtype=np.float64)
    assert lines.shape == (3, nq * nq, nq)
    out = [np.zeros((nq * nq, nq)) for _ in range(3)]
    exps = np.zeros((3, nq * nq), dtype=np.int32)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.sweep_case(nq, ptr(lines), ptr(out[0]), ptr(out[1]), ptr(out[2]), ptr(exps))
    return out[0], out[1], out[2], exps


def line_scale(nq, lines):
    """Largest |D| row sum times the line's largest value, summed over the directions."""
    from paper_1604_08501_gb300.numa_vol import diff_matrix
    rows = np.abs(diff_matrix(nq - 1)).sum(1).max()
    return (rows * np.abs(lines).max(2)).sum(0)[:, None]


@pytest.mark.parametrize("nq", range(2, 17))
@pytest.mark.parametrize("kind", ["random", "smooth", "graded", "tiny and large lines"])
def test_error_at_most_the_fp64_sweeps(lib, nq, kind):
    rng = np.random.default_rng(nq)
    worst_fix = worst_fp = 0.0
    for _ in range(20):
        x = rng.standard_normal((3, nq * nq, nq))
        if kind == "smooth":
            t = np.linspace(-1, 1, nq)
            c = rng.standard_normal((3, nq * nq, 1)) * 1e3
            x = c * (1 + 0.1 * np.sin(t + rng.uniform(0, 6, (3, nq * nq, 1))))
        elif kind == "graded":     # magnitudes over 30 binades along a line
            x = x * 2.0 ** rng.integers(-30, 1, x.shape)
        elif kind == "tiny and large lines":
            x = x * 2.0 ** rng.integers(-200, 200, (3, nq * nq, 1))
        fix, fp, ref, exps = sweep(lib, nq, x)
        assert np.all(exps > 0 if nq > 2 else exps == -1)   # Nq = 2 stays in FP64
        scale = line_scale(nq, x)
        # the bound derived in fixed_sweep.cuh: 2^-55 of the scale, and one rounding
        assert np.all(np.abs(fix - ref) <= scale * 2.0 ** -55 + 2 * EPS * np.abs(ref))
        worst_fix = max(worst_fix, np.sqrt(np.mean(((fix - ref) / scale) ** 2)))
        worst_fp = max(worst_fp, np.sqrt(np.mean(((fp - ref) / scale) ** 2)))
    assert worst_fix <= worst_fp


@pytest.mark.parametrize("nq", range(2, 17))
def test_lines_outside_fixed_point(lib, nq):
    """Infinities, NaN, values near overflow and tiny values take the FP64 sweep, alone or
    beside lines in fixed point, with its results; zeros of either sign give zero."""
    rng = np.random.default_rng(100 + nq)
    x = rng.standard_normal((3, nq * nq, nq))
    x[0, 0, 0] = np.inf
    x[1, 1, nq - 1] = np.nan
    x[2, 2] *= 1e306
    x[0, 3] *= 1e-300
    x[1, 3] *= 1e-260
    x[2, 3] = 0.0
    fix, fp, ref, exps = sweep(lib, nq, x)
    for d, line in ((0, 0), (1, 1), (2, 2), (0, 3), (1, 3)):
        assert exps[d, line] == -1
    for line in range(4):
        a, b = np.isfinite(fp[line]), np.isfinite(fix[line])
        assert np.array_equal(a, b)
        assert np.array_equal(np.isnan(fp[line]), np.isnan(fix[line]))
        tol = (line_scale(nq, x)[line] if line == 3 else np.abs(fp[line][a]).max(initial=0.0)) * 4 * EPS
        assert np.all(np.abs(fix[line][a] - fp[line][a]) <= tol)
    z = np.zeros_like(x)
    z[:, ::2] = -0.0
    z[0, 1, 1] = -0.0
    fix, _, _, exps = sweep(lib, nq, z)
    assert np.all(exps > 0 if nq > 2 else exps == -1) and np.all(fix == 0.0)


@pytest.mark.parametrize("nq", range(2, 17))
def test_largest_sums(lib, nq):
    """Values of the largest magnitudes a line holds, with the signs of D's rows: the sums
    reach the format's bounds in every direction at once."""
    from paper_1604_08501_gb300.numa_vol import diff_matrix
    D = diff_matrix(nq - 1)
    big = np.nextafter(2.0, 0.0)
    x = np.empty((3, nq * nq, nq))
    for line in range(nq * nq):
        x[:, line] = np.where(D[line % nq] < 0, -big, big) * (-1) ** (line // nq)
    fix, fp, ref, _ = sweep(lib, nq, x)
    assert np.all(np.abs(fix - ref) <= line_scale(nq, x) * 2.0 ** -55 + 2 * EPS * np.abs(ref))


@pytest.mark.parametrize("e", [200, 1023, 1900])
def test_scaled_sums_round_once(lib, e):
    """fix_scale against exact rational arithmetic: half a unit in the last place (and the
    truncation of the product at 2^-63) wherever the result is normal."""
    from fractions import Fraction
    rng = np.random.default_rng(e)
    n, shift = 400, 53
    R = rng.integers(-3 * 2 ** 60, 3 * 2 ** 60, n) >> rng.integers(0, 62, n)
    R[:6] = [0, 1, -1, 3 * 2 ** 60, -3 * 2 ** 60, 2 ** 53 + 1]
    y = rng.standard_normal(n) * 2.0 ** rng.integers(-60, 60, n)
    y[6:10] = [1.0, -1.0, 2.0, np.nextafter(1.0, 0.0)]
    if e == 1023:   # factors outside the integer multiply's range
        y[10:16] = [0.0, 1e-290, 1e290, np.inf, np.nan, -5e-324]
    out = np.zeros(n)
    lib.scale_case(n, R.ctypes.data_as(C.c_void_p), e, shift, y.ctypes.data_as(C.c_void_p),
                   out.ctypes.data_as(C.c_void_p))
    for k in range(n):
        if not np.isfinite(y[k]) or y[k] == 0.0 or R[k] == 0:
            if R[k] != 0:
                assert np.isnan(out[k]) == np.isnan(y[k]) and np.isinf(out[k]) == np.isinf(y[k])
            continue
        want = -Fraction(float(y[k])) * int(R[k]) * Fraction(2) ** (e - 1024 - shift)
        if not Fraction(2) ** -1021 < abs(want) < Fraction(2) ** 1022:
            continue
        got = Fraction(float(out[k]))
        ulp = Fraction(2) ** (int(np.frexp(out[k])[1]) - 53)
        assert abs(got - want) <= ulp * (Fraction(1, 2) + Fraction(1, 2 ** 9)), (k, R[k], y[k])
