"""The fixed-point D sums of the FP64 kernels (csrc/fixed_sweep.cuh), compiled for the host, row
by row: each row's error against the FP64 sweep's on the same lines, the bound derived in the
header, and that no integer sum leaves its 64 bits."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1604_08501_gb300.numa_vol import diff_matrix

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1604_08501_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = next((d for d in ("/usr/local/cuda/include", os.path.join(os.path.dirname(os.path.dirname(
        shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")) if os.path.isdir(d)), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    so = str(tmp_path_factory.mktemp("rows") / "fixed_rows.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "fixed_sweep", "fixed_rows_host.cpp"),
                    os.path.join(CSRC, "gll.cpp"), "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", cuda], check=True, capture_output=True, text=True)
    return C.CDLL(so)


def errors(lib, lines, offsets=(0, 0)):
    n, _, nq = lines.shape
    lines = np.ascontiguousarray(lines)
    fix, fp = np.zeros((n, nq)), np.zeros((n, nq))
    exps = np.zeros((n, 3), dtype=np.int32)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.rows_case(nq, n, offsets[0], offsets[1], ptr(lines), ptr(fix), ptr(fp), ptr(exps))
    assert np.all(exps == -1) if nq == 2 else (nq >= 10 or np.all(exps >= 0))
    return fix, fp, np.all(exps >= 0, axis=1)


def rms(x):
    return np.sqrt(np.mean(x * x, axis=0))


def make(kind, nq, n, rng):
    """n triples of lines; a kind's spikes stand in all three lines of a triple."""
    x = rng.standard_normal((n, 3, nq))
    t = np.linspace(-1, 1, nq)
    if kind == "smooth":
        x = 1e3 * rng.standard_normal((n, 3, 1)) * (1 + 0.1 * np.sin(t + rng.uniform(0, 6, (n, 3, 1))))
    elif kind == "nearly uniform":
        x = 1000.0 + 1e-3 * x
    elif kind == "graded":
        x *= 2.0 ** rng.integers(-30, 1, x.shape)
    elif kind == "lines of several sizes":
        x *= 2.0 ** rng.integers(-200, 200, (n, 3, 1))
    elif kind == "even, small differences":   # the centre row's fluxes cancel to 1e-12 of the line
        y = np.abs(x) * 2.0 ** rng.integers(-40, 1, x.shape)
        x = y + y[..., ::-1] + 1e-12 * x
    elif kind.startswith("spike"):
        _, where, size = kind.split()
        x[..., {"centre": nq // 2, "end": 0, "other": nq - 1, "beside": 1, "ends": [0, nq - 1],
                "three": [0, 1, nq // 2]}[where]] *= float(size)
    return x


@pytest.mark.parametrize("nq", range(2, 17))
@pytest.mark.parametrize("kind", ["random", "smooth", "nearly uniform", "graded", "lines of several sizes",
                                  "even, small differences", "spike centre 1e3", "spike centre 1e10",
                                  "spike end 1e3", "spike end 1e10", "spike other 1e10", "spike beside 1e3",
                                  "spike end 20", "spike beside 20", "spike ends 1e3", "spike three 1e3"])
def test_no_row_less_exact_than_the_fp64_sweeps(lib, nq, kind):
    """Root mean square over 2000 sums, one line alone and the sum of three, at the same row of
    each and at different rows: at most the FP64 sweep's, and 5 % for the sample."""
    rng = np.random.default_rng(nq)
    x = make(kind, nq, 2000, rng)
    alone = x.copy()
    alone[:, 1:] = 0.0
    for lines, offsets in ((alone, (0, 0)), (x, (0, 0)), (x, (1, nq // 2))):
        fix, fp, _ = errors(lib, lines, offsets)
        assert np.all(rms(fix) <= 1.05 * rms(fp)), (offsets, rms(fix) / rms(fp))


def units(nq, lines):
    """Bound of a line's error in each row: (1.5 pairs + 3) units, a unit of row i being
    2^(e - 1021 - s_i) with 2^(60 - s_i) <= row sum of |D| and 2^(e - 1023) <= largest value."""
    half = nq // 2
    row = np.frexp(np.abs(diff_matrix(nq - 1)).sum(1))[1]         # row sum < 2^row, s_i = 61 - row
    top = np.frexp(np.abs(lines).max(-1))[1]                      # largest < 2^top, e - 1022 = top
    return (1.5 * half + 3) * np.ldexp(1.0, row + top[..., None] - 60)


@pytest.mark.parametrize("nq", range(3, 17))
def test_bound(lib, nq):
    """Values just below a power of two with the signs of D's rows (the largest sums) and with
    random signs, and lines whose smaller values are cut: within the derived bound."""
    rng = np.random.default_rng(nq)
    D = diff_matrix(nq - 1)
    big = np.nextafter(2.0, 0.0)
    signs = np.where(D < 0, -big, big)
    x = np.concatenate([np.repeat(signs[:, None], 3, 1), -np.repeat(signs[:, None], 3, 1),
                        big * rng.choice([-1.0, 1.0], (500, 3, nq)),
                        (1 + rng.random((500, 3, nq))) * 2.0 ** rng.integers(-12, 1, (500, 3, nq))])
    for offsets in ((0, 0), (1, nq // 2)):
        fix, _, fixed = errors(lib, x, offsets)   # triples with a line left in FP64 are not fixed point
        u = units(nq, x)
        bound = sum(np.roll(u[:, d], -o, axis=-1) for d, o in enumerate((0,) + offsets))
        value = sum(np.roll(np.abs(x[:, d] @ D.T), -o, axis=-1) for d, o in enumerate((0,) + offsets))
        # two shifted directions, cut to the largest's unit; one rounding
        bound = bound + 2 * bound / (1.5 * (nq // 2) + 3) + 2.0 ** -53 * value
        assert fixed.sum() > 500 and np.all(np.abs(fix)[fixed] <= bound[fixed])


@pytest.mark.parametrize("nq", range(3, 17))
def test_tables(lib, nq):
    """The integer tables: within half a unit of D at each row's scale, words in range, and no
    partial sum of the middle words beyond 63 bits for any line."""
    half = nq // 2
    raw = np.zeros(4 * half * half + 4 * half + 1 + nq, dtype=np.int32)
    lib.tables_case(nq, raw.ctypes.data_as(C.c_void_p))
    t = [int(v) for v in raw]
    take = lambda n: [t.pop(0) for _ in range(n)]
    deh, del_, doh, dol = ([take(half) for _ in range(half)] for _ in range(4))
    dch, dcl, dcrh, dcrl = (take(half) for _ in range(4))
    shift, row = t[0], t[1:]
    D = diff_matrix(nq - 1)
    assert row == row[::-1] and min(row) == 0

    def value(h, l, r):   # twice the entry, at the row's scale
        assert abs(h) < 2 ** 31 and abs(l) <= 2 ** 30 and l % 2 == 0
        return (h * 2 ** 31 + l) / 2.0 ** (shift + 3 + row[r])

    eps = lambda r: 2.0 ** -(shift + 3 + row[r]) + 2.0 ** -52 * np.abs(D[r]).max()
    for r in range(half):
        assert 2 ** 60 <= np.abs(D[r]).sum() * 2.0 ** (shift + 3 + row[r]) < 2 ** 61
        for m in range(half):
            assert abs(value(deh[r][m], del_[r][m], r) - (D[r, m] + D[r, nq - 1 - m])) <= eps(r)
            assert abs(value(doh[r][m], dol[r][m], r) - (D[r, m] - D[r, nq - 1 - m])) <= eps(r)
        even = sum(2 ** 30 * abs(l) + 2 ** 31 * abs(h) for h, l in zip(deh[r], del_[r]))
        odd = sum(2 ** 30 * abs(l) + 2 ** 31 * abs(h) for h, l in zip(doh[r], dol[r]))
        if nq % 2:
            assert abs(value(dch[r], dcl[r], r) / 2 - D[r, half]) <= eps(r)
            assert abs(value(dcrh[r], dcrl[r], half) / 2 - D[half, r]) <= eps(half)
            even += 2 ** 29 * abs(dcl[r]) + 2 ** 31 * abs(dch[r])
        assert max(even, odd) + 2 ** 30 < 2 ** 63
    if nq % 2:
        assert sum(2 ** 30 * abs(l) + 2 ** 31 * abs(h) for h, l in zip(dcrh, dcrl)) + 2 ** 30 < 2 ** 63
