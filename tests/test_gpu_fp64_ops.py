"""The FP64 kernels' reciprocal and FP64 <-> FP32 moves (csrc/fp64_ops.cuh) value by value, and the
pressure series without its FP32 tail (gamma above about 5)."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import oracle
from conftest import rel_err
from paper_1604_08501_gb300 import build
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fp64_ops") / "fp64_ops.so")
    subprocess.run([build._nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", *build.ARCH, "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "fp64_ops", "fp64_ops_device.cu"), "-o", so], check=True,
                   capture_output=True, text=True)
    return C.CDLL(so)


def evaluate(lib, x, f):
    x, f = np.ascontiguousarray(x, np.float64), np.ascontiguousarray(f, np.float32)
    n = len(x)
    rcp, drcp, cut, wide = np.zeros(n), np.zeros(n), np.zeros(n, np.float32), np.zeros(n)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    assert lib.eval_case(n, ptr(x), ptr(f), ptr(rcp), ptr(drcp), ptr(cut), ptr(wide)) == 0
    return rcp, drcp, cut, wide


def doubles(rng, n):
    """Random mantissas and mantissas next to 1 and 2 at every exponent field, both signs."""
    m = rng.integers(0, 2 ** 52, n, dtype=np.uint64)
    m[::4] = rng.integers(0, 1 << 12, len(m[::4]), dtype=np.uint64)
    m[1::4] = (2 ** 52 - 1) - rng.integers(0, 1 << 12, len(m[1::4]), dtype=np.uint64)
    e = rng.integers(1, 2047, n, dtype=np.uint64)
    for k, field in enumerate((1, 22, 23, 24, 1022, 1023, 2022, 2023, 2024, 2046)):
        e[k::40] = field
    return ((rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)


def test_reciprocal(lib):
    x = doubles(np.random.default_rng(1), 40000)
    rcp, drcp, _, _ = evaluate(lib, x, np.zeros(len(x)))
    field = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(0x7FF)
    inner = (field >= 23) & (field <= 2023)
    assert np.array_equal(rcp[~inner].view(np.uint64), drcp[~inner].view(np.uint64))
    worst = Fraction(0)
    for a, y in zip(x[inner], rcp[inner]):
        # |y - 1/a| in units of y's last place: 1/2 and the iteration's e^3, at most 0.0005 of them
        worst = max(worst, abs(Fraction(float(y)) - 1 / Fraction(float(a))) / Fraction(float(np.spacing(abs(y)))))
    assert worst <= Fraction(5005, 10000), float(worst)
    print("largest error", float(worst), "units; not the correctly rounded", np.mean(rcp[inner] != drcp[inner]))
    special = np.array([0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1023, np.inf, -np.inf, np.nan, 1.0, -1.0, 2.0, 0.5])
    rcp, drcp, _, _ = evaluate(lib, special, np.zeros(len(special)))
    assert np.array_equal(np.isnan(rcp), np.isnan(drcp))
    keep = ~np.isnan(drcp)
    assert np.array_equal(rcp[keep].view(np.uint64), drcp[keep].view(np.uint64))


def test_moves_between_fp64_and_fp32(lib):
    rng = np.random.default_rng(2)
    x = doubles(rng, 40000)
    x = x[np.abs(x) < 2.0 ** 128]
    x[:4] = [0.0, -0.0, 2.0 ** -126, -np.nextafter(2.0 ** -126, 0.0)]
    f = rng.integers(0, 2 ** 32, len(x), dtype=np.uint32).view(np.float32)
    f[:6] = [0.0, -0.0, 1.0, -1.0, 2.0 ** -126, np.finfo(np.float32).max]
    f[~np.isfinite(f)] = 1.5
    _, _, cut, wide = evaluate(lib, x, f)
    # towards zero to 24 bits; zero below the normal floats
    want = np.where(np.abs(x) < 2.0 ** -126, 0.0, (x.view(np.uint64) & ~np.uint64(2 ** 29 - 1)).view(np.float64))
    assert np.array_equal(cut.astype(np.float64), want)
    assert np.array_equal(wide, np.where(np.abs(f) < 2.0 ** -126, 0.0, f.astype(np.float64)))


@pytest.mark.parametrize("N", [2, 4, 7, 11])
def test_series_without_the_fp32_tail(N):
    """gamma = 7.5: terms 6 to 9 are more than 2^-34 of the sum, so all nine run in FP64."""
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    w = wl.make_workload(N, (3, 2, 1), seed=N)
    prob = w.problem()
    prob["p0"], prob["R"], prob["cp"] = 1e5, 287.0, 287.0 * 7.5 / 6.5
    q = w.q.copy()
    x = np.random.default_rng(N).uniform(-1, 1, w.M) / 65
    q[4] = prob["rhotheta_ref"] * (1 + x)
    ref = oracle.vol_rhs_o2(prob, q)
    with VolumeTerm.from_problem(prob) as vt:
        got = vt.rhs(torch.from_numpy(q).cuda()).cpu().numpy()
    for mx, _ in rel_err(got, ref):
        assert mx <= 1e-12
