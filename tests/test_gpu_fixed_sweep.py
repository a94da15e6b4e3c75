"""NUMA_FP64 where lines leave the fixed-point range of the D sweeps: metric terms scaled
by a power of two and J^-1 by its inverse (exact), so that every line, or the lines of one
direction only, takes the FP64 sweep.  The rhs must stay that of the unscaled geometry."""
import numpy as np
import pytest

import oracle
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def rhs(prob, q):
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    with VolumeTerm.from_problem(prob) as vt:
        out = vt.rhs(torch.from_numpy(q).to("cuda:0"))
        return out.cpu().numpy()


@pytest.mark.parametrize("N", [1, 2, 4, 7, 8, 11, 15])
@pytest.mark.parametrize("power", [-880, 0, 940])
def test_lines_outside_the_fixed_point_range(N, power):
    w = wl.make_workload(N, (2, 1, 3), seed=5)
    prob = w.problem()
    ref = oracle.vol_rhs_o2(prob, w.q)
    prob["g"] = np.ldexp(prob["g"], power)
    prob["Jinv"] = np.ldexp(prob["Jinv"], -power)
    got = rhs(prob, w.q)
    for b in range(5):
        assert np.max(np.abs(got[b] - ref[b])) <= 1e-12 * np.max(np.abs(ref[b]))


@pytest.mark.parametrize("N", [2, 4, 7, 11])
@pytest.mark.parametrize("d", [0, 1, 2])
def test_one_direction_outside_the_fixed_point_range(N, d):
    w = wl.make_workload(N, (2, 1, 3), seed=6)
    prob = w.problem()
    g = prob["g"].copy()
    prob["g"] = g.copy()
    prob["g"][3 * d:3 * d + 3] = 0.0
    ref = oracle.vol_rhs_o2(prob, w.q)
    prob["g"][3 * d:3 * d + 3] = np.ldexp(g[3 * d:3 * d + 3], -900)   # adds nothing at 2^-53
    got = rhs(prob, w.q)
    for b in range(5):
        assert np.max(np.abs(got[b] - ref[b])) <= 1e-12 * np.max(np.abs(ref[b]))


@pytest.mark.parametrize("N", [2, 7, 11])
def test_not_finite_states(N):
    """An infinity or a NaN reaches the rhs of its own element and no other."""
    w = wl.make_workload(N, (3, 1, 1), seed=7)
    n3 = (N + 1) ** 3
    ref = rhs(w.problem(), w.q)
    q = w.q.copy()
    q[1, n3 + 2] = np.inf
    q[4, n3 + n3 // 2] = np.nan
    got = rhs(w.problem(), q)
    other = np.r_[0:n3, 2 * n3:3 * n3]
    assert np.array_equal(got[:, other], ref[:, other])
    assert np.isnan(got[4, n3:2 * n3]).any() and not np.isfinite(got[1, n3:2 * n3]).all()
