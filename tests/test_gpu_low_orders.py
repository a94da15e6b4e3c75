"""Low orders, whose CTAs hold several elements, at element counts around a CTA's and the
prefetch's, in NUMA_FP64 (1e-12) and NUMA_MIXED (1e-5) against the oracle; and an element's
rhs depends on that element alone, whichever elements share its CTA."""
import numpy as np
import pytest

import oracle
from conftest import eos_banded_theta_ratio, rel_err
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def evaluate(w, q, precision, cut=None):
    """rhs of the first `cut` elements of w (all without cut)."""
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    prob = w.problem()
    if cut is not None:
        m = cut * (w.N + 1) ** 3
        for key in ("g", "Jinv", "rho_ref", "rhotheta_ref"):
            prob[key] = np.ascontiguousarray(prob[key][..., :m])
        prob["Ne"] = cut
        q = np.ascontiguousarray(q[:, :m])
    if precision == "mixed":
        q = wl.perturbation_state(q, prob["rho_ref"], prob["rhotheta_ref"])
    with VolumeTerm.from_problem(prob, precision=precision) as vt:
        return vt.rhs(torch.from_numpy(q).cuda()).cpu().numpy()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("N,shape", [(1, (31, 1, 1)), (1, (8, 4, 1)), (1, (11, 3, 1)), (1, (13, 13, 13)),
                                     (2, (7, 1, 1)), (2, (4, 2, 1)), (2, (9, 1, 1)), (2, (19, 17, 13)),
                                     (3, (3, 1, 1)), (3, (5, 1, 1)), (3, (13, 11, 9)), (4, (17, 13, 11)),
                                     (5, (11, 9, 8)), (6, (11, 9, 5))])
def test_element_counts(N, shape, precision, tol):
    w = wl.make_workload(N, shape, seed=20 + N, tracers=shape[0] % 3)
    ref = oracle.vol_rhs_o2(w.problem(), w.q)
    for mx, _ in rel_err(evaluate(w, w.q, precision), ref):
        assert mx <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_an_element_stands_alone(N, precision):
    # Theta' in every range of the equation of state, mixed among neighbours
    w = wl.make_workload(N, (5, 3, 3), seed=60 + N)
    q = w.q.copy()
    q[4] = w.rhotheta_ref * (1.0 + eos_banded_theta_ratio(w.M, seed=N))
    n3 = (N + 1) ** 3
    full = evaluate(w, q, precision)
    for cut in (1, 7, 8, 9, 32, 33):
        assert np.array_equal(evaluate(w, q, precision, cut), full[:, :cut * n3])
    other = q.copy()
    other[:, 3 * n3:4 * n3] = np.nan
    got = evaluate(w, other, precision)
    keep = np.r_[0:3 * n3, 4 * n3:w.M]
    assert np.array_equal(got[:, keep], full[:, keep])
