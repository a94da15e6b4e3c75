"""NUMA_MIXED at N = 8..15: an element's result does not depend on the size of its mesh (which
chooses between two kernels), also where its points need different forms of the equation of state."""
import numpy as np
import pytest

import oracle
from conftest import rel_err
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(8, 16))
@pytest.mark.parametrize("tracers", [0, 2])
def test_an_element_in_a_small_and_in_a_large_mesh(N, tracers):
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = wl.make_workload(N, (2, sms, 1), seed=N, tracers=tracers)
    prob, n3 = w.problem(), (N + 1) ** 3
    q = w.q.copy()
    # |Theta'| / Theta_ref at random points: within the short series, the long one, beyond both
    x = np.random.default_rng(N).choice([1e-3, 0.1, -0.3, 0.8], w.M, p=[0.7, 0.15, 0.1, 0.05])
    ref0 = prob["rhotheta_ref"]
    q[4] = ref0 * (1 + x)
    given = q.astype(np.float64).copy()
    given[0] -= prob["rho_ref"]
    given[4] = ref0 * x
    given = given.astype(np.float32)
    few = 5
    with VolumeTerm.from_problem(prob, precision="mixed") as vt:
        large = vt.rhs(torch.from_numpy(given).cuda()).cpu().numpy()
    for key in ("g", "Jinv", "rho_ref", "rhotheta_ref"):
        prob[key] = np.ascontiguousarray(prob[key][..., :few * n3])
    prob["Ne"] = few
    with VolumeTerm.from_problem(prob, precision="mixed") as vt:
        small = vt.rhs(torch.from_numpy(np.ascontiguousarray(given[:, :few * n3])).cuda()).cpu().numpy()
    ref = oracle.vol_rhs_o2(prob, np.ascontiguousarray(q[:, :few * n3]))
    for mx, _ in rel_err(small, ref):
        assert mx <= 1e-5
    assert np.array_equal(small, large[:, :few * n3])
