"""NUMA_MIXED at N = 8..15 on meshes either side of the line between the whole-element kernel
(fewer than two elements per SM) and the plane-walking one: at 1e-5 of the oracle, and the
elements both evaluate equal to 1e-5 of each other; the host path bit for bit the device's."""
import numpy as np
import pytest

import oracle
from conftest import rel_err
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(8, 16))
@pytest.mark.parametrize("tracers", [0, 1, 3])
def test_both_sides_of_the_line(N, tracers):
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = wl.make_workload(N, (2, sms, 1), seed=N, tracers=tracers)
    prob, n3 = w.problem(), (N + 1) ** 3
    q = w.q_mixed()
    ref = oracle.vol_rhs_o2(prob, w.q)
    with VolumeTerm.from_problem(prob, precision="mixed") as vt:
        whole = vt.rhs(torch.from_numpy(q).cuda()).cpu().numpy()
        assert np.array_equal(vt.rhs_host(q), whole)
    for mx, _ in rel_err(whole, ref):
        assert mx <= 1e-5
    m = (2 * sms - 1) * n3
    for key in ("g", "Jinv", "rho_ref", "rhotheta_ref"):
        prob[key] = np.ascontiguousarray(prob[key][..., :m])
    prob["Ne"] = 2 * sms - 1
    with VolumeTerm.from_problem(prob, precision="mixed") as vt:
        part = vt.rhs(torch.from_numpy(np.ascontiguousarray(q[:, :m])).cuda()).cpu().numpy()
    for mx, _ in rel_err(part, whole[:, :m]):
        assert mx <= 1e-5
