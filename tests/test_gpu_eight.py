"""N = 7 without tracers in NUMA_FP64 and NUMA_DF64: a launch of many elements takes the kernel
of two points per thread, a launch of few the one of one point; an element's rhs is the same
bit for bit from both, also where it leaves the double-float range or is not finite."""
import numpy as np
import pytest

import oracle
from conftest import rel_err
from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("odd", [False, True])
def test_both_kernels_agree(precision, odd):
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = wl.make_workload(7, (6, sms, 1), seed=17)
    prob, q, n3 = w.problem(), w.q.copy(), 512
    if odd:   # a value beyond the double-float range, an infinity, a negative density
        q[1, 3 * n3 + 5] = 2.0 ** 45
        q[2, 5 * n3 + 300] = np.inf
        q[0, 6 * n3 + 511] *= -1.0
        q[4, 8 * n3:9 * n3] = w.rhotheta_ref[8 * n3:9 * n3] * 1.05   # |x| > 1/64
    with VolumeTerm.from_problem(prob, precision=precision) as vt:
        many = vt.rhs(torch.from_numpy(q).cuda()).cpu().numpy()
    if not odd:
        for mx, _ in rel_err(many, oracle.vol_rhs_o2(prob, q)):
            assert mx <= 1e-12
    m = 100 * n3
    for key in ("g", "Jinv", "rho_ref", "rhotheta_ref"):
        prob[key] = np.ascontiguousarray(prob[key][..., :m])
    prob["Ne"] = 100
    with VolumeTerm.from_problem(prob, precision=precision) as vt:
        few = vt.rhs(torch.from_numpy(np.ascontiguousarray(q[:, :m])).cuda()).cpu().numpy()
    assert np.array_equal(few, many[:, :m], equal_nan=True)
