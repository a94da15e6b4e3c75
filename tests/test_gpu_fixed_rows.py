"""NUMA_FP64, row by row of D: on unit metrics with p = 0 the rhs of rho is -(D_r U1 + D_s U2 +
D_t U3), so each row's error is that of its sum alone.  It must follow the terms of the row's
even-odd sum, in the centre row of odd Nq the differences D[c][m] (F_m - F_{N-m}) alone, also
where the centre flux, which that row does not use, dominates the line."""
import numpy as np
import pytest

from paper_1604_08501_gb300.numa_vol import diff_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 16))
@pytest.mark.parametrize("kind", ["random", "nearly uniform", "centre 1e10"])
@pytest.mark.parametrize("d", [0, 1, 2])
def test_each_row_to_its_own_terms(N, kind, d):
    import torch
    from paper_1604_08501_gb300.numa_vol import VolumeTerm
    nq = N + 1
    Ne = 6 * torch.cuda.get_device_properties(0).multi_processor_count + 1 if N == 7 else 37
    M = Ne * nq ** 3
    rng = np.random.default_rng(N)
    F = rng.standard_normal((Ne, nq, nq, nq))           # [e][k][j][i], lines along axis 3 - d
    axis = 3 - d
    if kind == "nearly uniform":
        F = 1000.0 + 1e-3 * F
    elif kind == "centre 1e10":
        F = np.moveaxis(F, axis, 3)
        F[..., nq // 2] *= 1e10
        F = np.moveaxis(F, 3, axis)
    g = np.zeros((9, M))
    g[0] = g[4] = g[8] = 1.0
    zero, one = np.zeros(M), np.ones(M)
    q = np.zeros((5, M))
    q[0], q[1 + d] = 1.0, F.reshape(-1)
    put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with VolumeTerm(N, Ne, put(g), put(one), put(zero), put(zero), 1.0, 1.0, 3.5, 0.0) as vt:
        got = vt.rhs(put(q))[0].cpu().numpy().reshape(F.shape)
    D = diff_matrix(N).astype(np.longdouble)
    L = np.moveaxis(F, axis, 3)[:64].astype(np.longdouble)
    ref = -(L @ D.T)
    # terms of the even-odd sums: De (F_m + F_{N-m}) and Do (F_m - F_{N-m}), at most
    # (|De| + |Do|) (|F_m| + |F_{N-m}|); the centre row's as they are
    own = np.abs(L) @ np.maximum(np.abs(D), np.abs(D[:, ::-1])).T
    if nq % 2:
        c = nq // 2
        own[..., c] = np.abs(L[..., :c] - L[..., :c:-1]) @ np.abs(D[c, :c])
    err = np.abs(np.moveaxis(got, axis, 3)[:64] - ref)
    assert np.all(err <= (nq // 2 + 3) * 2.0 ** -53 * own)
