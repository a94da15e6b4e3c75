"""The finer work items of small launches: a batch with the default tiles, from one element to
more passes than the grid holds, equals bit for bit the same batch with its tiles set."""
import pytest

from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("members", [[(7, (1, 1, 1))], [(3, (3, 3, 1)), (4, (7, 7, 7))],
                                     [(2, (25, 24, 23)), (7, (17, 16, 15)), (1, (2, 1, 1))]])
def test_items_of_small_launches(members, precision):
    import torch
    from paper_1604_08501_gb300.numa_vol import Batch, VolumeTerm
    made = []
    for n, (N, shape) in enumerate(members):
        w = wl.make_workload(N, shape, seed=30 + n, smooth_velocity=True)
        q = w.q_mixed() if precision == "mixed" else w.q
        made.append((VolumeTerm.from_problem(w.problem(), precision=precision), torch.from_numpy(q).cuda()))
    results = []
    for passes in (None, 3, 4, 32):
        with Batch(precision) as b:
            states = [q.clone() for _, q in made]
            for (vt, _), q in zip(made, states):
                b.add(vt, q)
            if passes:
                b.set_config(tile={nq: passes * (512 // nq ** 3) for nq in range(2, 9)})
            else:
                assert b.tile(8) == 4
            b.advance(2, 0.01)
            torch.cuda.synchronize()
            results.append(states)
    for states in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], states))
    assert not all(torch.equal(q, a) for (_, q), a in zip(made, results[0]))
    for vt, _ in made:
        vt.close()
