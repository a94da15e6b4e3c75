"""What a batch's configuration sets is what runs, also where it equals the default: four passes
set for a launch of few items are four passes; tiles never set stay automatic through a round trip."""
import ctypes as C

import pytest

from paper_1604_08501_gb300 import workload as wl

pytestmark = pytest.mark.gpu

FOUR = {nq: 4 * (512 // nq ** 3) for nq in range(2, 9)}


def best_ms(torch, b, nsteps=20, reps=5):
    b.advance(nsteps, 1e-6)
    times = []
    for _ in range(reps):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        b.advance(nsteps, 1e-6)
        t1.record()
        t1.synchronize()
        times.append(t0.elapsed_time(t1))
    return min(times)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_default_tiles_set_are_honoured(precision):
    """64 elements of N = 7: automatic, one element an item on 64 CTAs; four passes set, 16 CTAs
    taking four elements one after the other, about four times as long (twice is asked for)."""
    import torch
    from paper_1604_08501_gb300 import _lib
    from paper_1604_08501_gb300.numa_vol import Batch, VolumeTerm
    w = wl.make_workload(7, (4, 4, 4), seed=3, smooth_velocity=True)
    q = torch.from_numpy(w.q_mixed() if precision == "mixed" else w.q).cuda()
    lib = _lib.load()
    with VolumeTerm.from_problem(w.problem(), precision=precision) as vt, Batch(precision) as b:
        b.add(vt, q)
        auto = best_ms(torch, b)
        b.set_config(costliest_first=True)                  # tiles not given: automatic still
        assert best_ms(torch, b) < 1.5 * auto
        b.set_config(tile=FOUR)
        assert b.config()["tile"] == FOUR and best_ms(torch, b) > 2 * auto
        saved = _lib.numa_batch_config()
        assert lib.numa_batch_get_config(b.handle, C.byref(saved)) == 0
        with Batch(precision) as c:                         # a saved configuration, restored
            c.add(vt, q)
            untuned = _lib.numa_batch_config()
            assert lib.numa_batch_get_config(c.handle, C.byref(untuned)) == 0
            assert list(untuned.tile[2:]) == list(saved.tile[2:])
            assert lib.numa_batch_set_config(c.handle, C.byref(saved)) == 0
            assert best_ms(torch, c) > 2 * auto
            assert lib.numa_batch_set_config(c.handle, C.byref(untuned)) == 0
            assert best_ms(torch, c) < 1.5 * auto
        b.set_config(tile={8: 1})
        assert best_ms(torch, b) < 1.5 * auto
