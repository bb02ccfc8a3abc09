"""GPU energy over several batches of times (st_energy).

Every time is a row of its own in the level kernels, so a call over many times
(several batches, the last one ragged) has the bits of calls of one time each;
the first call allocates the workspace, later ones reuse or grow it.  Times at
0, T, on and next to the knots, in no order.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,count", [(W.travelling_wave(6), 333), (W.layered_2d(9, 2), 131)])
def test_many_times_equal_single_times(p, count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    rng = np.random.default_rng(5)
    times = np.concatenate([[p.T, 0.0, 0.5 * p.T, np.nextafter(0.5 * p.T, 0.0), p.T / 128],
                            rng.uniform(0.0, p.T, count - 5)])
    with Solver(p) as s:
        s.solve(-1)
        few = np.concatenate([s.energy(times[:1]), s.energy(times[1:2])])
        many = s.energy(times)
        single = np.array([s.energy(times[i:i + 1])[0] for i in range(0, count, 10)])
    assert np.isfinite(many).all() and many.max() > 0
    assert np.array_equal(few, many[:2])
    assert np.array_equal(single, many[::10])
