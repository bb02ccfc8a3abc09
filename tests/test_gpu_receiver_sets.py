"""GPU tests of changing receiver sets on one handle.

The device tables of a set serve the next one: alternating sets take no more memory
(one set's tables are 46 MB here; 8 MB allow for the allocator's own), and a set that
does not fit the memory cap is refused and leaves the set before in force.  Values
of a set are the same bits whenever they are asked for.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu


def _points(n, seed):
    return np.random.default_rng(seed).uniform(0.05, 0.95, (n, 2))


@pytest.fixture
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def test_alternating_sets_keep_their_memory_and_values(torch):
    from paper_2606_09688_gb300 import Solver
    a, b, c = _points(2000, 1), _points(7, 2), _points(1999, 3)
    with Solver(W.layered_2d(6, 2)) as s:
        s.solve(-1)
        first = [s.receiver_values(8, a).clone(), s.receiver_values(5, b).clone(), s.receiver_values(8, c).clone()]
        free = []
        for _ in range(4):
            assert torch.equal(s.receiver_values(8, a), first[0])
            assert torch.equal(s.receiver_values(5, b), first[1])
            assert torch.equal(s.receiver_values(8, c), first[2])
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
        assert free[0] - free[-1] < 8 << 20   # the first round also loads what the comparison needs


def test_a_refused_set_leaves_the_set_before_in_force(torch):
    from paper_2606_09688_gb300 import Solver, StError
    from paper_2606_09688_gb300 import st as B
    a, big, c = _points(40, 1), _points(100000, 2), _points(30, 3)   # big: 205 MB of values alone
    with Solver(W.layered_2d(6, 2), mem_cap_bytes=192 << 20) as s:
        s.solve(-1)
        first, third = s.receiver_values(6, a).clone(), s.receiver_values(6, c).clone()
        assert torch.equal(s.receiver_values(6, a), first)
        for _ in range(2):
            with pytest.raises(StError) as e:
                s.receiver_values(8, big)
            assert e.value.code == B.ST_ERR_OOM
            assert torch.equal(s.receiver_values(6, a), first)
        assert torch.equal(s.receiver_values(6, c), third)
