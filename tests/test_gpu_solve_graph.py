"""GPU tests of the refinement that runs as one graph (direct and space-eigenbasis components).

The first sweep reads F and overwrites U, the last one resets the sweep counter:
a repeated solve has the same bits and the same record, and zero data give zero
coefficients without a sweep being counted.  Neither needs a tolerance.
Cases: space eigenbasis (1D, many time rows), direct with one FP64 sweep, direct
with several FP32 sweeps, with split and plain time transforms.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu

CASES = [(1, 2, 9, 0), (1, 3, 4, 0), (2, 2, 5, 1), (2, 6, 2, 1), (2, 7, 3, 0), (3, 3, 3, 1)]


def _problem(d, jx, jt, scale):
    return W.Problem(d=d, lo=(0.0,) * d, hi=(1.0,) * d, T=1.0, c2=lambda x: 1.0 + 0.5 * (x[:, 0] > 0.4), J=0, mx=jx, mt=jt,
                     u0=lambda x: scale * np.prod(np.sin(np.pi * x), axis=1))


@pytest.mark.parametrize("d,jx,jt,prec", CASES)
def test_repeated_solves_are_the_same(d, jx, jt, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    with Solver(_problem(d, jx, jt, 1.0), precision=prec) as s:
        runs = [(s.solve(0), s.coeffs(0)) for _ in range(3)]
    assert runs[0][0].sweeps >= 1 and np.abs(runs[0][1]).max() > 0.1
    for info, U in runs[1:]:
        assert np.array_equal(U, runs[0][1])
        assert (info.sweeps, info.backward_error) == (runs[0][0].sweeps, runs[0][0].backward_error)


@pytest.mark.parametrize("d,jx,jt,prec", CASES)
def test_zero_data(d, jx, jt, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    with Solver(_problem(d, jx, jt, 0.0), precision=prec) as s:
        for _ in range(2):
            info = s.solve(0)
            assert info.status == 0 and info.sweeps == 0
            assert not s.coeffs(0).any()
