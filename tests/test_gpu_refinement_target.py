"""GPU test of where the refinement of components with FP32 factors stops.

Grids of 127^2 and 255^2, solved by FP32 factors, against FP64 solves refined as far as
they go (tol = 1e-30).  A backward error at the rounding unit leaves a forward error
of at most 1.8e4 times as much here (255^2, 5 rows, the largest ratio of the two
measured: 9.0e-12 at 6.5e-16), hence 4e-12 relative l2.  The same holds in the
host-driven loop, which the profiled solves take.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jx,jt", [(7, 3), (8, 2), (8, 3)])
@pytest.mark.parametrize("profiled", [False, True])
def test_fp32_factors_refine_to_the_rounding_unit(jx, jt, profiled):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    lo, hi = (-0.5, 0.0), (1.5, 0.75)

    def bump(x):
        s = (x - np.asarray(lo)) / (np.asarray(hi) - np.asarray(lo))
        return np.prod(np.sin(np.pi * s), axis=1) * np.exp(-x[:, 0])
    p = W.Problem(d=2, lo=lo, hi=hi, T=1.3, J=0, mx=jx, mt=jt, u0=bump, v0=lambda x: 0.5 * bump(x) * (x[:, 0] + 0.5),
                  c2=lambda x: 1.0 + 0.5 * np.sin(2 * x[:, 0] + 0.3) + 0.6 * (x[:, -1] > 0.4))
    with Solver(p, tol=1e-30) as s:
        s.solve(0)
        ref = s.coeffs(0)
    with Solver(p, precision=1) as s:
        s.profile(profiled)
        info = s.solve(0)
        U = s.coeffs(0)
    assert info.status == 0 and info.backward_error <= 2.0 ** -52
    assert np.linalg.norm(U - ref) / np.linalg.norm(ref) < 4e-12
