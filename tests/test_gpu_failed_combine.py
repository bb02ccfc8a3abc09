"""GPU test: st_solve_combine leaves the target alone when a solve fails.

The levels of the combination are queued before the solves that run as graphs have
reported, as st_solve_component followed by st_combine would not do; the target must
stay as it was all the same.  Failures: a NaN source (direct and space-eigenbasis
components; multigrid in graphs), and a sweep limit of one (not converged); target
times up to 11 levels finer than the component's (levels in pairs) and 12 (in FP64).
A good handle afterwards fills its target with what the two calls give.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu

CASES = [("nan", (2, 2, 8), 0, (6, 6), {}), ("nan", (1, 1, 12), 0, (8, 4), {}),
         ("nan", (2, 2, 8), 0, (5, 4), dict(max_direct_rows=500, device_loop=4)),
         ("sweeps", (2, 2, 8), 0, (6, 6), dict(precision=1, max_sweeps=1, tol=1e-15)),
         ("nan", (1, 3, 1), 1, (3, 12), {}), ("nan", (1, 3, 1), 1, (3, 13), {})]


@pytest.mark.parametrize("how,levels,single,target,options", CASES)
def test_target_is_untouched_after_a_failed_solve(how, levels, single, target, options):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver, StError
    d, a, b = levels
    bad = np.nan if how == "nan" else 1.0

    def problem(scale):
        J, mx, mt = (0, a, b) if single else (b - 2 * a, a, a)
        return W.Problem(d=d, lo=(0.0,) * d, hi=(1.0,) * d, T=1.0, J=J, mx=mx, mt=mt,
                         c2=lambda x: 1.0 + 0.5 * (x[:, 0] > 0.4),
                         terms=[(lambda x: scale * np.prod(np.sin(np.pi * x), axis=1), lambda t: np.sin(3 * t))])
    with Solver(problem(bad), **options) as s:
        out = torch.full(((1 << target[1]) + 1, ((1 << target[0]) + 1) ** d), 7.0, dtype=torch.float64, device="cuda")
        for sync in (True, False):
            with pytest.raises(StError):
                s.solve_combine(*target, out=out, sync=sync)
            torch.cuda.synchronize()
            assert bool((out == 7.0).all())
    if how == "nan":
        with Solver(problem(1.0), **options) as s:
            for _ in range(2):
                s.solve_combine(*target, out=out)
            s.solve(-1)
            torch.cuda.synchronize()
            assert torch.equal(out, s.combine(*target))
