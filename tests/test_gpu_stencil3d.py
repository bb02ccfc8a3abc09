"""GPU test of the plane-streaming 3D stencil kernel (FP32 multigrid levels of 24 or more nodes a side).

One multigrid component on a box with unequal sides and variable c^2: grids of
31 and 63 nodes (one and two tiles of 32 x 8 nodes across, the last one ragged;
chunks of 8 and more planes, the last one shorter), few and many modes.  The FP32
solve with FP64 refinement against the FP64 solve, which runs the general kernel:
1e-8 relative l2 as in the parity tests; a wrong stencil would cost the inner
iteration its convergence, so it may take no more iterations than FP64, whose
inner tolerance is tighter.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jx,jt", [(5, 1), (5, 4), (6, 2)])
def test_fp32_multigrid_component_matches_fp64(jx, jt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    lo, hi = (-0.5, 0.0, 0.25), (1.5, 0.75, 1.0)

    def bump(x):
        s = (x - np.asarray(lo)) / (np.asarray(hi) - np.asarray(lo))
        return np.prod(np.sin(np.pi * s), axis=1) * np.exp(-x[:, 0])
    p = W.Problem(d=3, lo=lo, hi=hi, T=1.3, J=0, mx=jx, mt=jt, u0=bump,
                  c2=lambda x: 1.0 + 0.5 * np.sin(2 * x[:, 0] + 0.3) + 0.6 * (x[:, -1] > 0.4))
    runs = []
    for prec in (0, 1):
        with Solver(p, precision=prec, max_direct_rows=3500) as s:
            runs.append((s.solve(0), s.coeffs(0)))
    (i64, ref), (i32, U) = runs
    assert i64.status == 0 and i32.status == 0 and i32.sweeps <= 4
    assert 0 < i32.max_inner_iters <= i64.max_inner_iters
    assert np.linalg.norm(U - ref) / np.linalg.norm(ref) < 1e-8
