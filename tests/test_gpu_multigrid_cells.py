"""GPU test of multigrid on cells that are not square: plates and oblong boxes.

One component (J = 0) with variable c^2, max_direct_rows small enough for two or
three levels: coarsest grids with an explicit inverse (31 x 31) and by nested
dissection (63 x 63, 15^3), whose modes finish at different iterations.  The
solution against the oracle's exact solve in 2D, with the tolerances of the parity
tests, and by the oracle's normwise backward error in 3D, bound 1e-12 as in the
full-size tests; the iterations may be no more than the damped weights 0.6 (3D
0.55) took on the same problems, which are stable for all of these cells.
"""
import numpy as np
import pytest

import st_workloads as W
from oracle import solve as osolve

pytestmark = pytest.mark.gpu

# sides, (jx, jt), max_direct_rows, iterations with the damped weights in FP64 and FP32
CASES = [((1.5, 1.0), (7, 2), 1000, (15, 5)), ((2.0, 1.0), (7, 2), 1000, (20, 6)),
         ((8.0 / 3.0, 1.0), (7, 2), 1000, (26, 8)), ((8.0 / 3.0, 1.0), (7, 2), 4096, (26, 8)),
         ((4.0, 1.0), (7, 2), 1000, (43, 14)),
         ((1.5, 1.5, 1.0), (5, 1), 3500, (15, 4)), ((2.0, 2.0, 1.0), (5, 1), 3500, (18, 5)),
         ((4.0, 1.0, 1.0), (5, 1), 3500, (45, 13))]


@pytest.mark.parametrize("sides,levels,rows,limits", CASES)
@pytest.mark.parametrize("prec", [0, 1])
def test_oblong_cells_converge(sides, levels, rows, limits, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    d, (jx, jt) = len(sides), levels
    p = W.Problem(d=d, lo=(0.0,) * d, hi=sides, T=1.0, J=0, mx=jx, mt=jt,
                  c2=lambda x: 1.0 + 0.5 * np.sin(2 * x[:, 0] + 0.3) + 0.6 * (x[:, -1] > 0.4),
                  u0=lambda x: np.prod(np.sin(np.pi * x / np.asarray(sides)), axis=1) * np.exp(-x[:, 0]))
    with Solver(p, precision=prec, max_direct_rows=rows) as s:
        info = s.solve(0)
        U = s.coeffs(0)
    assert info.status == 0 and 0 < info.max_inner_iters <= limits[prec]
    if d == 3:
        assert osolve.backward_error(p, jx, jt, U) < 1e-12
        return
    ref = osolve.solve_component(p, jx, jt, method="schur")
    assert np.linalg.norm(U - ref) / np.linalg.norm(ref) < (1e-10 if prec == 0 else 1e-8)
