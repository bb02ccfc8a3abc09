"""GPU test of nested dissection with many modes on several depths (the leaf size rule
depends on the number of modes): 33 and 65 modes on 15 x 15 and 31 x 31 nodes, 65
on 7^3, against the oracle's exact solve with the tolerances of the parity tests."""
import numpy as np
import pytest

import st_workloads as W
from oracle import solve as osolve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,jx,jt", [(2, 4, 6), (2, 4, 7), (2, 5, 6), (3, 3, 7)])
@pytest.mark.parametrize("prec", [0, 1])
def test_many_modes(d, jx, jt, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    lo, hi = (-0.5, 0.0, 0.25)[:d], (1.5, 0.75, 1.0)[:d]
    p = W.Problem(d=d, lo=lo, hi=hi, T=1.3, J=0, mx=jx, mt=jt,
                  c2=lambda x: 1.0 + 0.5 * np.sin(2 * x[:, 0] + 0.3) + 0.6 * (x[:, -1] > 0.4),
                  u0=lambda x: np.prod(np.sin(np.pi * (x - np.asarray(lo)) / (np.asarray(hi) - np.asarray(lo))), axis=1))
    with Solver(p, precision=prec) as s:
        info = s.component(0)
        assert info.method == 0 and info.n_modes >= 33
        assert s.solve(0).status == 0
        U = s.coeffs(0)
    ref = osolve.solve_component(p, jx, jt, method="schur")
    assert np.linalg.norm(U - ref) / np.linalg.norm(ref) < (1e-10 if prec == 0 else 1e-8)
