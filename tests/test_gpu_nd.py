"""GPU tests of the nested dissection solves of the spatial problems.

One component per problem (J = 0) on boxes with unequal sides and variable c^2,
against the oracle's exact solve of the same system: grids of one leaf (1 to 9
nodes), fronts that touch every, some and no side of the grid, separators
around the 32-row task and 32-pivot block (31, 63 and 127 nodes; 49 and 225 in
3D), few and many modes (leaf size rule), both precisions.  Tolerances: those of
the parity tests, 1e-10 (FP64) and 1e-8 (FP32 with FP64 refinement) relative l2;
refinement converges within three sweeps (a wrong factor would need more).
"""
import numpy as np
import pytest

import st_workloads as W
from oracle import solve as osolve

pytestmark = pytest.mark.gpu


def _problem(d, jx, jt):
    lo, hi = (-0.5, 0.0, 0.25)[:d], (1.5, 0.75, 1.0)[:d]

    def c2(x):
        return 1.0 + 0.5 * np.sin(2 * x[:, 0] + 0.3) + 0.6 * (x[:, -1] > 0.4)

    def bump(x):
        s = (x - np.asarray(lo)) / (np.asarray(hi) - np.asarray(lo))
        return np.prod(np.sin(np.pi * s), axis=1) * np.exp(-x[:, 0])
    return W.Problem(d=d, lo=lo, hi=hi, T=1.3, c2=c2, J=0, mx=jx, mt=jt, u0=bump,
                     v0=lambda x: 0.5 * bump(x) * (x[:, 0] + 0.5))


CASES = [(1, 1, 3), (1, 2, 4), (1, 5, 6), (1, 8, 2), (1, 11, 2), (2, 1, 4), (2, 2, 5), (2, 3, 3), (2, 4, 2), (2, 5, 3),
         (2, 6, 1), (2, 7, 1), (3, 1, 4), (3, 2, 2), (3, 3, 2), (3, 4, 1)]


@pytest.mark.parametrize("d,jx,jt", CASES)
@pytest.mark.parametrize("prec", [0, 1])
def test_direct_component_matches_the_oracle(d, jx, jt, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    p = _problem(d, jx, jt)
    with Solver(p, precision=prec) as s:
        info = s.solve(0)
        U = s.coeffs(0)
    ref = osolve.solve_component(p, jx, jt, method="schur")
    assert np.linalg.norm(U - ref) / np.linalg.norm(ref) < (1e-10 if prec == 0 else 1e-8)
    assert info.status == 0 and info.sweeps <= 3


def test_many_modes_and_one_node_per_leaf():
    """65 modes on 15 x 15 nodes (the rule takes small leaves) and 5 on 63 x 63, through one combination."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    p = W.anisotropic_2d(8, 2)
    with Solver(p) as s:
        s.solve(-1)
        for k, info in enumerate(s.components()):
            ref = osolve.solve_component(p, info.jx, info.jt, method="schur")
            assert np.linalg.norm(s.coeffs(k) - ref) / np.linalg.norm(ref) < 1e-10


@pytest.mark.parametrize("jx,jt", [(17, 1), (17, 3), (14, 6)])
def test_long_grids_backward_error(jx, jt):
    """131071 nodes with 3 and 9 time rows (time transforms with a thread per node, all outputs in one
    pass) and 16383 with 65 (transforms with split inputs, several time chunks of the residual): the oracle's
    own normwise backward error, bound 1e-12 as in the full-size tests."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import Solver
    p = _problem(1, jx, jt)
    with Solver(p) as s:
        assert s.solve(0).status == 0
        U = s.coeffs(0)
    assert osolve.backward_error(p, jx, jt, U) < 1e-12
