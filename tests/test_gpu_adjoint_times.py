"""GPU tests of the receiver misfit and its gradient over target time levels.

Target times coarser and finer than the components' own (the adjoint
right-hand side walks the target times of a row's three intervals), one
receiver and more receivers than a thread block, against the oracle's
gradient with the tolerances of the adjoint parity tests (values 1e-10, J
1e-9, gradients 1e-8 relative).
"""
import numpy as np
import pytest

import st_workloads as W
from oracle import adjoint as OA
from oracle import solve as osolve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jt_star,nrec", [(0, 3), (2, 300), (3, 1), (6, 7), (8, 40)])
def test_gradient_over_target_time_levels(jt_star, nrec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09688_gb300 import ST_FP64
    from paper_2606_09688_gb300.adjoint import nodal_solver
    st = W.inverse_2d(n=6, m=1, jp=3, n_receivers=nrec, seed=2)
    p = OA.with_parameters(st.base, st.c2_nodal, st.g_nodal, st.s, st.jp)
    comps, sols = osolve.solve_all(p, method="schur")
    t, _ = OA.target_times(p, jt_star)
    ref = osolve.combine(p, comps, sols, st.receivers, t)
    d_obs = 0.8 * ref + 1e-3 * np.cos(np.arange(ref.size)).reshape(ref.shape) * np.abs(ref).max()
    J0, gc0, gg0 = OA.gradient(st.base, st.c2_nodal, st.g_nodal, st.s, st.jp, st.receivers, jt_star, d_obs)
    with nodal_solver(st.base, st.c2_nodal, st.g_nodal, st.s, st.jp, ST_FP64) as s:
        s.solve(-1)
        vals = s.receiver_values(jt_star, st.receivers).cpu().numpy()
        J, gc, gg, info = s.misfit_gradient(jt_star, st.receivers, torch.from_numpy(d_obs).cuda(), st.jp)
    assert np.max(np.abs(vals - ref)) <= 1e-10 * np.max(np.abs(ref))
    assert info.status == 0 and abs(J - J0) <= 1e-9 * J0
    gc, gg = gc.cpu().numpy(), gg.cpu().numpy()
    assert np.linalg.norm(gc - gc0) <= 1e-8 * np.linalg.norm(gc0)
    assert np.linalg.norm(gg - gg0) <= 1e-8 * np.linalg.norm(gg0)
