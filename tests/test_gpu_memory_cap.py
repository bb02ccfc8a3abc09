"""GPU test of calls that run out of memory half way and are repeated.

A handle with a memory cap; receiver tables of growing sets take up what it leaves, from
all but a few kilobytes down in steps smaller than the arrays that combine() and
misfit_gradient() take on their first call: each of them either works or is refused
(ST_ERR_OOM) each time, and what works gives the bits of a handle without a cap.
"""
import numpy as np
import pytest

import st_workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _sweep(make, call, step):
    """call(solver) with less and less of the cap taken up, until it works; its results and the number of refusals."""
    from paper_2606_09688_gb300 import StError
    from paper_2606_09688_gb300 import st as B

    def filled(n):
        s = make()
        s.solve(-1)
        try:
            s.receiver_values(0, np.full((n, 2), 0.37))
        except StError as e:
            assert e.code == B.ST_ERR_OOM
            s.close()
            return None
        return s
    lo, hi = 1, 1 << 20
    while hi - lo > 1:
        mid = (lo + hi) // 2
        s = filled(mid)
        lo, hi = (lo, mid) if s is None else (mid, hi)
        if s is not None:
            s.close()
    refusals = 0
    for n in range(lo, lo - 400 * step, -step):
        with filled(n) as s:
            results = []
            for _ in range(3):
                try:
                    results.append(call(s))
                except StError as e:
                    assert e.code == B.ST_ERR_OOM
        if len(results) == 3:
            return results, refusals
        refusals += 1
        assert not results
    raise AssertionError("never enough")


def test_combine_is_refused_or_works(torch):
    from paper_2606_09688_gb300 import Solver
    p = W.standing_wave(2, 8, 2)   # with a lift, whose pairs are a third array per component
    with Solver(p) as s:
        s.solve(-1)
        ref = s.combine(5, 4)
    results, refusals = _sweep(lambda: Solver(p, mem_cap_bytes=128 << 20), lambda s: s.combine(5, 4).clone(), 40)
    assert refusals >= 4
    for out in results:
        assert torch.equal(out, ref)


def test_misfit_gradient_is_refused_or_works(torch):
    from paper_2606_09688_gb300.st import Solver
    from paper_2606_09688_gb300.adjoint import problem_with
    su = W.inverse_2d(6, 2, jp=3, n_receivers=5)
    obs = torch.zeros((1 << su.jt_star) + 1, 5, dtype=torch.float64, device="cuda")

    def make():
        return Solver(problem_with(su.base, su.s), c2_nodal=su.c2_nodal, g_nodal=su.g_nodal, param_level=3,
                      mem_cap_bytes=16 << 20)
    results, refusals = _sweep(make, lambda s: s.misfit_gradient(su.jt_star, su.receivers, obs, 3)[0], 5)
    assert refusals >= 4 and np.isfinite(results[0]) and results[0] > 0 and len(set(results)) == 1


def _pool_high(reset=False):
    """Most memory that the device's default pool has held since the last reset."""
    import ctypes
    cu = ctypes.CDLL("libcuda.so.1")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    reserved_high = 6
    if reset:
        assert cu.cuMemPoolSetAttribute(pool, reserved_high, ctypes.byref(v)) == 0
    assert cu.cuMemPoolGetAttribute(pool, reserved_high, ctypes.byref(v)) == 0
    return v.value


def test_set_up_under_a_cap_holds_one_workspace_at_a_time(torch):
    """The factorisation's workspaces are not part of the handle's memory, so the cap covers
    the largest of them, not their sum: a set-up of all components takes no more from the
    pool than the largest one alone (64 MB: twice the pool's granularity)."""
    import dataclasses

    from paper_2606_09688_gb300 import Solver
    p = W.layered_2d(11, 2)

    def high(q):
        torch.cuda.synchronize()
        _pool_high(reset=True)
        with Solver(q, mem_cap_bytes=64 << 30) as s:
            comps = [(c.jx, c.jt) for c in s.components()]
        return _pool_high(), comps
    total, comps = high(p)
    single = max(high(dataclasses.replace(p, J=0, mx=jx, mt=jt))[0] for jx, jt in comps if jx in (7, 8))
    assert single > 256 << 20
    assert total <= single + (64 << 20), (total >> 20, single >> 20)
