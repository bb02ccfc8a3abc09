"""Performance cases of the space-time sparse-grid wave solver.

Each case is one call sequence that a program using the library makes, through
its public entry points (Solver.solve_combine, Solver.solve and
misfit_gradient, Solver.energy, solve_batch and combine, receiver_misfit with
its backward pass), on a problem instance drawn from a seed:

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the problem instance, its Solver and output buffers
    run(state)           one pass
    work(case)           bytes and flops that a pass cannot do without
    exact(case, seed)    the same outputs from plain torch in 64 bits

Levels follow the library: components (m + a, n - m - a) with +1 and
(m + a - 1, n - m - a) with -1, level j meaning 2^j cells per direction in space
or 2^j intervals in time, Q1 elements x C^1 quadratic splines.
"""
import dataclasses
import math
from typing import Any

import numpy as np
import torch

from paper_2606_09688_gb300 import ST_FP32_IR, ST_FP64, Solver, solve_batch
from paper_2606_09688_gb300.adjoint import nodal_solver, receiver_misfit

PRECISION = {"fp64": ST_FP64, "fp32ir": ST_FP32_IR}


@dataclasses.dataclass
class Problem:
    """One instance of the wave problem, with the fields that Solver reads."""
    d: int
    lo: tuple
    hi: tuple
    T: float
    c2: Any
    J: int
    mx: int
    mt: int
    terms: list = dataclasses.field(default_factory=list)
    f_general: Any = None
    u0: Any = None
    v0: Any = None
    layers: Any = None   # (y, c^2 below, c^2 above) where c^2 depends on y alone


# ------------------------------------------------------------------- cases
def _combine(name, medium, d, n, m, precision, jx, jt, T=1.0, fp=8.0):
    c = dict(kind="combine", medium=medium, d=d, n=n, m=m, precision=precision, jx=jx, jt=jt, T=T, fp=fp)
    return dict(name=name, **c) if name else c


def _energy(name, medium, d, n, m, precision, times, T=1.0, fp=8.0):
    c = dict(kind="energy", medium=medium, d=d, n=n, m=m, precision=precision, times=times, T=T, fp=fp)
    return dict(name=name, **c) if name else c


def _gradient(name, kind, n, m, precision, jp, receivers, jt, T=1.0, fp=8.0):
    c = dict(kind=kind, medium="nodal", d=2, n=n, m=m, precision=precision, jp=jp, receivers=receivers, jt=jt, T=T,
             fp=fp)
    return dict(name=name, **c) if name else c


def _batch(name, levels, m, precision, T=1.0, fp=8.0):
    c = dict(kind="batch", medium="jump", d=2, levels=",".join(str(n) for n in levels), m=m, precision=precision,
             T=T, fp=fp)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a 1D string with nine components of at most 31 x 33 unknowns, solved and combined
        # (a convergence table, a unit test, the inner call of a parameter scan): latency and launches
        _combine("string_1d_n6_fp64", "standing", 1, 6, 1, "fp64", 5, 5),
        # a travelling pulse on a string with its energy at 800 instants, as in an energy-conservation study
        _energy("energy_1d_n13_fp64", "travelling", 1, 13, 3, "fp64", 800),
        # ordinary 2D runs through a two-layer medium with a Ricker source, the whole field delivered
        _combine("layered_2d_n8_fp32ir", "layered", 2, 8, 2, "fp32ir", 6, 6),
        _combine("layered_2d_n10_fp64", "layered", 2, 10, 2, "fp64", 8, 8),
        # a non-square box, T = 1.7, initial data, a target that is finer in time than in space (odd shape)
        _combine("box_2d_n9_fp64", "box", 2, 9, 2, "fp64", 6, 8, T=1.7, fp=3.0),
        # the full-size 2D run of the benchmark in both precisions: 12.1 M unknowns, 8.6 GB of field values
        _combine("layered_2d_n12_fp64", "layered", 2, 12, 2, "fp64", 10, 10),
        _combine("layered_2d_n12_fp32ir", "layered", 2, 12, 2, "fp32ir", 10, 10),
        # a 3D random medium: the small grid (every component solved directly), and the benchmark's 26.8 M unknowns
        _combine("random_3d_n7_fp64", "random", 3, 7, 3, "fp64", 4, 4),
        _combine("random_3d_n10_fp32ir", "random", 3, 10, 3, "fp32ir", 7, 7),
        # forward and adjoint solves on one handle: the receiver misfit's gradient of the differentiation study
        _gradient("gradient_2d_n10_fp64", "gradient", 10, 2, "fp64", 6, 32, 8),
        # one step of an inversion through autograd: new parameters every call, so the set-up belongs to the pass
        _gradient("inversion_2d_n8_fp32ir", "inversion", 8, 2, "fp32ir", 5, 24, 6),
        # many instances together (an ensemble of media), each field collected as 17 snapshots
        _batch("ensemble_2d_fp32ir", [11, 8, 9, 10, 8, 9, 10, 11, 9, 8, 10, 9], 2, "fp32ir"),
    ]


def draw(rng):
    pr = rng.choice(["fp64", "fp32ir"])
    T = round(rng.uniform(0.9, 1.7), 3)
    fp = round(rng.uniform(3.0, 8.0), 2)
    u = rng.random()
    if u < 0.12:
        n = rng.randint(4, 10)
        return _combine("", rng.choice(["standing", "travelling"]), 1, n, 1, pr, rng.randint(max(1, n - 3), n),
                        rng.randint(max(1, n - 3), n), T, fp)
    if u < 0.55:
        n = rng.randint(6, 11)
        return _combine("", rng.choice(["layered", "layered", "box"]) if n < 11 else "layered", 2, n, 2, pr,
                        n - 2 - rng.randint(0, 2), n - 2 - rng.randint(-1 if n < 10 else 0, 2), T, fp)
    if u < 0.7:
        n = rng.randint(7, 9)
        return _combine("", "random", 3, n, 3, pr, n - 3 - rng.randint(0, 1), n - 3 - rng.randint(-1, 2), T, fp)
    if u < 0.78:
        if rng.random() < 0.5:
            n = rng.randint(6, 13)
            return _energy("", "travelling", 1, n, rng.randint(1, 3) if n < 11 else 3, pr, rng.randint(101, 901), T, fp)
        return _energy("", "layered", 2, rng.randint(6, 9), 2, pr, rng.randint(33, 201), T, fp)
    if u < 0.92:
        n = rng.randint(6, 10)
        kind = "gradient" if n > 8 else rng.choice(["gradient", "inversion"])
        return _gradient("", kind, n, 2, pr, rng.randint(3, 6), rng.randint(5, 48), n - 2 - rng.randint(0, 1), T, fp)
    return _batch("", [rng.randint(7, 10) for _ in range(rng.randint(3, 11))], 2, pr, T, fp)


# ------------------------------------------------------------- the problems
def _gaussian(centre, sigma):
    c = np.asarray(centre)
    return lambda x: np.exp(-np.sum((x - c) ** 2, axis=1) / (2.0 * sigma * sigma))


def _ricker(fp):
    def s(t):
        a = (np.pi * fp * (np.asarray(t) - 1.0 / fp)) ** 2
        return (1.0 - 2.0 * a) * np.exp(-a)
    return s


def _fourier(rng, d, modes, amp, kmax):
    kap = rng.integers(-kmax, kmax + 1, size=(modes, d)).astype(np.float64)
    kap[np.all(kap == 0, axis=1), 0] = 1.0
    a, ph = rng.normal(0.0, amp, size=modes), rng.uniform(0.0, 2.0 * np.pi, size=modes)

    def g(x):
        out = np.zeros(len(x))
        for k in range(modes):
            arg = np.full(len(x), ph[k])
            for j in range(d):
                if kap[k, j] != 0.0:
                    arg += (2.0 * np.pi * kap[k, j]) * x[:, j]
            out += a[k] * np.cos(arg)
        return out
    return g


def _prod_sin(x):
    return np.prod(np.sin(np.pi * x), axis=1)


def problem(case, seed, n=None, item=0):
    """The instance of a case: the medium and data of its kind, with what a user varies drawn from the seed."""
    rng = np.random.default_rng([int(seed) & 0x7fffffff, item])
    d, m, T, fp = case["d"], case["m"], case["T"], case["fp"]
    n = case["n"] if n is None else n
    lev = dict(J=n - 2 * m, mx=m, mt=m)
    unit = dict(d=d, lo=(0.0,) * d, hi=(1.0,) * d, T=T)
    med = case["medium"]
    if med == "standing":  # the first string modes with random amplitudes, at rest
        a = rng.uniform(0.2, 1.0, size=3)

        def u0(x):
            return sum(a[k] * np.sin((k + 1) * np.pi * x[:, 0]) for k in range(3))
        return Problem(**unit, c2=lambda x: np.ones(len(x)), u0=u0, **lev)
    if med == "travelling":  # a pulse moving right on (-1, 1), reflected at x = 1
        c, x0, w = 0.8, rng.uniform(0.45, 0.6), rng.uniform(14.0, 18.0)

        def g(s):
            return np.exp(-w * (s - x0) ** 2)

        def dg(s):
            return -2.0 * w * (s - x0) * g(s)
        return Problem(d=1, lo=(-1.0,), hi=(1.0,), T=T, c2=lambda x: np.full(len(x), c * c),
                       u0=lambda x: g(x[:, 0]) - g(2.0 - x[:, 0]),
                       v0=lambda x: -c * dg(x[:, 0]) + c * dg(2.0 - x[:, 0]), **lev)
    if med == "layered":  # c^2 1 below and 3..4 above an interface, a point-like source
        y, top = rng.uniform(0.4, 0.6), rng.uniform(3.0, 4.0)
        src = _gaussian(rng.uniform(0.25, 0.75, size=2), 0.05)
        return Problem(**unit, c2=lambda x: np.where(x[:, 1] < y, 1.0, top), terms=[(src, _ricker(fp))],
                       layers=(y, 1.0, top), **lev)
    if med == "box":  # cells 2.67 times wider than tall, smooth and jumping c^2, initial data and a source
        lo, hi = np.array((-0.5, 0.0)), np.array((1.5, 0.75))
        ph, q = rng.uniform(0.0, 1.0), rng.uniform(0.6, 0.8)

        def bump(x):
            return np.prod(np.sin(np.pi * (x - lo) / (hi - lo)), axis=1) * np.exp(-((x[:, 0] - 0.3) ** 2))
        return Problem(d=2, lo=tuple(lo), hi=tuple(hi), T=T,
                       c2=lambda x: 1.0 + 0.5 * np.sin(2 * x[:, 0] + ph) * np.cos(3 * x[:, 1]) + q * (x[:, 1] > 0.4),
                       terms=[(_gaussian((0.3 + ph, 0.3), 0.1), _ricker(fp))], u0=bump,
                       v0=lambda x: 0.5 * bump(x) * (x[:, 0] + 0.5), **lev)
    if med == "random":  # a 16-mode random medium
        g = _fourier(rng, d, 16, 0.35, 4)
        return Problem(**unit, c2=lambda x: np.clip(np.exp(g(x)), 0.25, 4.0), u0=_prod_sin, **lev)
    if med == "jump":  # a smooth random medium with a jump, a source at a random place
        g, y, up = _fourier(rng, d, 8, 0.25, 3), rng.uniform(0.3, 0.7), rng.uniform(1.0, 1.6)
        src = _gaussian(rng.uniform(0.2, 0.8, size=2), 0.05)
        return Problem(**unit, c2=lambda x: np.clip(np.clip(np.exp(g(x)), 0.5, 2.0) * np.where(x[:, 1] < y, 1.0, up),
                                                    0.5, 2.0), terms=[(src, _ricker(fp))], **lev)
    # "nodal": c^2 and the source's factor as nodal fields, given beside the problem
    return Problem(**unit, c2=lambda x: np.ones(len(x)), **lev)


def inverse_data(case, seed):
    """Nodal c^2 and source factor on the level-jp grid, receivers on a line, and recorded traces."""
    rng = np.random.default_rng(int(seed) & 0x7fffffff)
    ax = np.linspace(0.0, 1.0, (1 << case["jp"]) + 1)
    x = np.stack([np.tile(ax, len(ax)), np.repeat(ax, len(ax))], axis=1)
    c2 = 0.5 + 0.75 * (1.0 + np.tanh(_fourier(rng, 2, 6, 1.0, 2)(x)))
    centre = rng.uniform(0.25, 0.75, size=2)
    g = _gaussian(centre, 0.05 if case["jp"] > 4 else 0.12)(x)
    nr = case["receivers"]
    rec = np.stack([(np.arange(nr) + 0.5) / nr, np.full(nr, 0.9)], axis=1)
    t = np.linspace(0.0, case["T"], (1 << case["jt"]) + 1)
    delay = np.hypot(rec[:, 0] - centre[0], rec[:, 1] - centre[1]) / rng.uniform(0.9, 1.2)
    obs = 1e-3 * _ricker(case["fp"])(t[:, None] - delay[None, :]) / (0.2 + delay[None, :])
    return c2, g, rec, obs


# ------------------------------------------------------------ prepare, run
def prepare(case, seed):
    prec = PRECISION[case["precision"]]
    kind = case["kind"]
    st = dict(case=case)
    if kind == "combine":
        p = problem(case, seed)
        st["solver"] = Solver(p, precision=prec)
        nodes = ((1 << case["jx"]) + 1) ** case["d"]
        st["out"] = torch.empty(((1 << case["jt"]) + 1, nodes), dtype=torch.float64, device="cuda")
    elif kind == "energy":
        p = problem(case, seed)
        st["solver"] = Solver(p, precision=prec)
        st["times"] = _instants(case)
    elif kind == "gradient":
        c2, g, rec, obs = inverse_data(case, seed)
        st["solver"] = nodal_solver(problem(case, seed), c2, g, _ricker(case["fp"]), case["jp"], prec)
        st["receivers"], st["obs"] = rec, torch.from_numpy(obs).cuda()
    elif kind == "inversion":
        c2, g, rec, obs = inverse_data(case, seed)
        st["base"], st["s"] = problem(case, seed), _ricker(case["fp"])
        st["receivers"], st["obs"] = rec, torch.from_numpy(obs).cuda()
        st["c2"] = torch.from_numpy(c2).cuda().requires_grad_(True)
        st["g"] = torch.from_numpy(g).cuda().requires_grad_(True)
    else:  # batch: the solves of an ensemble as graphs, which is the library's setting for it
        levels = [int(v) for v in case["levels"].split(",")]
        st["solvers"] = [Solver(problem(case, seed, n, i), precision=prec, device_loop=4)
                         for i, n in enumerate(levels)]
        st["targets"] = [(n - case["m"] - 1, 4) for n in levels]
        st["outs"] = [torch.empty((17, ((1 << jx) + 1) ** 2), dtype=torch.float64, device="cuda")
                      for jx, _ in st["targets"]]
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "combine":
        out, _ = state["solver"].solve_combine(case["jx"], case["jt"], state["out"], sync=False)
        return out
    if kind == "energy":
        state["solver"].solve(-1, sync=False)
        return state["solver"].energy(state["times"])
    if kind == "gradient":
        s = state["solver"]
        s.solve(-1, sync=False)
        J, dc2, dg, _ = s.misfit_gradient(case["jt"], state["receivers"], state["obs"], case["jp"])
        return dict(J=J, dc2=dc2, dg=dg)
    if kind == "inversion":
        c2, g = state["c2"], state["g"]
        c2.grad = g.grad = None
        J = receiver_misfit(c2, g, state["base"], state["s"], case["jp"], state["receivers"], case["jt"],
                            state["obs"], PRECISION[case["precision"]])
        J.backward()
        return dict(J=J.detach(), dc2=c2.grad, dg=g.grad)
    solve_batch(state["solvers"], sync=False)
    return [s.combine(jx, jt, out) for s, (jx, jt), out in zip(state["solvers"], state["targets"], state["outs"])]


def _instants(case):
    k = case["times"]
    return case["T"] * (np.arange(k) + 0.5) / k


# -------------------------------------------------------------------- work
def _components(n, m):
    J = n - 2 * m
    return [(m + a, m + J - a, 1) for a in range(J + 1)] + [(m + a - 1, m + J - a, -1) for a in range(1, J + 1)]


def work(case):
    """Per component: c^2 read, the right-hand side read and the solution written once, and one application of the
    space-time operator; per pass: the field, energies or gradients written once."""
    d, m = case["d"], case["m"]
    levels = [int(v) for v in case["levels"].split(",")] if case["kind"] == "batch" else [case["n"]]
    solves = 2 if case["kind"] in ("gradient", "inversion") else 1
    b = f = 0.0
    for n in levels:
        for jx, jt, _ in _components(n, m):
            dofs = ((1 << jx) - 1.0) ** d * ((1 << jt) + 1)
            b += solves * (16.0 * dofs + 8.0 * (1 << jx) ** d)
            f += solves * dofs * (4.0 * 3 ** d + 20.0)
    if case["kind"] == "combine":
        out = ((1 << case["jx"]) + 1.0) ** d * ((1 << case["jt"]) + 1)
    elif case["kind"] == "energy":
        out = case["times"]
        f += out * 30.0 * (1 << (case["n"] - m)) ** d
    elif case["kind"] == "batch":
        out = sum(17.0 * ((1 << (n - m - 1)) + 1) ** 2 for n in levels)
    else:
        out = 2.0 * ((1 << case["jp"]) + 1) ** 2
    return {"bytes": b + 8.0 * out, "flops": f + 7.0 * out}


# ------------------------------------------------------------------- exact
# The same discretisation in plain torch: quadratic B-splines and 8-point
# Gauss-Legendre in time, Q1 elements in space, and each component's system
# A (x) M + B (x) K solved through the spatial eigenbasis (dense) or, where c^2
# depends on y alone, through the sine basis in x and block elimination in y.
F64 = torch.float64


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=F64, device=_dev())


def _splines(t, N, T):
    """Values, first and second derivatives of the basis (the first B-spline removed) at times t, (len(t), N + 1)."""
    t = np.asarray(t, dtype=np.float64)
    h = T / N
    k = np.clip(np.floor(t / h).astype(int), 0, N - 1)
    kn = lambda i: np.clip(i, 0, N) * h  # noqa: E731
    a, b, c, d = kn(k - 1), kn(k), kn(k + 1), kn(k + 2)
    left, right = (c - t) / (c - b), (t - b) / (c - b)
    v = [(c - t) / (c - a) * left, (t - a) / (c - a) * left + (d - t) / (d - b) * right, (t - b) / (d - b) * right]
    v1 = [-2 / (c - a) * left, 2 / (c - a) * left - 2 / (d - b) * right, 2 / (d - b) * right]
    e0, e2 = 2 / ((c - a) * (c - b)), 2 / ((d - b) * (c - b))
    v2 = [e0, -(e0 + e2), e2]
    out = np.zeros((3, len(t), N + 2))
    for j, vs in enumerate((v, v1, v2)):
        for s in range(3):
            out[j, np.arange(len(t)), k + s] = vs[s]
    return [_t(o[:, 1:]) for o in out]


def _time_system(jt, T):
    """A, B, the quadrature times, Q (nt x nq) with (s, psi_i')_e = Q s, psi_i'(0) and (1, psi_i')_e."""
    N = 1 << jt
    x, w = np.polynomial.legendre.leggauss(8)
    h = T / N
    t = (np.arange(N)[:, None] * h + (x[None, :] + 1.0) * 0.5 * h).ravel()
    P, P1, P2 = _splines(t, N, T)
    we = _t(np.tile(w * 0.5 * h, N) * np.exp(-t / T))
    d0 = _splines([0.0], N, T)[1][0]
    Q = (P1 * we[:, None]).T.contiguous()
    return Q @ P2 + torch.outer(d0, d0), Q @ P, t, Q, d0, Q @ torch.ones_like(we)


def _nodes(p, j):
    ax = [p.lo[k] + (p.hi[k] - p.lo[k]) / (1 << j) * np.arange((1 << j) + 1) for k in range(p.d)]
    return np.stack([g.ravel() for g in np.meshgrid(*ax[::-1], indexing="ij")[::-1]], axis=1)


def _centres(p, j):
    ax = [p.lo[k] + (p.hi[k] - p.lo[k]) / (1 << j) * (np.arange(1 << j) + 0.5) for k in range(p.d)]
    return np.stack([g.ravel() for g in np.meshgrid(*ax[::-1], indexing="ij")[::-1]], axis=1)


def _widths(p, j):
    return [(p.hi[k] - p.lo[k]) / (1 << j) for k in range(p.d)]


def _elements(p, j):
    """Element mass and stiffness, and the node of each corner of each cell (all nodes, x fastest)."""
    h, nc = _widths(p, j), 1 << p.d
    bit = lambda a, k: (a >> k) & 1  # noqa: E731
    M, K = np.zeros((nc, nc)), np.zeros((nc, nc))
    for a in range(nc):
        for b in range(nc):
            m1 = [h[k] / 6.0 * (2.0 if bit(a, k) == bit(b, k) else 1.0) for k in range(p.d)]
            k1 = [(1.0 if bit(a, k) == bit(b, k) else -1.0) / h[k] for k in range(p.d)]
            M[a, b] = np.prod(m1)
            K[a, b] = sum(k1[k] * np.prod(m1[:k] + m1[k + 1:]) for k in range(p.d))
    N = 1 << j
    ids = np.indices((N,) * p.d).reshape(p.d, -1)[::-1]
    corner = np.stack([sum((ids[k] + bit(c, k)) * (N + 1) ** k for k in range(p.d)) for c in range(nc)], axis=1)
    return _t(M), _t(K), torch.as_tensor(corner, device=_dev())


def _inner(p, j):
    N = 1 << j
    ids = np.indices((N + 1,) * p.d).reshape(p.d, -1)
    return torch.as_tensor(np.nonzero(np.all((ids > 0) & (ids < N), axis=0))[0], device=_dev())


def _apply(E, corner, x, scale=None):
    """Sum of element matrices times x (rows of values on all nodes)."""
    y = x[:, corner] @ E
    if scale is not None:
        y = y * scale[None, :, None]
    out = torch.zeros_like(x)
    return out.index_add_(1, corner.reshape(-1), y.reshape(x.shape[0], -1))


class _Dense:
    """The spatial eigenbasis of each level of a problem."""

    def __init__(self, p, c2=None, g=None):
        self.p, self.c2, self.g, self.level = p, c2 or p.c2, g, {}

    def space(self, j):
        if j not in self.level:
            p = self.p
            Me, Ke, corner = _elements(p, j)
            inner = _inner(p, j)
            c2 = _t(self.c2(_centres(p, j)))
            na = ((1 << j) + 1) ** p.d
            nc = 1 << p.d
            at = (corner[:, :, None] * na + corner[:, None, :]).reshape(-1)
            full = [torch.zeros(na * na, dtype=F64, device=_dev()).index_add_(0, at, v.reshape(-1)).view(na, na)[inner][:, inner]
                    for v in (Me.expand(len(corner), nc, nc), c2[:, None, None] * Ke)]
            L = torch.linalg.cholesky(full[0])
            C = torch.linalg.solve_triangular(L, full[1], upper=False)
            C = torch.linalg.solve_triangular(L, C.T.contiguous(), upper=False)
            del full
            mu, V = torch.linalg.eigh(0.5 * (C + C.T))
            self.level[j] = (Me, Ke, corner, inner, c2, mu, torch.linalg.solve_triangular(L.T, V, upper=True))
        return self.level[j]

    def rhs(self, jx, jt):
        p = self.p
        Me, Ke, corner, inner, c2, _, _ = self.space(jx)
        _, _, tq, Q, d0, one = _time_system(jt, p.T)
        x = _nodes(p, jx)
        F = torch.zeros((len(d0), len(inner)), dtype=F64, device=_dev())
        for r, (g, s) in enumerate(p.terms):
            gv = (self.g if r == 0 and self.g is not None else g)(x)
            F += torch.outer(Q @ _t(s(tq)), _apply(Me, corner, _t(gv)[None])[0, inner])
        if p.v0 is not None:
            F += torch.outer(d0, _apply(Me, corner, _t(p.v0(x))[None])[0, inner])
        if p.u0 is not None:
            F -= torch.outer(one, _apply(Ke, corner, _t(p.u0(x))[None], c2)[0, inner])
        return F

    def solve(self, jx, jt, F=None, transposed=False):
        mu, Phi = self.space(jx)[5:]
        A, B = _time_system(jt, self.p.T)[:2]
        if transposed:
            A, B = A.T, B.T
        F = self.rhs(jx, jt) if F is None else F
        Y = (F @ Phi).T.contiguous()
        C = torch.empty_like(Y)
        step = max(1, (1 << 27) // (len(A) ** 2))
        for a in range(0, len(mu), step):
            S = A[None] + mu[a:a + step, None, None] * B[None]
            C[a:a + step] = torch.linalg.solve(S, Y[a:a + step, :, None])[:, :, 0]
        return C.T @ Phi.T


class _Layered:
    """c^2(y): sine basis in x, block elimination along y (blocks in time), all sine modes together."""

    def __init__(self, p):
        self.p = p

    def solve(self, jx, jt):
        p = self.p
        N = 1 << jx
        hx, hy = _widths(p, jx)
        A, B, tq, Q, _, _ = _time_system(jt, p.T)
        c2 = _t(p.c2(np.stack([np.full(N, 0.5), p.lo[1] + hy * (np.arange(N) + 0.5)], axis=1)))
        th = torch.arange(1, N, dtype=F64, device=_dev()) * (math.pi / N)
        S = math.sqrt(2.0 / N) * torch.sin(torch.outer(torch.arange(1, N, dtype=F64, device=_dev()), th))
        mx, kx = hx / 6.0 * (4.0 + 2.0 * torch.cos(th)), (2.0 - 2.0 * torch.cos(th)) / hx
        my, mc = torch.full((N - 1,), 4.0 * hy / 6.0, dtype=F64, device=_dev()), hy / 3.0 * (c2[:-1] + c2[1:])
        kc = (c2[:-1] + c2[1:]) / hy
        myo, mco, kco = hy / 6.0, hy / 6.0 * c2[1:-1], -c2[1:-1] / hy
        b = torch.stack([Q @ _t(s(tq)) for _, s in p.terms])
        x = _nodes(p, jx)
        loads = []
        for g, _ in p.terms:
            v = _t(g(x)).view(N + 1, N + 1)
            v = hx / 6.0 * (v[:, :-2] + 4.0 * v[:, 1:-1] + v[:, 2:])
            loads.append(hy / 6.0 * (v[:-2] + 4.0 * v[1:-1] + v[2:]) @ S)
        loads = torch.stack(loads)                                     # term, y, sine mode
        nt, n = len(A), N - 1
        X = torch.empty((n, n, nt, nt), dtype=F64, device=_dev()) if n > 1 else None
        y = torch.empty((n, n, nt), dtype=F64, device=_dev())
        D = prev = None
        for a in range(n):
            new = (mx * my[a])[:, None, None] * A + (kx * mc[a] + mx * kc[a])[:, None, None] * B
            f = torch.einsum("ri,rp->pi", b, loads[:, a])
            if prev is not None:
                new = new - prev @ X[a - 1]
                f = f - (prev @ y[a - 1][:, :, None])[:, :, 0]
            D = new
            if a + 1 < n:
                prev = (mx * myo)[:, None, None] * A + (kx * mco[a] + mx * kco[a])[:, None, None] * B
                sol = torch.linalg.solve(D, torch.cat([prev, f[:, :, None]], dim=2))
                X[a], y[a] = sol[:, :, :nt], sol[:, :, nt]
            else:
                y[a] = torch.linalg.solve(D, f[:, :, None])[:, :, 0]
        for a in range(n - 2, -1, -1):
            y[a] -= (X[a] @ y[a + 1][:, :, None])[:, :, 0]
        del X
        U = torch.einsum("ypi,px->iyx", y, S)
        return U.reshape(nt, -1)


def _solver64(p):
    """A solver for the problem's components, or None where the dense one would take too long."""
    if p.layers is not None and p.u0 is None and p.v0 is None:
        return _Layered(p)
    return _Dense(p) if ((1 << (p.mx + p.J)) - 1) ** p.d <= 4100 else None


def _refine(v, d):
    """Nodal values of a level to the next finer one (rows of (N + 1)^d values)."""
    N = round(v.shape[1] ** (1.0 / d)) - 1
    v = v.view((v.shape[0],) + (N + 1,) * d)
    for k in range(1, d + 1):
        s = list(v.shape)
        s[k] = 2 * N + 1
        w = torch.empty(s, dtype=v.dtype, device=v.device)
        w.narrow(k, 0, 2 * N + 1)[(slice(None),) * k + (slice(0, None, 2),)] = v
        w[(slice(None),) * k + (slice(1, None, 2),)] = 0.5 * (v.narrow(k, 0, N) + v.narrow(k, 1, N))
        v = w
    return v.reshape(v.shape[0], -1)


def _field(p, sols, times, jx_star, deriv=0):
    """The combined solution (or its time derivative) on all nodes of level jx_star at the times."""
    acc = None
    finest = max(c[0] for c in sols)
    for j in range(min(min(c[0] for c in sols), jx_star), max(finest, jx_star) + 1):
        if acc is not None and j <= jx_star:
            acc = _refine(acc, p.d)
        for (jx, jt, coef), U in sols.items():
            if jx != j:
                continue
            full = torch.zeros((len(times), ((1 << jx) + 1) ** p.d), dtype=F64, device=_dev())
            full[:, _inner(p, jx)] = _splines(times, 1 << jt, p.T)[deriv] @ U
            if deriv == 0 and p.u0 is not None:
                full += _t(p.u0(_nodes(p, jx)))[None]
            if jx > jx_star:  # by injection
                s = 1 << (jx - jx_star)
                full = full.view((len(times),) + ((1 << jx) + 1,) * p.d)
                full = full[(slice(None),) + (slice(None, None, s),) * p.d].reshape(len(times), -1)
            acc = coef * full if acc is None else acc.add_(full, alpha=coef)
    return acc


def _solutions(p, solver):
    return {(jx, jt, c): solver.solve(jx, jt) for jx, jt, c in _components(p.J + 2 * p.mx, p.mx)}


def _interp(x, jp, vals):
    """Multilinear interpolation of nodal values on the unit square, as weights and indices."""
    N = 1 << jp
    w = np.ones((len(x), 4))
    at = np.zeros((len(x), 4), dtype=np.int64)
    for k in range(2):
        s = x[:, k] * N
        i = np.clip(np.floor(s).astype(np.int64), 0, N - 1)
        for c in range(4):
            b = (c >> k) & 1
            w[:, c] *= (s - i) if b else 1.0 - (s - i)
            at[:, c] += (i + b) * (N + 1) ** k
    return w, at, (np.sum(w * vals[at], axis=1) if vals is not None else None)


def _exact_gradient(case, seed):
    c2n, gn, rec, obs = inverse_data(case, seed)
    jp, T = case["jp"], case["T"]
    p = dataclasses.replace(problem(case, seed), terms=[(None, _ricker(case["fp"]))])
    if ((1 << (p.mx + p.J)) - 1) ** 2 > 4100:
        return None
    S = _Dense(p, c2=lambda x: _interp(x, jp, c2n)[2], g=lambda x: _interp(x, jp, gn)[2])
    sols = _solutions(p, S)
    nts = (1 << case["jt"]) + 1
    times = np.linspace(0.0, T, nts)
    wt = np.full(nts, T / (nts - 1))
    wt[0] = wt[-1] = 0.5 * T / (nts - 1)
    w = _t(wt)[:, None]
    e = -_t(obs)
    ev = {}
    for (jx, jt, c), U in sols.items():
        wr, at, _ = _interp(rec, jx, None)
        E = torch.zeros((len(rec), ((1 << jx) + 1) ** 2), dtype=F64, device=_dev())
        E.scatter_add_(1, torch.as_tensor(at, device=_dev()), _t(wr))
        E = E[:, _inner(p, jx)]
        P = _splines(times, 1 << jt, T)[0]
        ev[(jx, jt, c)] = (E, P)
        e = e + c * (P @ U) @ E.T
    J = 0.5 * torch.sum(w * e * e)
    npar = ((1 << jp) + 1) ** 2
    dc2, dg = (torch.zeros(npar, dtype=F64, device=_dev()) for _ in range(2))
    for (jx, jt, c), U in sols.items():
        E, P = ev[(jx, jt, c)]
        L = S.solve(jx, jt, c * (P.T @ (w * e)) @ E, transposed=True)
        Me, Ke, corner, inner = S.space(jx)[:4]
        _, B, tq, Q, _, _ = _time_system(jt, T)
        na = ((1 << jx) + 1) ** 2
        full = [torch.zeros((len(B), na), dtype=F64, device=_dev()) for _ in range(2)]
        full[0][:, inner], full[1][:, inner] = L, B @ U
        cell = -torch.einsum("icp,pq,icq->c", full[0][:, corner], Ke, full[1][:, corner])
        wc, at, _ = _interp(_centres(p, jx), jp, None)
        dc2.index_add_(0, torch.as_tensor(at, device=_dev()).reshape(-1), (_t(wc) * cell[:, None]).reshape(-1))
        b = Q @ _t(p.terms[0][1](tq))
        node = _apply(Me, corner, (b @ full[0])[None])[0]
        wn, at, _ = _interp(_nodes(p, jx), jp, None)
        dg.index_add_(0, torch.as_tensor(at, device=_dev()).reshape(-1), (_t(wn) * node[:, None]).reshape(-1))
    return dict(J=float(J) if case["kind"] == "gradient" else J, dc2=dc2, dg=dg)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gradient", "inversion"):
        return _exact_gradient(case, seed)
    if kind == "batch":  # the dense solver for the small members of the ensemble, the first two of them
        out = []
        for i, n in enumerate(int(v) for v in case["levels"].split(",")):
            p = problem(case, seed, n, i)
            S = _solver64(p) if sum(o is not None for o in out) < 2 else None
            out.append(None if S is None else
                       _field(p, _solutions(p, S), np.linspace(0.0, p.T, 17), n - case["m"] - 1))
        return out
    p = problem(case, seed)
    S = _solver64(p)
    if S is None:
        return None
    sols = _solutions(p, S)
    if kind == "combine":
        return _field(p, sols, np.linspace(0.0, p.T, (1 << case["jt"]) + 1), case["jx"])
    j = p.mx + p.J
    Me, Ke, corner = _elements(p, j)
    c2 = _t(p.c2(_centres(p, j)))
    parts, times = [], _instants(case)
    step = max(1, (1 << 25) // len(corner))
    for a in range(0, len(times), step):
        y, z = (_field(p, sols, times[a:a + step], j, deriv)[:, corner] for deriv in (0, 1))
        parts.append(0.5 * (torch.einsum("tcp,pq,tcq->t", z, Me, z) +
                            torch.einsum("c,tcp,pq,tcq->t", c2, y, Ke, y)))
    return torch.cat(parts).cpu().numpy()
