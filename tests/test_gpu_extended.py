"""Accuracy of the complex128 steps in 64-bit fixed point against the oracle's
scheme in extended precision (oracle/extended.py), which an FP64 oracle, itself
off by 2e-15 to 7e-15 after these steps, cannot tell.

Tolerance: per step and axis 2e-16 for the fixed-point FFTs and products
(fix64.cuh) and 1.1e-16 for the rounding of the tables' phases, at most about
1 rad on the modes these states hold, added up linearly.  A shared exponent or
a factor table that is off by more than a few bits, in one pass or one branch,
leaves more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import extended as X  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import tables as T  # noqa: E402

PER_STEP = 2e-16 + 1.1e-16
NSTEPS = 12


def _problem(n):
    """The single-instance workload's contour and spacing (h = 0.39)."""
    hw = 200.0 * n / 1024
    return P.Problem1D(n, -hw, hw, 0.75 * hw, theta=0.5, kind=T.SHARP, a2=2.0, dt=0.05), hw


def _state(where, x, hw):
    if where == "broad":
        return np.exp(-x ** 2 / (0.5 * hw) ** 2 + 0.7j * x)
    return np.exp(-(x - 0.9 * hw) ** 2 / max(0.02 * hw, 3.0) ** 2 + 0.3j * x)     # inside a scaled strip


def _err(got, ref, psi):
    """relative to the initial norm (the strips absorb)"""
    d = np.sqrt(np.sum(np.abs(got.astype(X.CL) - ref) ** 2))
    return float(d / np.linalg.norm(psi))


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384])
@pytest.mark.parametrize("where", ["broad", "strip"])
def test_single_steps(n, where):
    p, hw = _problem(n)
    psi = _state(where, p.x, hw)
    plan = S.soft_create(n, (-hw, hw), 0.75 * hw, 0.5, 0.05, prec=S.SOFT_C128, contour=S.CONTOUR_SHARP, soft_a2=2.0)
    try:
        d = torch.tensor(psi, dtype=torch.complex128, device="cuda")
        S.soft_step(plan, d, NSTEPS, 0.0)
        torch.cuda.synchronize()
    finally:
        S.soft_destroy(plan)
    assert _err(d.cpu().numpy(), X.step1d(p, psi, NSTEPS), psi) < NSTEPS * PER_STEP


@pytest.mark.parametrize("persistent", [0, 1])
def test_batch_steps(persistent):
    ns = [1024, 2048, 4096, 8192, 16384]
    ps, hws = zip(*[_problem(n) for n in ns])
    psis = [_state("broad", p.x, hw) for p, hw in zip(ps, hws)]
    plan = S.soft_create_batch(ns, [(-w, w) for w in hws], [0.75 * w for w in hws], [0.5] * len(ns), None, 0.05,
                               prec=S.SOFT_C128, contour=S.CONTOUR_SHARP, soft_a2=2.0, persistent=persistent)
    try:
        off, _ = S.soft_batch_layout(plan)
        d = torch.tensor(np.concatenate(psis), dtype=torch.complex128, device="cuda")
        S.soft_step_batch(plan, d, NSTEPS, 0.0)
        torch.cuda.synchronize()
    finally:
        S.soft_destroy(plan)
    got = d.cpu().numpy()
    for n, o, p, psi in zip(ns, off, ps, psis):
        assert _err(got[o:o + n], X.step1d(p, psi, NSTEPS), psi) < NSTEPS * PER_STEP, n


@pytest.mark.parametrize("n", [(256, 512), (1024, 256), (256, 2048), (64, 64, 128), (128, 64, 64)])
def test_grid_steps(n):
    hw, steps, nd = 16.0, 3, len(n)
    box = (-hw, hw) * nd
    psi = np.ones([1] * nd, dtype=complex)
    for d, m in enumerate(n):
        x = -hw + 2 * hw / m * (np.arange(m) + 0.5)
        v = np.exp(-(x - 0.1 * d * hw) ** 2 / (0.4 * hw) ** 2 + (0.5 - 0.3 * d) * 1j * x)
        psi = psi * v.reshape([-1 if e == d else 1 for e in reversed(range(nd))])
    if nd == 2:
        p = P.Problem2D(n[0], n[1], box, 0.75 * hw, theta=0.4, kind=T.SHARP, a2=1.0, dt=0.02)
        axes = [(p.kx,) + tuple(p.Cx), (p.ky,) + tuple(p.Cy)]
    else:
        p = P.Problem3D(n, box, 0.75 * hw, theta=0.4, kind=T.SHARP, a2=1.0, dt=0.02)
        axes = [(p.k[d],) + tuple(p.C[d]) for d in range(3)]
    plan = S.soft_create(n, box, 0.75 * hw, 0.4, 0.02, prec=S.SOFT_C128, contour=S.CONTOUR_SHARP, soft_a2=1.0)
    try:
        d = torch.tensor(np.ascontiguousarray(psi), dtype=torch.complex128, device="cuda")
        S.soft_step(plan, d, steps, 0.0)
        torch.cuda.synchronize()
    finally:
        S.soft_destroy(plan)
    assert _err(d.cpu().numpy(), X.step_grid(p, axes, psi, steps), psi) < steps * nd * PER_STEP


@pytest.mark.parametrize("n", [256, 2048, 16384])
def test_norm_over_many_steps(n):
    """Without scaling (theta = 0) a step is unitary; 2^-60 per step, the size
    of a factor's modulus error, plus the final conversion's 2^-53."""
    hw = 200.0 * n / 1024
    x = -hw + 2 * hw / n * (np.arange(n) + 0.5)
    psi = np.exp(-x ** 2 / (0.2 * hw) ** 2 + 0.5j * x)
    plan = S.soft_create(n, (-hw, hw), 0.75 * hw, 0.0, 0.05, prec=S.SOFT_C128, contour=S.CONTOUR_SECS, soft_a2=2.0)
    steps = 4000
    try:
        d = torch.tensor(psi, dtype=torch.complex128, device="cuda")
        S.soft_step(plan, d, steps, 0.0)
        torch.cuda.synchronize()
    finally:
        S.soft_destroy(plan)
    nrm = lambda v: np.sqrt(np.sum(np.abs(v.astype(X.CL)) ** 2))  # noqa: E731
    assert abs(float(nrm(d.cpu().numpy()) / nrm(psi) - 1)) < steps * 2.0 ** -60 + 2.0 ** -53
