"""The complex128 1D step in 64-bit fixed point (shared exponent per state):
states of any scale, packets that sit inside the scaled strips, plans whose
factors do not fit fixed point (gains, backward steps), and the ends of its
range, against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import tables as T  # noqa: E402

# as in the other step tests: a few 1e-16 per step for the two FFTs and the
# phase tables, far below 1e-11 for the steps taken here
TOL = 1e-11
NSTEPS = 12


def _problem(n, kind=T.SECS, dt=0.02, theta=0.5):
    hw = 8.0 * n / 1024
    plan = S.soft_create(n, (-hw, hw), 0.75 * hw, theta, dt, prec=S.SOFT_C128,
                         contour={T.SECS: S.CONTOUR_SECS, T.SHARP: S.CONTOUR_SHARP}[kind])
    return plan, P.Problem1D(n, -hw, hw, 0.75 * hw, theta=theta, kind=kind, a2=2.0, dt=dt), hw


def _run(plan, psi, steps=NSTEPS, t=0.0, field=None):
    d = torch.tensor(psi, dtype=torch.complex128, device="cuda")
    S.soft_step(plan, d, steps, t, field=field)
    torch.cuda.synchronize()
    return d.cpu().numpy()


def _err(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _state(where, x, hw, rng):
    if where == "broad":
        return np.exp(-x ** 2 / (0.5 * hw) ** 2 + 0.7j * x) * (1 + 0.01 * rng.standard_normal(len(x)))
    if where == "strip":                 # all of the norm inside one scaled strip
        return np.exp(-(x - 0.9 * hw) ** 2 / (0.02 * hw) ** 2 + 0.3j * x)
    psi = np.zeros(len(x), dtype=complex)        # a single point of the strip, next to the box edge
    psi[-2] = 1.0 - 0.5j
    return psi


@pytest.mark.parametrize("n", [64, 128, 512, 2048, 4096, 8192, 16384])
@pytest.mark.parametrize("where", ["broad", "strip", "point"])
def test_states_inside_the_strips(n, where):
    plan, p, hw = _problem(n)
    try:
        psi = _state(where, p.x, hw, np.random.default_rng(n))
        assert _err(_run(plan, psi), p.step(psi, NSTEPS)) < TOL
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("scale", [1e-290, 1e-30, 1e40, 1e280])
@pytest.mark.parametrize("n", [256, 4096, 16384])
def test_any_scale_of_the_state(n, scale):
    """The step is linear: the result of a scaled state is the scaled result."""
    plan, p, hw = _problem(n)
    try:
        psi = _state("broad", p.x, hw, np.random.default_rng(n))
        assert _err(_run(plan, psi * scale) / scale, p.step(psi, NSTEPS)) < TOL
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", [256, 2048, 16384])
@pytest.mark.parametrize("gain", [0.5, 30.0, 3000.0])
def test_potentials_with_gain(n, gain):
    """|e^{-iU tau}| of 1.01, 1.8 (a scaled table) and 1e26 (applied in FP64)
    on part of the grid, strip rows included."""
    plan, p, hw = _problem(n)
    try:
        psi = _state("broad", p.x, hw, np.random.default_rng(n))
        U = p.U0 + 1j * gain * np.exp(-(p.x - 0.8 * hw) ** 2 / (0.03 * hw) ** 2)
        S.soft_set_potential(plan, U)
        p.U0 = U
        q = P.Problem1D(n, -hw, hw, 0.75 * hw, theta=0.5, kind=T.SECS, a2=2.0, dt=0.02)
        q.U0 = U
        steps = 2 if gain > 1000 else NSTEPS
        field = (0.05, 0.5, 3.0)
        assert _err(_run(plan, psi, steps, 1.0, field), q.step(psi, steps, t0=1.0, field=field)) < TOL
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", [64, 1024, 4096])
@pytest.mark.parametrize("kind", [T.SECS, T.SHARP])
def test_backward_steps(n, kind):
    """dt < 0: the strips amplify, the strip multipliers exceed 1."""
    plan, p, hw = _problem(n, kind=kind, dt=-0.002, theta=0.2)
    try:
        psi = np.exp(-p.x ** 2 / (0.15 * hw) ** 2) + 0j
        ref = p.step(psi, 4)
        assert _err(_run(plan, psi, 4), ref) < TOL * max(1.0, np.linalg.norm(ref) / np.linalg.norm(psi))
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", [64, 1024, 16384])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_zero_and_non_finite_states(n, bad):
    plan, p, hw = _problem(n)
    try:
        z = _run(plan, np.zeros(n, dtype=complex))
        assert np.all(z == 0)
        S.soft_step_status(plan)
        psi = _state("broad", p.x, hw, np.random.default_rng(n))
        psi[n // 3] = bad
        assert np.all(np.isnan(_run(plan, psi).real))
        with pytest.raises(S.SoftError):
            S.soft_step_status(plan)
    finally:
        S.soft_destroy(plan)
