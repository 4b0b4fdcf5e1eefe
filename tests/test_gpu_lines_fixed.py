"""The complex128 2D and 3D line passes in 64-bit fixed point (one exponent
per line): states of any scale and with empty lines, packets inside the scaled
strips, potentials whose factors do not fit fixed point, backward steps and
non-finite samples, against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import tables as T  # noqa: E402

# a few 1e-16 per line FFT pair and step, as in the other step tests
TOL = 1e-11
SHAPES = [(256, 512), (1024, 256), (64, 64, 128), (128, 256, 64)]     # x fastest
KIND = {T.SECS: S.CONTOUR_SECS, T.SHARP: S.CONTOUR_SHARP}


def _problem(n, kind=T.SHARP, dt=0.02, theta=0.4, hw=16.0):
    box = (-hw, hw) * len(n)
    plan = S.soft_create(n, box, 0.75 * hw, theta, dt, prec=S.SOFT_C128, contour=KIND[kind], soft_a2=1.0)
    if len(n) == 2:
        return plan, P.Problem2D(n[0], n[1], box, 0.75 * hw, theta=theta, kind=kind, a2=1.0, dt=dt), hw
    return plan, P.Problem3D(n, box, 0.75 * hw, theta=theta, kind=kind, a2=1.0, dt=dt), hw


def _state(n, hw, where):
    psi = np.ones([1] * len(n), dtype=complex)
    for d, m in enumerate(n):
        x = -hw + 2 * hw / m * (np.arange(m) + 0.5)
        if where == "strip":                      # in the corner of the strips, far lines (nearly) empty
            v = np.exp(-(x - 0.88 * hw) ** 2 / (0.04 * hw) ** 2 + 0.4j * x)
        else:
            v = np.exp(-(x - 0.1 * d * hw) ** 2 / (0.4 * hw) ** 2 + (0.5 - 0.3 * d) * 1j * x)
        psi = psi * v.reshape([-1 if e == d else 1 for e in reversed(range(len(n)))])
    return psi


def _run(plan, psi, steps):
    d = torch.tensor(np.ascontiguousarray(psi), dtype=torch.complex128, device="cuda")
    S.soft_step(plan, d, steps, 0.0)
    torch.cuda.synchronize()
    return d.cpu().numpy()


def _err(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("where,scale", [("broad", 1.0), ("broad", 1e-290), ("broad", 1e280), ("strip", 1.0),
                                         ("strip", 1e-30)])
def test_scales_and_strips(n, where, scale):
    plan, p, hw = _problem(n)
    try:
        psi = _state(n, hw, where)
        assert _err(_run(plan, psi * scale, 3) / scale, p.step(psi, 3)) < TOL
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("gain", [30.0, 300.0])
def test_potentials_with_gain(n, gain):
    """|e^{-iU tau/2}| up to 1.35 (a scaled table) and 20 (applied in FP64);
    setting the first potential back restores its run."""
    plan, p, hw = _problem(n)
    try:
        psi = _state(n, hw, "broad")
        U0 = p.U.copy()
        g = np.abs(_state(n, hw, "broad")) ** 8 + np.abs(_state(n, hw, "strip"))
        S.soft_set_potential(plan, U0)
        base = _run(plan, psi, 2)
        S.soft_set_potential(plan, U0 + 1j * gain * g)
        p.U = U0 + 1j * gain * g
        assert _err(_run(plan, psi, 2), p.step(psi, 2)) < TOL
        S.soft_set_potential(plan, U0)
        assert np.array_equal(_run(plan, psi, 2), base)
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("kind", [T.SHARP, T.SECS])
def test_backward_steps(n, kind):
    """dt < 0: the strip multipliers exceed 1 (strips solved in FP64)."""
    plan, p, hw = _problem(n, kind=kind, dt=-0.002, theta=0.2)
    try:
        psi = _state(n, hw, "broad")
        ref = p.step(psi, 2)
        assert _err(_run(plan, psi, 2), ref) < TOL * max(1.0, np.linalg.norm(ref) / np.linalg.norm(psi))
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", SHAPES)
def test_zero_and_non_finite(n):
    plan, p, hw = _problem(n)
    try:
        psi = np.zeros(tuple(reversed(n)), dtype=complex)
        assert np.all(_run(plan, psi, 2) == 0)
        psi = _state(n, hw, "broad")
        psi.reshape(-1)[7] = np.inf
        assert np.all(np.isnan(_run(plan, psi, 2).real))
    finally:
        S.soft_destroy(plan)
