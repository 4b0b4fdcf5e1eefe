"""Complex128 steps in potentials that absorb at every point: the fixed-point
products round relative to a line's norm before the factor, so what is left
must not be measured against that.  Against the scheme in extended precision.

Tolerance: as in test_gpu_extended.py per step and axis, plus the roundings of
the factors in FP64: the logarithm's (half a unit of |log|), the exponential's
and the product's, two of each per step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import extended as X  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import tables as T  # noqa: E402

PER_STEP, ULP, NSTEPS, DT = 2e-16 + 1.1e-16, 1.1e-16, 3, 1 / 32


def _run(plan, U, psi):
    try:
        S.soft_set_potential(plan, U)
        d = torch.tensor(np.ascontiguousarray(psi), dtype=torch.complex128, device="cuda")
        S.soft_step(plan, d, NSTEPS, 0.0)
        torch.cuda.synchronize()
        return d.cpu().numpy()
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n", [64, 256, 2048, 16384])
@pytest.mark.parametrize("loss", [1.5, 4.0, 14.0, 60.0])
def test_single(n, loss):
    """e^-loss per step on every point."""
    hw = 200.0 * n / 1024
    p = P.Problem1D(n, -hw, hw, 0.75 * hw, theta=0.5, kind=T.SHARP, a2=2.0, dt=DT)
    p.U0 = p.U0 - 1j * loss / DT
    psi = np.exp(-p.x ** 2 / (0.3 * hw) ** 2 + 0.7j * p.x)
    plan = S.soft_create(n, (-hw, hw), 0.75 * hw, 0.5, DT, prec=S.SOFT_C128, contour=S.CONTOUR_SHARP, soft_a2=2.0)
    got = _run(plan, p.U0, psi)
    assert X.rel(got, X.step1d(p, psi, NSTEPS)) < NSTEPS * (PER_STEP + (loss + 4) * ULP)


@pytest.mark.parametrize("n", [(256, 512), (64, 64, 128)])
@pytest.mark.parametrize("loss", [1.5, 14.0, 60.0])
def test_grids(n, loss):
    hw, nd = 16.0, len(n)
    box = (-hw, hw) * nd
    if nd == 2:
        p = P.Problem2D(n[0], n[1], box, 0.75 * hw, theta=0.4, kind=T.SHARP, a2=1.0, dt=DT)
        axes = [(p.kx,) + tuple(p.Cx), (p.ky,) + tuple(p.Cy)]
    else:
        p = P.Problem3D(n, box, 0.75 * hw, theta=0.4, kind=T.SHARP, a2=1.0, dt=DT)
        axes = [(p.k[d],) + tuple(p.C[d]) for d in range(3)]
    p.U = p.U - 1j * loss / DT
    psi = np.ones([1] * nd, dtype=complex)
    for d, m in enumerate(n):
        x = -hw + 2 * hw / m * (np.arange(m) + 0.5)
        psi = psi * np.exp(-x ** 2 / (0.3 * hw) ** 2 + 0.5j * x).reshape([-1 if e == d else 1 for e in reversed(range(nd))])
    plan = S.soft_create(n, box, 0.75 * hw, 0.4, DT, prec=S.SOFT_C128, contour=S.CONTOUR_SHARP, soft_a2=1.0)
    got = _run(plan, p.U, psi)
    assert X.rel(got, X.step_grid(p, axes, psi, NSTEPS)) < NSTEPS * (nd * PER_STEP + (loss + 4) * ULP)
