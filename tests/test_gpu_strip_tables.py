"""The complex64 strip Crank-Nicolson with tabulated scans (1D kernels, 2D and
3D line passes): all of the norm inside the strips, chunks without rows, and
steps so long that the recurrences reach across warps, against the FP64
oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import tables as T  # noqa: E402

# complex64 is held to 1e-5 over up to 2000 steps elsewhere; a step's own
# rounding is about 1.5e-7
TOL = 1e-5


def _err(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# dt = 8: |mf| = 0.99 (h = 1/64), so that a warp's 32 chunks leave 1e-2 to 1e-4 of a carry
@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384])
@pytest.mark.parametrize("dt", [0.02, 8.0])
@pytest.mark.parametrize("frac", [0.75, 0.97])
def test_1d(n, dt, frac):
    hw = 8.0 * n / 1024
    R0 = int(frac * n / 2) * 2 * hw / n            # a cell edge
    plan = S.soft_create(n, (-hw, hw), R0, 0.5, dt, prec=S.SOFT_C64, contour=S.CONTOUR_SECS, soft_a2=2.0)
    p = P.Problem1D(n, -hw, hw, R0, theta=0.5, kind=T.SECS, a2=2.0, dt=dt)
    rng = np.random.default_rng(n)
    psi = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * np.where(abs(p.x) > R0, 1.0, 1e-3)
    d = torch.tensor(psi, dtype=torch.complex64, device="cuda")
    try:
        S.soft_step(plan, d, 3, 0.0)
        assert _err(d.cpu().numpy(), p.step(psi.astype(np.complex64).astype(complex), 3)) < TOL
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("nx,ny", [(256, 256), (1024, 256), (256, 2048)])
@pytest.mark.parametrize("dt", [0.02, 8.0])
def test_2d(nx, ny, dt):
    box, R0, th = (-4.0, 4.0, -4.0, 4.0), 3.0, 0.4
    plan = S.soft_create((nx, ny), box, R0, th, dt, prec=S.SOFT_C64, soft_a2=1.0)
    p = P.Problem2D(nx, ny, box, R0, theta=th, a2=1.0, dt=dt)
    rng = np.random.default_rng(nx + ny)
    psi = rng.standard_normal((ny, nx)) + 1j * rng.standard_normal((ny, nx))
    d = torch.tensor(psi, dtype=torch.complex64, device="cuda")
    try:
        S.soft_step(plan, d, 2, 0.0)
        assert _err(d.cpu().numpy(), p.step(psi.astype(np.complex64).astype(complex), 2)) < TOL
    finally:
        S.soft_destroy(plan)
