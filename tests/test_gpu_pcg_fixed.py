"""A and the preconditioners of the 2D solver in 64-bit fixed point (one
exponent per line): rectangular grids at the ends of the sizes, states of any
scale, empty lines, the simple and the banded preconditioner, against the FP64
oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import propagate as P  # noqa: E402
from oracle import stationary as ST  # noqa: E402
from oracle import tables as T  # noqa: E402


def _err(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# tolerances of test_gpu_pcg: 1e-12 for A, 1e-11 for the preconditioners
@pytest.mark.parametrize("nx,ny", [(256, 512), (2048, 256), (256, 1024)])
@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e200])
def test_A_and_preconditioners(nx, ny, scale):
    box, R0, th = (-40.0, 40.0, -40.0, 40.0), 30.0, 0.4
    plan = S.soft_create((nx, ny), box, R0, th, 0.02, prec=S.SOFT_C128, soft_a2=1.0)
    p2 = P.Problem2D(nx, ny, box, R0, theta=th, a2=1.0, dt=0.02)
    st = ST.Stationary2D(p2, nbw=10, kind=T.SHARP, R0=R0, theta=th)
    rng = np.random.default_rng(nx + ny)
    x = rng.standard_normal((ny, nx)) + 1j * rng.standard_normal((ny, nx))
    x[ny // 3] = 0.0                              # an empty row ...
    x[:, 5:9] *= 1e-9                             # ... and nearly empty columns
    try:
        dx = torch.tensor(x * scale, dtype=torch.complex128, device="cuda")
        dy = torch.zeros_like(dx)
        get = lambda: dy.cpu().numpy() / scale    # noqa: E731
        S.sse_apply_A(plan, 0.7, dx, dy)
        assert _err(get(), st.apply_A(x, 0.7)) < 1e-12
        S.sse_apply_precond(plan, 0.7, 0, dx, dy)
        assert _err(get(), st.precond_simple(x, 0.7)) < 1e-11
        S.sse_apply_precond(plan, 0.7, 1, dx, dy)
        assert _err(get(), st.precond_band(x, 0.7)) < 1e-11
        dx[3, 4] = float("nan")
        S.sse_apply_precond(plan, 0.7, 1, dx, dy)
        assert torch.isnan(dy.real).all()
    finally:
        S.soft_destroy(plan)
