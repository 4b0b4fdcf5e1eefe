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


# tolerances of test_gpu_pcg1d: 1e-12 for A, 1e-11 for the preconditioners
@pytest.mark.parametrize("n", [256, 512, 1024, 2048])
@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e200])
def test_1d_A_and_preconditioners(n, scale):
    hw, R0, th = 51.2 * n / 1024, 40.0 * n / 1024, 0.6
    plan = S.soft_create(n, (-hw, hw), R0, th, 0.02, prec=S.SOFT_C128, contour=S.CONTOUR_SECS, soft_a2=2.0)
    p = P.Problem1D(n, -hw, hw, R0, theta=th, kind=T.SECS, a2=2.0, dt=0.02)
    st = ST.Stationary1D(p, nbw=10)
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    x[n // 4:n // 2] *= 1e-9
    try:
        dx = torch.tensor(x * scale, dtype=torch.complex128, device="cuda")
        dy = torch.zeros_like(dx)
        get = lambda: dy.cpu().numpy() / scale    # noqa: E731
        S.sse_apply_A(plan, 0.7, dx, dy)
        assert _err(get(), st.apply_A(x, 0.7)) < 1e-12
        for kind, ref in ((0, st.precond_simple), (1, st.precond_band)):
            S.sse_apply_precond(plan, 0.7, kind, dx, dy)
            assert _err(get(), ref(x, 0.7)) < 1e-11
        dx[3] = float("nan")
        S.sse_apply_precond(plan, 0.7, 1, dx, dy)
        assert torch.isnan(dy.real).all()
    finally:
        S.soft_destroy(plan)


@pytest.mark.parametrize("n,precond", [(256, 0), (256, 1), (2048, 1)])
def test_1d_solve_of_a_scaled_source(n, precond):
    """x is linear in f; a non-finite source is refused as before."""
    hw, R0 = 51.2 * n / 1024, 40.0 * n / 1024
    plan = S.soft_create(n, (-hw, hw), R0, 0.6, 0.02, prec=S.SOFT_C128, contour=S.CONTOUR_SECS, soft_a2=2.0)
    p = P.Problem1D(n, -hw, hw, R0, theta=0.6, kind=T.SECS, a2=2.0, dt=0.02)
    st = ST.Stationary1D(p, nbw=10)
    f = np.exp(-(p.x - 1.0) ** 2 / 3.0 + 0.4j * p.x)
    Es = [0.35, 1.2, 2.5]
    try:
        for scale in (1.0, 1e-60, 1e60):
            out = torch.zeros((3, n), dtype=torch.complex128, device="cuda")
            rc, its, rr = S.sse_pcg_solve(plan, Es, torch.tensor(f * scale, device="cuda"), out, tol=1e-10,
                                          maxit=3000, precond=precond)
            assert rc == 0
            for e, E in enumerate(Es):
                res = np.linalg.norm(f - st.apply_A(out[e].cpu().numpy() / scale, E)) / np.linalg.norm(f)
                assert res < 2e-10
        bad = torch.tensor(f, device="cuda")
        bad[5] = float("inf")
        with pytest.raises(S.SoftError) as err:
            S.sse_pcg_solve(plan, Es, bad, out, tol=1e-10, maxit=30, precond=precond)
        assert err.value.status == -8
    finally:
        S.soft_destroy(plan)
