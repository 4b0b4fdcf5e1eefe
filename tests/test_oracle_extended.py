"""The extended-precision steps agree with the FP64 oracle to FP64 rounding."""
import numpy as np
import pytest

from oracle import extended as X
from oracle import propagate as P
from oracle import tables as T


@pytest.mark.parametrize("kind", [T.SHARP, T.SECS])
@pytest.mark.parametrize("field", [None, (0.05, 0.5, 3.0)])
def test_1d(kind, field):
    n, hw = 256, 50.0
    p = P.Problem1D(n, -hw, hw, 0.75 * hw, theta=0.5, kind=kind, a2=2.0, dt=0.05)
    psi = np.exp(-(p.x - 30.0) ** 2 / 80.0 + 0.9j * p.x)      # reaches a strip
    assert X.rel(p.step(psi, 20, t0=1.0, field=field), X.step1d(p, psi, 20, 1.0, field)) < 5e-14


def test_strip_across_the_box_edge_and_none():
    sub = np.zeros(16, dtype=complex)
    diag, sup = sub.copy(), sub.copy()
    rows = [13, 14, 15, 0, 1]
    rng = np.random.default_rng(1)
    diag[rows] = rng.standard_normal(5) + 1j * rng.standard_normal(5)
    for a, b in zip(rows[:-1], rows[1:]):
        sup[a] = sub[b] = rng.standard_normal() + 1j * rng.standard_normal()
    C = np.diag(diag) + 0j
    for i in range(16):
        C[i, (i + 1) % 16] += sup[i]
        C[i, (i - 1) % 16] += sub[i]
    v = rng.standard_normal((3, 16)) + 1j * rng.standard_normal((3, 16))
    one = np.eye(16)
    M = np.linalg.solve(one + 0.05j * C, one - 0.05j * C)
    got = X._Strip(sub, diag, sup, 0.1).apply(v.astype(X.CL))
    assert X.rel(v @ M.T, got) < 1e-14
    z = np.zeros(16, dtype=complex)
    assert np.array_equal(X._Strip(z, z, z, 0.1).apply(v), v)


@pytest.mark.parametrize("n", [(32, 16), (16, 32, 8)])
def test_grids(n):
    box, nd = (-12.0, 12.0) * len(n), len(n)
    rng = np.random.default_rng(nd)
    psi = rng.standard_normal(n[::-1]) + 1j * rng.standard_normal(n[::-1])
    if nd == 2:
        p = P.Problem2D(n[0], n[1], box, 9.0, dt=0.02)
        axes = [(p.kx,) + tuple(p.Cx), (p.ky,) + tuple(p.Cy)]
    else:
        p = P.Problem3D(n, box, 9.0, dt=0.02)
        axes = [(p.k[d],) + tuple(p.C[d]) for d in range(3)]
    assert X.rel(p.step(psi, 4), X.step_grid(p, axes, psi, 4)) < 1e-14
