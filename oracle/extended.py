"""The split step of ``propagate`` in the platform's extended precision (80 or
128 bits, numpy longdouble), from the same per-axis tables: what tells errors
of FP64 size apart, which another FP64 run cannot.

TEST INFRASTRUCTURE (see ``oracle/__init__``)."""
from __future__ import annotations

import math

import numpy as np

LD, CL = np.longdouble, np.clongdouble


class _Strip:
    """(1 + i tau C/2)^-1 (1 - i tau C/2) on the rows where C is not zero: a
    cyclic run of rows, eliminated without pivoting."""

    def __init__(self, sub, diag, sup, tau):
        n = len(diag)
        on = (np.abs(sub) + np.abs(diag) + np.abs(sup)) > 0
        self.rows = np.nonzero(on)[0]
        if len(self.rows) == 0:
            return
        first = next(int(r) for r in self.rows if not on[(r - 1) % n])
        self.rows = (first + np.arange(len(self.rows))) % n
        assert on[self.rows].all()
        a = CL(0.5j) * LD(tau)
        self.c = [a * v[self.rows].astype(CL) for v in (sub, diag, sup)]
        s, d, u = self.c
        self.inv = np.empty(len(s), dtype=CL)       # pivots, inverted
        p = 1 + d[0]
        self.inv[0] = 1 / p
        for i in range(1, len(s)):
            p = 1 + d[i] - s[i] * self.inv[i - 1] * u[i - 1]
            self.inv[i] = 1 / p

    def apply(self, v, axis=-1):
        if len(self.rows) == 0:
            return v
        s, d, u = self.c
        v = np.moveaxis(v, axis, 0).copy()
        r = v[self.rows]
        col = (-1,) + (1,) * (r.ndim - 1)
        y = r - d.reshape(col) * r
        y[1:] -= s[1:].reshape(col) * r[:-1]
        y[:-1] -= u[:-1].reshape(col) * r[1:]
        for i in range(1, len(s)):
            y[i] -= s[i] * self.inv[i - 1] * y[i - 1]
        y[-1] *= self.inv[-1]
        for i in range(len(s) - 2, -1, -1):
            y[i] = (y[i] - u[i] * y[i + 1]) * self.inv[i]
        v[self.rows] = y
        return np.moveaxis(v, 0, axis)


def step1d(p, psi, nsteps, t0=0.0, field=None):
    """nsteps of ``propagate.Problem1D`` p (field: E0, omega, ncycles)."""
    tau = LD(p.dt)
    kh = np.exp(CL(-0.25j) * tau * p.k.astype(LD) ** 2)
    vh = np.exp(CL(-0.5j) * tau * p.U0.astype(CL))
    cn = _Strip(p.Cs, p.Cd, p.Cu, p.dt)
    v = psi.astype(CL)
    for s in range(nsteps):
        w = vh
        if field is not None:
            E0, om, nc = field
            T = nc * 2 * math.pi / om
            t = t0 + (s + 0.5) * p.dt
            E = E0 * math.sin(math.pi * t / T) ** 2 * math.sin(om * t) if 0 <= t <= T else 0.0
            w = vh * np.exp(CL(-0.5j) * tau * LD(E) * p.xc.astype(LD))
        v = np.fft.ifft(kh * np.fft.fft(v)) * w
        v = np.fft.ifft(kh * np.fft.fft(cn.apply(v) * w))
    return v


def step_grid(p, axes, psi, nsteps):
    """nsteps of a 2D or 3D problem p (U of shape psi.shape); axes: x first, each
    with k and the three diagonals Cs, Cd, Cu."""
    tau, nd = LD(p.dt), len(axes)
    vh = np.exp(CL(-0.5j) * tau * p.U.reshape(psi.shape).astype(CL))
    dims = [nd - 1 - d for d in range(nd)]
    col = lambda d, a: a.reshape([-1 if e == dims[d] else 1 for e in range(nd)])
    kh = [col(d, np.exp(CL(-0.25j) * tau * a[0].astype(LD) ** 2)) for d, a in enumerate(axes)]
    cns = [_Strip(a[1], a[2], a[3], p.dt) for a in axes]

    def kinetic(v):
        for d in range(nd):
            v = np.fft.ifft(kh[d] * np.fft.fft(v, axis=dims[d]), axis=dims[d])
        return v

    v = psi.astype(CL)
    for _ in range(nsteps):
        v = kinetic(v) * vh
        for d in range(nd):
            v = cns[d].apply(v, dims[d])
        v = kinetic(v * vh)
    return v


def rel(a, b):
    """relative L2 distance of a from b in extended precision"""
    return float(np.sqrt(np.sum(np.abs(a.astype(CL) - b) ** 2) / np.sum(np.abs(b) ** 2)))
