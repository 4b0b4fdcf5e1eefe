"""What users of this library wait for: timed cases over its public calls.

Every case is one call (or the few calls a program makes together) of the
package: time steps of single 1D instances, laser batches, 2D and 3D grids, a
propagation with surface samples, stationary solves, one application of A and
of the preconditioner, and a gradient of the learned correction.  Grids,
contours and states are those of ``workloads`` scaled to the case's size.

``exact`` evaluates the same scheme (merged split steps, Crank-Nicolson by
dense inverses, FFTs, dense or Krylov solves) in complex128 torch."""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1505_06707_gb300 as S

DEV = "cuda"
CONTOURS = {"sharp": S.CONTOUR_SHARP, "secs": S.CONTOUR_SECS, "tfecs": S.CONTOUR_TFECS}
OMEGA, NCYC = 0.057, 4.0            # the laser batch's pulse
T_PULSE = 100.0                     # start time of the cases with a field (inside the pulse)


def listed():
    return [
        # a real-time loop: one step of a small instance per call
        dict(name="step1d-128-c128", kind="step1d", n=128, prec="c128", contour="sharp", field=False, steps=1),
        # the single-instance workload (N = 1024, sharp contour) in both precisions,
        # the second one in a laser field
        dict(name="step1d-1024-c64", kind="step1d", n=1024, prec="c64", contour="sharp", field=False, steps=200),
        dict(name="step1d-4096-c128-field", kind="step1d", n=4096, prec="c128", contour="secs", field=True,
             steps=50),
        # the paper's test propagation with surface samples (t-SURFF)
        dict(name="surface-1024", kind="surface", n=1024, steps=201),
        # the laser batch: many instances of four sizes, each with its pulse
        dict(name="batch-1024-c128", kind="batch", count=1024, prec="c128", sizes="2048,4096,8192,16384", steps=32),
        dict(name="batch-4096-c64", kind="batch", count=4096, prec="c64", sizes="2048,4096,8192,16384", steps=32),
        # the 2D workload in complex64, and a rectangular complex128 grid
        dict(name="plane-2048x2048-c64", kind="plane", nx=2048, ny=2048, prec="c64", steps=33),
        dict(name="plane-1024x512-c128", kind="plane", nx=1024, ny=512, prec="c128", steps=17),
        # the 3D workload
        dict(name="cube-256-c64", kind="cube", nx=256, ny=256, nz=256, prec="c64", steps=9),
        # the paper's stationary test: 30 energies, banded preconditioner, 1e-12
        dict(name="solve1d-1024", kind="solve1d", n=1024, energies=30, charge=0.0),
        # one step of a caller's own 2D Krylov method: A p and P^-1 r in FP64
        dict(name="krylov2d-1024", kind="krylov2d", nx=1024, ny=1024),
        # one gradient of the learned correction on a minibatch of crops
        dict(name="nn-grad-32x128x128", kind="nn_grad", fields=32, height=128, width=128),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step1d", "step1d", "surface", "batch", "batch", "plane", "plane", "cube", "solve1d",
                       "krylov2d", "nn_grad"])
    prec = rng.choice(["c64", "c128"])
    if kind == "step1d":
        n = 2 ** rng.randint(6, 14)
        contour = rng.choice(["sharp", "secs"])
        return dict(kind=kind, n=n, prec=prec, contour=contour, field=contour == "secs" and rng.random() < 0.5,
                    steps=_logint(rng, 1, 300))
    if kind == "surface":
        return dict(kind=kind, n=2 ** rng.randint(8, 11), steps=_logint(rng, 2, 300))
    if kind == "batch":
        sizes = sorted(rng.sample([1024, 2048, 4096, 8192, 16384], rng.randint(1, 4)))
        mean = sum(sizes) / len(sizes)
        budget = (2.5e8 if prec == "c128" else 1e9)          # point-steps of the listed cases
        count = _logint(rng, 8, 2000)
        return dict(kind=kind, count=count, prec=prec, sizes=",".join(map(str, sizes)),
                    steps=max(1, min(_logint(rng, 1, 100), int(budget / (1.3 * count * mean)))))
    if kind == "plane":
        nx, ny = 2 ** rng.randint(8, 11), 2 ** rng.randint(8, 11)
        return dict(kind=kind, nx=nx, ny=ny, prec=prec, steps=_logint(rng, 1, 40 if prec == "c64" else 10))
    if kind == "cube":
        n = [2 ** rng.randint(6, 8) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], prec=prec, steps=_logint(rng, 1, 12))
    if kind == "solve1d":
        return dict(kind=kind, n=2 ** rng.randint(8, 11), energies=rng.randint(1, 60),
                    charge=rng.choice([0.0, 1.0]))
    if kind == "krylov2d":
        return dict(kind=kind, nx=2 ** rng.randint(8, 11), ny=2 ** rng.randint(8, 10))
    return dict(kind="nn_grad", fields=_logint(rng, 1, 40), height=rng.randint(16, 150),
                width=rng.choice([128, 256]))


# ------------------------------------------------------------------ problems
def _axis(n, hw):
    h = 2.0 * hw / n
    return -hw + h * (np.arange(n) + 0.5), h


def _box(case):
    """(half width, R0, theta, dt, a2) of a 1D case."""
    n = case["n"]
    if case["kind"] == "surface" or case["kind"] == "solve1d":    # the paper's test grid, h = 0.1
        hw = 51.2 * n / 1024
        return hw, hw * 40.0 / 51.2, math.pi / 4, (2 * hw / n) ** 2, 2.0
    if case["contour"] == "sharp":                                # the single-instance workload, h = 0.39
        hw = 200.0 * n / 1024
        return hw, 0.75 * hw, 0.5, 0.05, 2.0
    hw = 8.0 * n / 1024                                           # the laser batch, h = 1/64
    return hw, 0.75 * hw, 0.5, 0.02, 2.0


def _prec(case):
    return (S.SOFT_C64, torch.complex64) if case["prec"] == "c64" else (S.SOFT_C128, torch.complex128)


def _packet(g, x, hw):
    """A bound-looking packet near the centre and broad outgoing ones that
    reach the scaled strips, as a propagated state has."""
    psi = np.exp(-(x - g.uniform(-0.1, 0.1) * hw) ** 2 / (2 * (0.08 * hw) ** 2) + 1j * g.uniform(0, 6.28))
    for s in (-1.0, 1.0):
        k = s * g.uniform(0.3, 1.5)
        psi = psi + 0.3 * np.exp(-(x - s * 0.55 * hw) ** 2 / (2 * (0.25 * hw) ** 2) + 1j * k * x
                                 + 1j * g.uniform(0, 6.28))
    return psi


def _batch_problem(case, seed):
    sizes = [int(v) for v in case["sizes"].split(",")]
    ns = [int(v) for v in np.random.default_rng(1505).choice(sizes, size=case["count"])]
    E0 = np.random.default_rng(seed).uniform(0.01, 0.1, size=case["count"])
    return ns, E0


def _batch_states(case, seed, ns):
    """Packed complex128 state on the device, size by size."""
    off = np.concatenate([[0], np.cumsum(ns)])
    psi = torch.zeros(int(off[-1]), dtype=torch.complex128, device=DEV)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    for n in sorted(set(ns)):
        idx = [i for i, v in enumerate(ns) if v == n]
        hw = 8.0 * n / 1024
        x = torch.as_tensor(_axis(n, hw)[0], device=DEV)[None, :]
        u = torch.rand((len(idx), 6), dtype=torch.float64, device=DEV, generator=gen)
        s = (1.0 + u[:, 0:1]) * min(1.0, hw / 16)
        v = torch.exp(torch.complex(-x ** 2 / (2 * s * s), 6.28 * u[:, 1:2].expand(-1, n)))
        for sg, c in ((-1.0, 2), (1.0, 4)):
            k = sg * (0.3 + 1.2 * u[:, c:c + 1])
            v = v + 0.3 * torch.exp(torch.complex(-(x - sg * 0.55 * hw) ** 2 / (2 * (0.25 * hw) ** 2),
                                                  k * x + 6.28 * u[:, c + 1:c + 2]))
        st = torch.as_tensor([int(off[i]) for i in idx], device=DEV)[:, None]
        psi[(st + torch.arange(n, device=DEV)[None, :]).reshape(-1)] = v.reshape(-1)
    return psi, off


def _grid_axes(case):
    """Per axis (x fastest): (n, half width, R0); theta, dt, a2."""
    if case["kind"] == "cube":
        h, names = 80.0 / 256, ("nx", "ny", "nz")
    else:
        h, names = 400.0 / (1024 if case["kind"] == "krylov2d" else 2048), ("nx", "ny")
    # one box for all axes (a power of 2 times the workload's, so that R0 is a cell edge on each)
    hw = 0.5 * h * 2 ** round(sum(math.log2(case[k]) for k in names) / len(names))
    return [(case[k], hw) for k in names], 0.75 * hw, 0.4, 0.02, 1.0


def _grid_state(case, seed):
    g = np.random.default_rng(seed)
    axes = _grid_axes(case)[0]
    psi = None
    for _ in range(4):
        f = torch.ones([1] * len(axes), dtype=torch.complex128, device=DEV)
        for d, (n, hw) in enumerate(axes):
            x = torch.as_tensor(_axis(n, hw)[0], device=DEV)
            w = g.uniform(0.08, 0.3) * hw
            v = torch.exp(torch.complex(-(x - g.uniform(-0.25, 0.25) * hw) ** 2 / (2 * w * w), g.uniform(-1.5, 1.5) * x))
            f = f * v.reshape([-1 if e == d else 1 for e in reversed(range(len(axes)))])
        psi = f if psi is None else psi + f
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    noise = torch.randn(psi.shape + (2,), dtype=torch.float64, device=DEV, generator=gen)
    return psi + 1e-3 * torch.view_as_complex(noise)


def _nn_inputs(case, seed):
    g = np.random.default_rng(seed)
    F, H, W = case["fields"], case["height"], case["width"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    z = torch.fft.fft2(torch.randn((2, F, H, W), dtype=torch.complex64, device=DEV, generator=gen))
    ky = torch.fft.fftfreq(H, device=DEV)[:, None]
    kx = torch.fft.fftfreq(W, device=DEV)[None, :]
    z = torch.fft.ifft2(z * torch.exp(-60.0 * (kx ** 2 + ky ** 2)))
    z = z / z.abs().square().mean(dim=(-2, -1), keepdim=True).sqrt() * math.sqrt(2.0)
    w = np.concatenate([g.standard_normal(576) * math.sqrt(2 / 18), 0.05 * g.standard_normal(32),
                        g.standard_normal(9216) * math.sqrt(2 / 288), 0.05 * g.standard_normal(32),
                        0.1 * g.standard_normal(576) * math.sqrt(2 / 288), np.zeros(2)]).astype(np.float32)
    return z[0].contiguous(), (0.1 * z[1]).contiguous(), w


def _solve_energies(case):
    return [0.5 * k * k for k in np.linspace(0.2, 6.0, case["energies"] + 1)[:case["energies"]]]


def _solve_rhs(case, seed):
    """The paper's packet (v0 = 2) spread freely up to t = 20, seeded phase."""
    hw = _box(case)[0]
    g = np.random.default_rng(seed)
    x = _axis(case["n"], hw)[0] / (hw / 51.2)
    s = 1.0 + 20.0j
    v = (math.pi ** -0.25 / np.sqrt(s) * np.exp(-(x - 40.0) ** 2 / (2 * s) + 2j * x - 40.0j)
         + 0.2 * np.exp(-(x + 10.0 * g.uniform(-1, 1)) ** 2 / 18))
    return v * np.exp(6.28j * g.uniform())


def _krylov_vectors(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    v = torch.view_as_complex(torch.randn((2, case["ny"], case["nx"], 2), dtype=torch.float64, device=DEV,
                                          generator=gen))
    return _grid_state(case, seed) + 0.1 * v[0], v[1].contiguous(), 0.05 + 1.95 * float(
        np.random.default_rng(seed).uniform())


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    g = np.random.default_rng(seed)
    if kind == "step1d":
        hw, R0, th, dt, a2 = _box(case)
        sp, tt = _prec(case)
        plan = S.Plan(S.soft_create(case["n"], (-hw, hw), R0, th, dt, prec=sp, contour=CONTOURS[case["contour"]],
                                    soft_a2=a2))
        psi = torch.as_tensor(_packet(g, _axis(case["n"], hw)[0], hw)).to(DEV, tt)
        return dict(case=case, plan=plan, psi=psi, t=T_PULSE,
                    field=(float(g.uniform(0.01, 0.1)), OMEGA, NCYC) if case["field"] else None)
    if kind == "surface":
        hw, R0, th, dt, a2 = _box(case)
        plan = S.Plan(S.soft_create(case["n"], (-hw, hw), R0, th, dt, prec=S.SOFT_C128,
                                    contour=S.CONTOUR_TFECS, charge=0.0))
        psi = torch.as_tensor(_packet(g, _axis(case["n"], hw)[0], hw)).to(DEV)
        samples = torch.zeros((case["steps"] + 1, 4), dtype=torch.complex128, device=DEV)
        return dict(case=case, plan=plan, psi=psi, t=0.0, samples=samples)
    if kind == "batch":
        ns, E0 = _batch_problem(case, seed)
        sp, tt = _prec(case)
        hws = [8.0 * n / 1024 for n in ns]
        plan = S.Plan(S.soft_create_batch(ns, [(-w, w) for w in hws], [0.75 * w for w in hws], [0.5] * len(ns),
                                          [(float(e), OMEGA, NCYC) for e in E0], 0.02, prec=sp,
                                          contour=S.CONTOUR_SECS, soft_a2=2.0))
        return dict(case=case, plan=plan, psi=_batch_states(case, seed, ns)[0].to(tt), t=T_PULSE)
    if kind in ("plane", "cube", "krylov2d"):
        axes, R0, th, dt, a2 = _grid_axes(case)
        sp, tt = _prec(case) if kind != "krylov2d" else (S.SOFT_C128, torch.complex128)
        box = tuple(v for _, hw in axes for v in (-hw, hw))
        plan = S.Plan(S.soft_create(tuple(n for n, _ in axes), box, R0, th, dt, prec=sp, soft_a2=a2))
        if kind == "krylov2d":
            p, r, E = _krylov_vectors(case, seed)
            return dict(case=case, plan=plan, p=p, r=r, E=E, w=torch.zeros_like(p), z=torch.zeros_like(p))
        return dict(case=case, plan=plan, psi=_grid_state(case, seed).to(tt).contiguous(), t=0.0)
    if kind == "solve1d":
        hw, R0, th, dt, a2 = _box(case)
        plan = S.Plan(S.soft_create(case["n"], (-hw, hw), R0, th, dt, prec=S.SOFT_C128, contour=S.CONTOUR_SECS,
                                    charge=case["charge"], soft_a2=a2))
        rhs = torch.as_tensor(_solve_rhs(case, seed)).to(DEV)
        return dict(case=case, plan=plan, E=_solve_energies(case), rhs=rhs,
                    x=torch.zeros((case["energies"], case["n"]), dtype=torch.complex128, device=DEV))
    plan = S.Plan(S.soft_create((256, 256), (-40.0, 40.0, -40.0, 40.0), 30.0, 0.4, 0.02))
    x, t, w = _nn_inputs(case, seed)
    S.sse_nn_set_weights(plan.h, w)
    return dict(case=case, plan=plan, x=x, t=t)


# ----------------------------------------------------------------------- run
def run(state):
    case, h = state["case"], state["plan"].h
    kind = case["kind"]
    if kind in ("step1d", "plane", "cube"):
        state["t"] = S.soft_step(h, state["psi"], case["steps"], state["t"], field=state.get("field"))
        return state["psi"]
    if kind == "surface":
        state["t"] = S.soft_step_surface(h, state["psi"], case["steps"], state["t"], state["samples"])
        return state["psi"], state["samples"]
    if kind == "batch":
        state["t"] = S.soft_step_batch(h, state["psi"], case["steps"], state["t"])
        return state["psi"]
    if kind == "solve1d":
        S.sse_pcg_solve(h, state["E"], state["rhs"], state["x"], tol=1e-12, maxit=1000, precond=1)
        return state["x"]
    if kind == "krylov2d":
        S.sse_apply_A(h, state["E"], state["p"], state["w"])
        S.sse_apply_precond(h, state["E"], 1, state["r"], state["z"])
        return state["w"], state["z"]
    loss, grad = S.sse_nn_grad(h, state["x"], state["t"])
    return loss, grad


# ---------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; the operations of the FFTs
    (5 N log2 N each, two per axis and step), the phase factors and the
    Crank-Nicolson rows."""
    kind = case["kind"]
    cs = 8 if case.get("prec") == "c64" else 16
    fft = lambda n: 10.0 * math.log2(n)
    if kind in ("step1d", "surface", "batch"):
        if kind == "batch":
            ns = _batch_problem(case, 0)[0]
        else:
            ns = [case["n"]]
        field = 6 if case.get("field", kind == "batch") else 0
        pts = sum(ns)
        fl = case["steps"] * sum(n * (fft(n) + 12 + field + 8) for n in ns)
        by = 2 * cs * pts
        if kind == "surface":
            fl += case["steps"] * 32 * pts
            by += 64 * (case["steps"] + 1)
        return {"bytes": by, "flops": fl}
    if kind in ("plane", "cube"):
        ax = _grid_axes(case)[0]
        pts = math.prod(n for n, _ in ax)
        fl = case["steps"] * pts * (sum(fft(n) + 6 + 8 for n, _ in ax) + 12)
        return {"bytes": pts * (2 * cs + cs), "flops": fl}
    if kind == "krylov2d":
        pts = case["nx"] * case["ny"]
        # A: one FFT pair per axis, the factors, C and U - E; P^-1: the same
        # FFT pairs, two band products of ten terms per axis, the division
        fl = pts * (2 * (fft(case["nx"]) + fft(case["ny"])) + 2 * 2 + 8 + 4 * 80 + 16)
        return {"bytes": pts * 16 * 5, "flops": fl}
    if kind == "solve1d":
        n, nE = case["n"], case["energies"]
        # about 30 iterations of an A and a preconditioner application
        return {"bytes": 16 * n * (1 + nE), "flops": nE * 30 * n * (2 * fft(n) + 160 + 60)}
    px = case["fields"] * case["height"] * case["width"]
    # three layers forward, the data gradients of two, the weight gradients of three
    return {"bytes": px * 16 + 4 * S.NN_PARAMS * 2, "flops": px * 2 * (3 * 576 * 2 + 3 * 9216 - 576)}


# --------------------------------------------------------------------- exact
def _kvec(n, hw):
    m = np.arange(n)
    return np.where(m < n // 2, 2 * np.pi * m / (2 * hw), -2 * np.pi * (n - m) / (2 * hw))


def _q(x, contour, R0, hw, theta):
    ax = np.abs(x)
    q = np.ones(len(x), dtype=np.complex128)
    o = ax > R0
    if contour == "sharp":
        q[o] = np.exp(1j * theta)
    elif contour == "secs":
        q[o] = np.exp(1j * theta * (ax[o] - R0) / (hw - R0))
    else:
        s = (ax[o] - R0) / (hw - R0)
        with np.errstate(divide="ignore", invalid="ignore"):
            q[o] = np.sqrt(1 + 0.5j * ((1 - s) ** -2.0 - (1 + s) ** -2.0 - 4 * s))
    return q


def _z(x, contour, R0, hw, theta):
    ax, z = np.abs(x), x.astype(np.complex128)
    o = ax > R0
    if contour == "sharp":
        z[o] = np.sign(x[o]) * (R0 + np.exp(1j * theta) * (ax[o] - R0))
    elif contour == "secs":
        c = 1j * theta / (hw - R0)
        z[o] = np.sign(x[o]) * (R0 + (np.exp(c * (ax[o] - R0)) - 1) / c)
    return z


def _cmat(n, hw, contour, R0, theta):
    """C = K_s - K_FD as (sub, diag, sup), periodic."""
    x, h = _axis(n, hw)
    qi = _q(x, contour, R0, hw, theta) ** -0.5
    qm = _q(x + 0.5 * h, contour, R0, hw, theta)
    iq = np.zeros(n, dtype=np.complex128)
    f = np.isfinite(qm)
    iq[f] = 1 / qm[f]
    c = -0.5 / (h * h)
    sup = c * qi * np.roll(qi, -1) * iq - c
    sub = c * qi * np.roll(qi, 1) * np.roll(iq, 1) - c
    return sub, -c * qi * qi * (iq + np.roll(iq, 1)) + 2 * c, sup


def _cn(n, hw, contour, R0, theta, dt):
    """The non-zero rows of C and (1 + i dt C/2)^-1 (1 - i dt C/2) on them."""
    sub, diag, sup = _cmat(n, hw, contour, R0, theta)
    rows = np.nonzero(np.abs(sub) + np.abs(diag) + np.abs(sup))[0]
    pos = {int(r): i for i, r in enumerate(rows)}
    C = np.zeros((len(rows), len(rows)), dtype=np.complex128)
    for i, r in enumerate(rows):
        C[i, i] += diag[r]
        for d, v in ((-1, sub[r]), (1, sup[r])):
            j = pos.get((int(r) + d) % n)
            if j is not None:
                C[i, j] += v
    C = torch.as_tensor(0.5j * dt * C, device=DEV)
    one = torch.eye(len(rows), dtype=torch.complex128, device=DEV)
    return torch.as_tensor(rows, device=DEV), torch.linalg.solve(one + C, one - C)


def _apply_cn(v, cn, dim):
    rows, M = cn
    if len(rows) == 0:
        return v
    w = v.movedim(dim, -1).clone()
    w[..., rows] = w[..., rows] @ M.T
    return w.movedim(-1, dim)


def _field(t, E0):
    T = NCYC * 2 * math.pi / OMEGA
    return E0 * math.sin(math.pi * t / T) ** 2 * math.sin(OMEGA * t) if 0 <= t <= T else 0.0 * E0


def _exact_1d(psi, n, hw, contour, R0, theta, dt, a2, charge, steps, t0, E0=None, sample=False):
    """psi [B][n] advanced by `steps`; E0: field amplitudes [B] or None."""
    x, h = _axis(n, hw)
    k = _kvec(n, hw)
    cn = _cn(n, hw, contour, R0, theta, dt)
    U = -charge / np.sqrt(_z(x, contour, R0, hw, theta) ** 2 + a2) if charge else np.zeros(n, dtype=np.complex128)
    Vh = torch.as_tensor(np.exp(-0.5j * dt * U), device=DEV)
    Kh = torch.as_tensor(np.exp(-0.25j * dt * k * k), device=DEV)
    xc = torch.as_tensor(np.clip(x, -R0, R0), device=DEV)
    rows = None
    if sample:
        rows = []
        for xs in (R0, -R0):
            e = np.exp(1j * k * (xs - x[0])) / n
            rows += [e, 1j * k * e]
        rows = torch.as_tensor(np.array(rows), device=DEV)
    c = torch.fft.fft(psi)
    out = [] if rows is None else [c @ rows.T]
    for s in range(steps):
        v = torch.fft.ifft(c * Kh)
        V = Vh
        if E0 is not None:
            f = 0.5 * dt * _field(t0 + (s + 0.5) * dt, E0)
            V = Vh * torch.exp(-1j * f[:, None] * xc[None, :])
        v = _apply_cn(v * V, cn, -1) * V
        c = torch.fft.fft(v) * Kh
        if rows is not None:
            out.append(c @ rows.T)
    return torch.fft.ifft(c), out


def _exact_grid(case, seed):
    axes, R0, th, dt, a2 = _grid_axes(case)
    psi = _grid_state(case, seed).to(_prec(case)[1]).to(torch.complex128)
    nd = len(axes)
    shp = lambda d: [-1 if e == d else 1 for e in reversed(range(nd))]
    zz, K, cns = a2 + 0.0j, 0.0, []
    for d, (n, hw) in enumerate(axes):
        x = _axis(n, hw)[0]
        zz = zz + torch.as_tensor(_z(x, "sharp", R0, hw, th) ** 2, device=DEV).reshape(shp(d))
        K = K + torch.as_tensor(_kvec(n, hw) ** 2, device=DEV).reshape(shp(d))
        cns.append((_cn(n, hw, "sharp", R0, th, dt), nd - 1 - d))
    Vh = torch.exp(0.5j * dt / torch.sqrt(zz))
    Kh = torch.exp(-0.25j * dt * K)
    c = torch.fft.fftn(psi)
    for _ in range(case["steps"]):
        v = torch.fft.ifftn(c * Kh) * Vh
        for cn, dim in cns:
            v = _apply_cn(v, cn, dim)
        c = torch.fft.fftn(v * Vh) * Kh
    return torch.fft.ifftn(c)


def _bands(n, width=10):
    npos = n // 2 - 1
    q, r = divmod(npos, width)
    ws = [npos] if q == 0 else [width] * (q - 1) + [width + r]
    out, m = [(0, 1)], 1
    for w in ws:
        out.append((m, w))
        m += w
    out.append((m, 1))
    m += 1
    for w in reversed(ws):
        out.append((m, w))
        m += w
    return out


def _band_eig(n, hw, R0, theta):
    """Block-diagonal eigenvectors V, V^-1 and eigenvalues of the banded
    kinetic matrix in the basis e^{ikx}, composed with that basis."""
    x = _axis(n, hw)[0]
    k = _kvec(n, hw)
    q2 = _q(x, "sharp", R0, hw, theta) ** -2.0
    V = np.zeros((n, n), dtype=np.complex128)
    Vi = np.zeros((n, n), dtype=np.complex128)
    lam = np.zeros(n, dtype=np.complex128)
    d = np.arange(-25, 26)
    gd = np.exp(2j * np.pi * np.outer(d, x) / (2 * hw)) @ q2 / n
    for m, w in _bands(n):
        s = slice(m, m + w)
        i = np.arange(w)
        l, v = np.linalg.eig(0.5 * np.outer(k[s], k[s]) * gd[(i[None, :] - i[:, None]) + 25])
        lam[s], V[s, s], Vi[s, s] = l, v, np.linalg.inv(v)
    F = np.exp(1j * np.outer(k, x)) / math.sqrt(n)
    F, V, Vi, lam = (torch.as_tensor(a, device=DEV) for a in (F, V, Vi, lam))
    return F.conj().T @ V, Vi @ F, lam


def _exact_krylov(case, seed):
    axes, R0, th, dt, a2 = _grid_axes(case)
    p, r, E = _krylov_vectors(case, seed)
    zz, w = a2 + 0.0j, 0.0
    for d, (n, hw) in enumerate(axes):
        x, dim = _axis(n, hw)[0], 1 - d
        shp = (1, -1) if d == 0 else (-1, 1)
        zz = zz + torch.as_tensor(_z(x, "sharp", R0, hw, th) ** 2, device=DEV).reshape(shp)
        K = torch.as_tensor(0.5 * _kvec(n, hw) ** 2, device=DEV).reshape(shp)
        sub, diag, sup = (torch.as_tensor(v, device=DEV).reshape(shp) for v in _cmat(n, hw, "sharp", R0, th))
        w = w + torch.fft.ifft(torch.fft.fft(p, dim=dim) * K, dim=dim)
        w = w + sub * p.roll(1, dim) + diag * p + sup * p.roll(-1, dim)
    w = w + (-1.0 / torch.sqrt(zz) - E) * p
    (nx, hx), (ny, hy) = axes
    bx, fx, lx = _band_eig(nx, hx, R0, th)
    by, fy, ly = _band_eig(ny, hy, R0, th)
    z = by @ ((fy @ r @ fx.T) / (ly[:, None] + lx[None, :] - E)) @ bx.T
    return w, z


def _exact_solve1d(case, seed):
    hw, R0, th, dt, a2 = _box(case)
    n = case["n"]
    x = _axis(n, hw)[0]
    eye = torch.eye(n, dtype=torch.complex128, device=DEV)
    K = torch.as_tensor(0.5 * _kvec(n, hw) ** 2, device=DEV)
    A = torch.fft.ifft(torch.fft.fft(eye, dim=0) * K[:, None], dim=0)
    sub, diag, sup = _cmat(n, hw, "secs", R0, th)
    U = -case["charge"] / np.sqrt(_z(x, "secs", R0, hw, th) ** 2 + a2)
    i = torch.arange(n, device=DEV)
    for d, v in ((-1, sub), (0, diag + U), (1, sup)):
        A[i, (i + d) % n] += torch.as_tensor(v, device=DEV)
    f = torch.as_tensor(_solve_rhs(case, seed), device=DEV)
    out = []
    for E in _solve_energies(case):
        lu = torch.linalg.lu_factor(A - E * eye)
        v = torch.linalg.lu_solve(*lu, f[:, None])
        v = v + torch.linalg.lu_solve(*lu, f[:, None] - (A @ v - E * v))     # one refinement
        out.append(v[:, 0])
    return torch.stack(out)


def _exact_grad(case, seed):
    """Inputs, weights and activations rounded to BF16 as the network defines
    them, everything else in 64 bits; gradients by autograd (the rounding
    passes them unchanged)."""
    x, t, w = _nn_inputs(case, seed)
    bf = lambda v: v + (v.detach().to(torch.bfloat16).double() - v.detach())
    P = torch.as_tensor(w, device=DEV).double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(P, [576, 32, 9216, 32, 576, 2])
    total = 2.0 * x.numel()
    loss = torch.zeros((), dtype=torch.float64, device=DEV)

    def conv(v, Wt, b, cin):
        v = torch.nn.functional.pad(v, (1, 1, 1, 1), mode="circular")
        u = torch.nn.functional.unfold(v, 3)
        return (bf(Wt).reshape(-1, cin * 9) @ u).reshape(v.shape[0], -1, v.shape[2] - 2, v.shape[3] - 2) \
            + b[None, :, None, None]

    for f in range(x.shape[0]):
        v = torch.view_as_real(x[f]).double().permute(2, 0, 1)[None]
        v = bf(torch.relu(conv(bf(v), W1, b1, 2)))
        v = bf(torch.relu(conv(v, W2, b2, 32)))
        d = conv(v, W3, b3, 32) - torch.view_as_real(t[f]).double().permute(2, 0, 1)[None]
        part = (d * d).sum() / total
        part.backward(retain_graph=True)
        loss += part.detach()
    return float(loss), P.grad.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    g = np.random.default_rng(seed)
    if kind in ("step1d", "surface"):
        hw, R0, th, dt, a2 = _box(case)
        tt = _prec(case)[1] if kind == "step1d" else torch.complex128
        psi = torch.as_tensor(_packet(g, _axis(case["n"], hw)[0], hw)).to(DEV, tt).to(torch.complex128)[None]
        if kind == "surface":
            v, s = _exact_1d(psi, case["n"], hw, "tfecs", R0, th, dt, a2, 0.0, case["steps"], 0.0, None, True)
            return v[0], torch.cat(s)
        E0 = torch.tensor([float(g.uniform(0.01, 0.1))], dtype=torch.float64, device=DEV) if case["field"] else None
        return _exact_1d(psi, case["n"], hw, case["contour"], R0, th, dt, a2, 1.0, case["steps"], T_PULSE, E0)[0][0]
    if kind == "batch":
        ns, E0 = _batch_problem(case, seed)
        psi, off = _batch_states(case, seed, ns)
        psi = psi.to(_prec(case)[1]).to(torch.complex128)
        for n in sorted(set(ns)):
            idx = [i for i, v in enumerate(ns) if v == n]
            st = torch.as_tensor([int(off[i]) for i in idx], device=DEV)[:, None] + torch.arange(n, device=DEV)
            hw = 8.0 * n / 1024
            e = torch.as_tensor(E0[idx], device=DEV)
            v = _exact_1d(psi[st], n, hw, "secs", 0.75 * hw, 0.5, 0.02, 2.0, 1.0, case["steps"], T_PULSE, e)[0]
            psi[st.reshape(-1)] = v.reshape(-1)
        return psi
    if kind in ("plane", "cube"):
        return _exact_grid(case, seed)
    if kind == "krylov2d":
        return _exact_krylov(case, seed)
    if kind == "solve1d":
        return _exact_solve1d(case, seed)
    return _exact_grad(case, seed)
