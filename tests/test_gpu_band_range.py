"""Range of the fixed-point band products in the 1D stationary solver
(pcg_fix.cuh): the line that meets a band row has a norm just below 2^60.8, and
the product's cross sum must stay below 2^63 for every entry of the row.  With
the simple preconditioner (one entry per row) and a source of one Fourier mode
the whole norm sits in a single sample; its phase is chosen, from a model of
the integer product, so that the cross sum is as large as it gets."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402

E0 = 0.37
HALF = 2.0 ** 32


def _halves(v):
    """v = h 2^32 + l, both signed 32-bit."""
    h = np.round(v / HALF)
    return h, v - h * HALF


def _cross(v, w):
    """|cross sums| of fx_mul<2> / 2^63, v in units (modulus up to 2^60.8), w a factor."""
    (ah, al), (bh, bl) = _halves(4 * v.real), _halves(4 * v.imag)
    (wx, wy), (wz, ww) = _halves(w.real * 2.0 ** 62), _halves(w.imag * 2.0 ** 62)
    m = ah * wy + al * wx - bh * ww - bl * wz
    n = ah * ww + al * wz + bh * wy + bl * wx
    return np.maximum(np.abs(m), np.abs(n)) / 2.0 ** 63


@pytest.mark.parametrize("n", [256, 512, 1024, 2048])
def test_one_mode_with_the_whole_norm(n):
    hw = 51.2 * n / 1024
    R0 = 40.0 * n / 1024
    h = 2 * hw / n
    x0 = -hw + 0.5 * h
    k = 2 * np.pi * np.fft.fftfreq(n, h)
    rng = np.random.default_rng(n)
    # backward row of mode m: e^{-i k x0}, times sqrt(2) where the FFT's half bit goes with the table
    phase = rng.uniform(0, 2 * np.pi, 4096)
    cases = []
    for m in range(1, n):
        w = np.sqrt(2.0) * np.exp(-1j * k[m] * x0)
        v = np.round(2.0 ** 60.79 * np.exp(1j * phase) / 2 ** 8) * 2 ** 8
        c = _cross(v, w)
        i = int(np.argmax(c))
        cases.append((float(c[i]), m, phase[i]))
    cases.sort(reverse=True)
    assert cases[0][0] > 1.0                   # some pair would not fit at modulus sqrt(2)
    plan = S.soft_create(n, (-hw, hw), R0, 0.6, 0.02, prec=S.SOFT_C128, contour=S.CONTOUR_SECS, soft_a2=2.0)
    j = np.arange(n)
    try:
        for _, m, ph in cases[:24]:
            lam = 0.5 * k[m] ** 2 - E0
            # c = F r / (lambda - E) is 2^0.79 e^{i ph} in mode m and 0 elsewhere
            c = 2.0 ** 0.79 * np.exp(1j * (ph - k[m] * x0)) * np.sign(lam)
            r = c * abs(lam) * np.exp(-2j * np.pi * ((m * j) % n) / n) / np.sqrt(n)
            z = torch.zeros(n, dtype=torch.complex128, device="cuda")
            S.sse_apply_precond(plan, E0, 0, torch.tensor(r, device="cuda"), z)
            # the mode's own amplitude (roundings in the modes near E0 are amplified by lambda - E0)
            got = np.vdot(r, z.cpu().numpy()) / np.vdot(r, r).real * lam
            assert abs(got - 1) < 1e-12, (m, got)      # as the other preconditioner tests; a wrap leaves 2e-9
    finally:
        S.soft_destroy(plan)
