"""Packs of several instances per CTA in the persistent batch kernel (named
barriers side by side, part-filled packs): what large batches run where tuning
prefers them, here on a small batch by rebuilding its plan's packs.  Bitwise
the per-size kernels' results."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
import workloads as W  # noqa: E402


@pytest.mark.parametrize("prec", [S.SOFT_C64, S.SOFT_C128])
@pytest.mark.parametrize("cap", [2, 3, 4])
def test_packs_match_per_size_kernels(prec, cap):
    ns = [2048] * 9 + [4096] * 5 + [8192] * 3 + [16384] * 2 + [1024]
    hw = [8.0 * n / 1024 for n in ns]
    rng = np.random.default_rng(cap)
    ns, hw = zip(*[(ns[i], hw[i]) for i in rng.permutation(len(ns))])
    args = (list(ns), [(-w, w) for w in hw], [0.75 * w for w in hw], [0.5] * len(ns),
            [(float(e), W.W2_OMEGA, W.W2_NCYC) for e in rng.uniform(0.01, 0.1, len(ns))], W.W2_DT)
    psi = np.concatenate([np.exp(-np.linspace(-w, w, n) ** 2 / (0.3 * w) ** 2 + 0.7j * np.linspace(-w, w, n))
                          for n, w in zip(ns, hw)])
    lib = S.load()
    build_packs = lib._ZN9soft_plan11build_packsEm           # soft_plan::build_packs(size_t)
    build_packs.argtypes = [C.c_void_p, C.c_size_t]
    outs = []
    for packed in (True, False):
        plan = S.soft_create_batch(*args, prec=prec, contour=W.W2_CONTOUR, persistent=1 if packed else 0)
        try:
            if packed:
                assert build_packs(plan, cap) == 0
            d = torch.tensor(psi, dtype=torch.complex64 if prec == S.SOFT_C64 else torch.complex128, device="cuda")
            t = 3.0
            for _ in range(2):
                t = S.soft_step_batch(plan, d, 7, t)
            torch.cuda.synchronize()
            # pulse table, time advance, and the persistent kernel beside one size, or five sizes
            assert S.soft_last_launches(plan) == (4 if packed else 7)
            outs.append(d.cpu().numpy())
        finally:
            S.soft_destroy(plan)
    assert np.isfinite(outs[0].view(outs[0].real.dtype)).all()
    assert np.array_equal(outs[0], outs[1])
