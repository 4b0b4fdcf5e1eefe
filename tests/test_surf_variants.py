"""soft_step_surface runs on every plan it takes: the sampled step kernel
exists for each (elements per thread, radix) variant that tuning can give a
single complex128 plan of N = 256 .. 8192."""
import ctypes as C

import numpy as np
import pytest

import paper_1505_06707_gb300 as S


def test_every_variant_is_built_with_samples():
    from paper_1505_06707_gb300 import _build
    lib = C.CDLL(_build.build())
    variants = lib._ZN4soft15soft1d_variantsEiiPiS0_i        # soft::soft1d_variants(int, int, int*, int*, int)
    sampled = lib._ZN4soft21soft1d_surf_supportedEiii        # soft::soft1d_surf_supported(int, int, int)
    sampled.restype = C.c_bool
    missing, total = [], 0
    for logn in range(8, 14):
        le, lr = (C.c_int * 16)(), (C.c_int * 16)()
        for v in range(variants(S.SOFT_C128, logn, le, lr, 16)):
            total += 1
            if not sampled(logn, le[v], lr[v]):
                missing.append((logn, le[v], lr[v]))
    assert total >= 6 and not missing, missing


@pytest.mark.gpu
@pytest.mark.parametrize("n", [256, 512, 1024, 2048, 4096, 8192])
def test_tuned_plans_sample_the_surface(n):
    torch = pytest.importorskip("torch")
    hw = 51.2 * n / 1024
    x = -hw + 2 * hw / n * (np.arange(n) + 0.5)
    psi = np.exp(-x ** 2 / (0.3 * hw) ** 2 + 0.8j * x)
    out = []
    for tune in (0, 1):
        plan = S.soft_create(n, (-hw, hw), 40.0 / 51.2 * hw, 0.6, 0.01, prec=S.SOFT_C128, contour=S.CONTOUR_SECS,
                             charge=0.0, autotune=tune)
        try:
            d = torch.tensor(psi, device="cuda")
            smp = torch.zeros((13, 4), dtype=torch.complex128, device="cuda")
            S.soft_step_surface(plan, d, 12, 0.0, smp)
            torch.cuda.synchronize()
            out.append((d.cpu().numpy(), smp.cpu().numpy()))
        finally:
            S.soft_destroy(plan)
    for a, b in zip(out[0], out[1]):           # as the sampled step against the oracle
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(a)
