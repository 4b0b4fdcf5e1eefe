"""soft_step on a single 1D plan inside a caller's stream capture is refused:
a replay would repeat the recorded call's start time and field.  The capture
stays valid, and neither the plan, the state nor the time has changed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402


@pytest.mark.parametrize("prec", [S.SOFT_C64, S.SOFT_C128])
@pytest.mark.parametrize("n", [128, 1024, 16384])
def test_single_steps_are_not_recorded(n, prec):
    hw = 8.0 * n / 1024
    x = -hw + 2 * hw / n * (np.arange(n) + 0.5)
    psi = torch.tensor(np.exp(-x ** 2 / (0.2 * hw) ** 2 + 0.3j * x), device="cuda")
    psi = psi.to(torch.complex64 if prec == S.SOFT_C64 else torch.complex128)
    plan = S.soft_create(n, (-hw, hw), 0.75 * hw, 0.5, 0.02, prec=prec, contour=S.CONTOUR_SECS)
    calls = [lambda d, s: S.soft_step(plan, d, 3, 1.0, stream=s),
             lambda d, s: S.soft_step(plan, d, 3, 1.0, field=(0.05, 0.5, 3.0), stream=s),
             lambda d, s: S.soft_step_batch(plan, d, 3, 1.0, stream=s)]
    try:
        side = torch.cuda.Stream()
        ref = psi.clone()
        for c in calls:                        # also outside a capture, before and after
            c(ref, None)
        torch.cuda.synchronize()
        d = psi.clone()
        mark = torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            mark += 1.0
            for c in calls:
                with pytest.raises(S.SoftError) as err:
                    c(d, side)
                assert err.value.status == -4
        g.replay()
        torch.cuda.synchronize()
        assert mark.item() == 1.0 and torch.equal(d, psi)
        for c in calls:
            c(d, None)
        torch.cuda.synchronize()
        assert torch.equal(d, ref)
    finally:
        S.soft_destroy(plan)
