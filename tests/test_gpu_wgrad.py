"""Weight and bias gradients of the learned correction on the tensor cores at
ragged sizes: fewer rows than CTAs, CTAs whose rows cross segments and fields,
the smallest height, against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import conv as CV  # noqa: E402
from test_gpu_learned import bf16, flat, small_plan, to_chw, unflat  # noqa: E402


@pytest.mark.parametrize("n,h,w", [(1, 3, 128), (1, 5, 256), (3, 17, 128), (2, 131, 128), (2, 131, 256)])
def test_gradients_at_ragged_sizes(n, h, w):
    rng = np.random.default_rng(100 * h + w)
    params = CV.init_params(rng, scale_last=1.0)
    for _, b in params:
        b[:] = 0.1 * rng.standard_normal(b.shape)
    x = (rng.standard_normal((n, h, w)) + 1j * rng.standard_normal((n, h, w))).astype(np.complex64)
    t = (rng.standard_normal((n, h, w)) + 1j * rng.standard_normal((n, h, w))).astype(np.complex64)
    plan = small_plan()
    try:
        S.sse_nn_set_weights(plan, flat(params))
        loss, g = S.sse_nn_grad(plan, torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
        again = S.sse_nn_grad(plan, torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))[1]
    finally:
        S.soft_destroy(plan)
    assert np.array_equal(g, again)               # sums in a fixed order
    lref, gref = CV.loss_and_grads([[bf16(W), b] for W, b in params], bf16(to_chw(x)), to_chw(t))
    assert abs(loss - lref) < 1e-2 * lref
    for got, ref in zip(unflat(g), gref):
        for a, b in zip(got, ref):                # BF16 activations: 8 significant bits, as in test_gpu_learned
            assert np.linalg.norm(a - b) / np.linalg.norm(b) < 6e-2
