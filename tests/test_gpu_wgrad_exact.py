"""Weight and bias gradients of the learned correction (wgrad.cuh) against the
FP64 contraction of the very operands the kernels read.  Every hidden channel
has one tap of weight +-1/2, 1 or 2 (a permutation of the channels between the
hidden layers), so activations and data gradients are exact in BF16, and what is left
is the contraction: the three-term split of FP32 operands, halos, rows across
segments and fields, and the sums.

Tolerances, relative to a gradient's norm.  A weight's sum rounded to FP32 leaves
2^-24 at most, 2.4e-8 in the mean square; the few FP32 additions of a small
field's partial sums another 3e-8 (they average out over many CTAs).  A bias is
one of 2 to 32 numbers, so up to 2^-24 each.  Sums in chains of eight truncating
tensor-core products leave 5.5e-8, operands without the third term of the split
(17 bits) 2e-6.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1505_06707_gb300 as S  # noqa: E402
from oracle import conv as CV  # noqa: E402
from test_gpu_learned import bf16, flat, small_plan, unflat  # noqa: E402

TOL_W, TOL_B = 4.5e-8, 1e-7


def _one_tap(rng, cout, cin, src):
    W = np.zeros((cout, cin, 3, 3))
    for o in range(cout):
        W[o, src[o], rng.integers(3), rng.integers(3)] = rng.choice([-1, 1]) * rng.choice([0.5, 1.0, 2.0])
    return W


def problem(n, h, w, seed):
    rng = np.random.default_rng(seed)
    W1 = _one_tap(rng, 32, 2, rng.permutation(32) % 2)
    W2 = _one_tap(rng, 32, 32, rng.permutation(32))
    W3 = np.zeros((2, 32, 3, 3))
    for c in range(32):
        W3[c % 2, c, rng.integers(3), rng.integers(3)] = rng.choice([-1.0, 1.0])
    params = [[W1, np.zeros(32)], [W2, np.zeros(32)], [W3, np.zeros(2)]]
    # full 24-bit values of magnitude 1/4 .. 1: the BF16 form has the grid 2^-10,
    # on which the sums of 16 channels are exact
    x = (rng.uniform(0.25, 1.0, (n, 2, h, w)) * rng.choice([-1.0, 1.0], (n, 2, h, w))).astype(np.float32)
    t = rng.standard_normal((n, 2, h, w)).astype(np.float32)
    return params, x, t


def reference(params, x, t):
    (W1, _), (W2, _), (W3, _) = params
    z = [np.zeros(32), np.zeros(32), np.zeros(2)]
    h1 = np.maximum(CV.conv3x3(bf16(x), W1, z[0]), 0.0)
    h2 = np.maximum(CV.conv3x3(h1, W2, z[1]), 0.0)
    out = CV.conv3x3(h2, W3, z[2])
    assert np.array_equal(h1, bf16(h1)) and np.array_equal(h2, bf16(h2))
    gout = (np.float32(2.0) / np.float32(out.size)) * (out.astype(np.float32) - t)     # as the loss kernel, in FP32
    g2 = CV.conv3x3_backward(h2, W3, bf16(gout))[0] * (h2 > 0)
    g1 = CV.conv3x3_backward(h1, W2, g2)[0] * (h1 > 0)
    assert np.array_equal(g2, bf16(g2)) and np.array_equal(g1, bf16(g1))
    return [CV.conv3x3_backward(a, W, g.astype(np.float64))[1:]
            for a, W, g in ((x.astype(np.float64), W1, g1), (h1, W2, g2), (h2, W3, gout))]


def errors(n, h, w, seed=0):
    params, x, t = problem(n, h, w, seed)
    plan = small_plan()
    try:
        S.sse_nn_set_weights(plan, flat(params))
        c = lambda v: torch.tensor((v[:, 0] + 1j * v[:, 1]).astype(np.complex64), device="cuda")  # noqa: E731
        g = S.sse_nn_grad(plan, c(x), c(t))[1]
    finally:
        S.soft_destroy(plan)
    return [[np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got, ref)]
            for got, ref in zip(unflat(g), reference(params, x, t))]


@pytest.mark.parametrize("n,h,w", [(1, 3, 128), (1, 5, 256), (3, 17, 128), (2, 131, 128), (2, 131, 256),
                                   (8, 128, 128)])
def test_gradients_of_exact_operands(n, h, w):
    for layer, (ew, eb) in enumerate(errors(n, h, w, 10 * h + w)):
        assert ew < TOL_W and eb < TOL_B, (layer, ew, eb)
