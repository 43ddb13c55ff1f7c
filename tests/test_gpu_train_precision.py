"""Range and precision of the gradient of the training step (csrc/mlp_train.cu, GPU).

With W3 = 0 the outputs are s_c = 1 + b3_c for every input, and with a Gram matrix H = 0 the loss is
linear in <s_c^2>: dL/ds_c of a sample is d_rc s_c with d_rc = 4 g_rc / (R 6 K B), so that the gradients of
W3 and b3 are sums of known factors."""
import math

import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_1010_1233_gb300 import learned, workloads as W

pytestmark = pytest.mark.gpu


def _gradient(X, g, w, K):
    """(gradient, d) for the slopes g (R, 6) of the loss."""
    R, B = X.shape[:2]
    gram = np.zeros((R, 43))
    gram[:, 1:7] = g
    _, _, grad = learned.Trainer(X, torch.tensor(gram, device="cuda"), K, w).loss_and_grad()
    return grad, (1.0 / (float(R) * 6 * K)) * (2.0 * g) * 2.0 / B


@pytest.mark.parametrize("d,s", [(1e-42, 2.0 ** 20), (3e-45, 2.0 ** 40), (1e-30, 1.0), (1e40, 2.0 ** -20)])
def test_loss_slopes_outside_fp32(d, s):
    # d_rc has FP64's range and precision; only the product d s is rounded to FP32.  Tolerance: hidden
    # layers of ~70 FP32 operations, 70 x 2^-24 = 4e-6 of the largest value, and sums of one sign.
    R, B, K = 2, 50, 7
    X = np.stack([W.mlp_inputs(B, r) for r in range(R)]).astype(np.float32)
    w = W.mlp_weights(3, out_scale=0.0)
    w["W3"][:] = 0
    w["b3"][:] = s - 1
    g = np.outer([1.0, 0.7], [1, -1, 0.5, 2, -0.25, 1]) * d * R * 6 * K * B / 4
    grad, d = _gradient(X, g, w, K)
    w64 = {k: v.astype(np.float64) for k, v in w.items()}
    h1 = np.maximum(X.astype(np.float64) @ w64["W1"].T + w64["b1"], 0)
    h2 = np.maximum(h1 @ w64["W2"].T + w64["b2"], 0)
    for name, want in (("b3", B * s * d.sum(0)), ("W3", s * np.einsum("rc,rbh->ch", d, h2))):
        assert np.abs(grad[name] - want).max() <= 1e-5 * np.abs(want).max(), name


@pytest.mark.parametrize("pairs,B", [(1000, 8), (3, 900), (200, 177)])
def test_cancelling_sums(pairs, B):
    # Runs in pairs of opposite slopes and almost the same inputs, so that each gradient of W3 is 10^-6 to
    # 10^-9 of the sum of its terms' magnitudes.  Hidden unit h passes input h % 3 through (positive
    # inputs, one-hot weights), so a term is the product of two known FP32 numbers and math.fsum of the
    # FP64 products is the exact sum.
    # Tolerance: half an ulp for the rounding to FP32, and of the sum of magnitudes gamma_n^2 for Dot2 on n
    # terms (Ogita, Rump & Oishi, Prop. 5.5; gamma_n = n 2^-24 / (1 - n 2^-24)) and 2^-53 per FP64 addition
    # of the blocks' two partials.  n: half of a block's samples, in groups of four.
    R, N = 2 * pairs, 2 * pairs * B
    rng = np.random.default_rng(pairs + B)
    X = np.exp2(rng.uniform(-12, 6, (pairs, 2, B, 3))).astype(np.float32)
    X[:, 1] = X[:, 0, ::-1]
    few = rng.integers(0, B, pairs)
    X[np.arange(pairs), 1, few] = np.nextafter(X[np.arange(pairs), 1, few], np.float32(np.inf))
    X = X.reshape(R, B, 3)
    w = {k: np.zeros_like(v) for k, v in W.mlp_weights(1).items()}
    for h in range(32):
        w["W1"][h, h % 3] = 1
        w["W2"][h, h] = 1
    g = np.tile(rng.uniform(0.5, 2, (pairs, 6)), 2).reshape(R, 6) * np.tile([[1.0], [-1.0]], (pairs, 1))
    grad, d = _gradient(X, g, w, 11)
    d = d.astype(np.float32).astype(np.float64)                      # dL/ds at s = 1
    blocks = min(304, -(-N // 64))
    n = 4 * (-(-(-(-N // blocks)) // 8)) + 4
    gamma = n * 2.0 ** -24 / (1 - n * 2.0 ** -24)
    for c in range(6):
        for h in range(3):
            t = (d[:, None, c] * X[:, :, h].astype(np.float64)).ravel()
            want, size = math.fsum(t), np.abs(t).sum()
            assert abs(want) < 1e-6 * size
            tol = 2.0 ** -24 * abs(want) + (gamma * gamma + (2 * blocks + 16) * 2.0 ** -53) * size
            assert (np.abs(grad["W3"][c, h::3] - want) <= tol).all(), (c, h, grad["W3"][c, h::3], want, tol)


@pytest.mark.parametrize("R,B", [(64, 3), (65, 3), (700, 2), (3000, 1)])
def test_many_runs(R, B):
    # the loss pass over several blocks from 65 runs on, against the FP64 oracle.  Tolerance: as for the
    # gradient over the sample split (100 FP32 operations a sample, averaged over the sum's terms)
    w = W.mlp_weights(R, out_scale=0.3)
    X = np.stack([W.mlp_inputs(B, 10 + r) for r in range(R)]).astype(np.float32)
    Sp, G = W.correlator_tables(R, 4, 5)
    tr = learned.Trainer(X, learned.gram(Sp, G), 4, w)
    loss, m, grad = tr.loss_and_grad()
    w64 = {k: v.astype(np.float64) for k, v in w.items()}
    L0, g0, _ = omlp.loss_grad(w64, X.astype(np.float64), Sp, G)
    _, m0 = omlp.loss(w64, X.astype(np.float64), Sp, G)
    assert abs(loss - L0) < 1e-5 * abs(L0)
    assert np.abs(m - m0).max() < 1e-5
    for k in w:
        assert np.abs(grad[k] - g0[k]).max() < 1e-4 * np.abs(g0[k]).max() + 1e-9, k
