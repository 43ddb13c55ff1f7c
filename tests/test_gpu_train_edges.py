"""Gradient pass of the training step at the edges of its sample split (GPU): one sample,
less than a block's share, one tile exactly, ranges that cross runs, several tiles per block.

Tolerance: a sample's forward and backward are chains of at most ~100 FP32 operations,
relative error ~100 x 2^-24 = 6e-6 of the summed magnitudes; sums of random-sign terms are
smaller than those by the square root of their number, here at most sqrt(30000) = 170 times,
over which the errors average likewise: 1e-4 of the largest entry of each array."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_1010_1233_gb300 import learned, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,B", [(1, 1), (1, 7), (3, 59), (2, 88), (1, 176), (1, 177), (7, 100), (40, 500), (3, 10001)])
def test_gradient_over_the_sample_split(R, B):
    w = W.mlp_weights(R + B, out_scale=0.3)
    X = np.stack([W.mlp_inputs(B, 10 + r) for r in range(R)]).astype(np.float32)
    Sp, G = W.correlator_tables(R, 24, 5)
    tr = learned.Trainer(X, learned.gram(Sp, G), 24, w)
    loss, m, grad = tr.loss_and_grad()
    w64 = {k: v.astype(np.float64) for k, v in w.items()}
    L0, g0, _ = omlp.loss_grad(w64, X.astype(np.float64), Sp, G)
    _, m0 = omlp.loss(w64, X.astype(np.float64), Sp, G)
    assert abs(loss - L0) < 1e-5 * abs(L0)
    assert np.abs(m - m0).max() < 1e-5
    for k in w:
        assert np.abs(grad[k] - g0[k]).max() < 1e-4 * np.abs(g0[k]).max() + 1e-9, k
