"""The training step's weight-gradient contraction at ragged sizes: fewer
pixels than one shared-memory block of 32, a last block that is part full,
and several blocks per CTA group, against the FP64 oracle."""

import numpy as np
import pytest

from oracle import dwf as O
from oracle import nn as N
from paper_2203_17119_gb300 import inputs
from tests import test_gpu_nn as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,Ls,nrhs", [((2, 2, 2, 2), 2, 1),     # 48 pixels a parity: one full, one half block
                                          ((2, 2, 2, 2), 10, 3),    # 720 = 22.5 blocks
                                          ((6, 4, 2, 4), 8, 2)])
def test_ragged_pixel_counts(dims, Ls, nrhs):
    rng, U, h = T.setup(dims, Ls, nrhs, 29)
    W1, W2 = T.rand_weights(rng, scale=0.2)
    K = T.G.NN()
    K.set_weights(W1, W2)

    def draw():
        return O.parity_part(inputs.gaussian_source(dims, Ls, rng=rng), 1)

    pairs = [(draw(), draw()) for _ in range(nrhs)]
    loss = K.train_step(h, T.odd_gpu([p[0] for p in pairs], dims), T.odd_gpu([p[1] for p in pairs], dims), nrhs,
                        lr=0.0, loss_kind="error")
    g1, g2 = K.last_grad(h)
    L, w1, w2 = N.loss_and_grad(U, pairs, W1, W2)
    # FP32 rounding 6e-8 through sums of up to ~1e3 terms, with a factor of ten
    assert abs(loss - L) <= 2e-5 * abs(L)
    assert np.linalg.norm(g1 - w1) <= 2e-5 * np.linalg.norm(w1)
    assert np.linalg.norm(g2 - w2) <= 2e-5 * np.linalg.norm(w2)
