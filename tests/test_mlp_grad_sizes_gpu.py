"""The network gradient (csrc/mlp.cuh) around the samples of a CTA (64) and of the reduction's slices (8 CTAs).

Against the oracle's FP64 backprop, per parameter block (weights and biases
of each layer) to 1e-4 of the block's norm: a product read in the wrong
order or a missed sample changes a block by a share of order 1/n or more.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

BLOCKS = np.cumsum([0, 384, 64, 4096, 64, 64, 1])


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 511, 512, 513, 577, 4097])
def test_sizes(hydro_lib, n):
    rng = np.random.default_rng(n)
    w = (0.3 * rng.standard_normal(hydro_lib.HYDRO_MLP_NPARAM)).astype(np.float32)
    X = rng.normal(size=(n, 6)).astype(np.float32).astype(np.float64)
    T = rng.normal(size=n).astype(np.float32).astype(np.float64)
    loss_o, g_o = O.mlp_loss_grad(w, X, T)
    loss, g = hydro_lib.hydro_mlp_loss_grad(w, X, T)
    assert abs(loss - loss_o) <= 1e-5 * loss_o
    for a, b in zip(BLOCKS[:-1], BLOCKS[1:]):
        assert np.linalg.norm(g[a:b] - g_o[a:b]) <= 1e-4 * np.linalg.norm(g_o[a:b]), (a, b)
