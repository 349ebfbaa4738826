"""Training's products of a batch in one kernel: rows around each count of rows a cluster
takes (8, 16, 24) and past what one round of clusters holds, widths at the edges of the
quarters of 64 columns, the slices of 32 k and the 16-byte copies, one layer and sixteen.

Gradients against the FP64 reference: sums of at most 256 products in FP32 over at most
sixteen layers and back, 32 x 16 x 2^-24 = 3e-5 of a layer's largest; asserted at 1e-4."""
import numpy as np
import pytest

from oracle import mlp
from tests.mlp_util import unflat
from tests.test_gpu_mlp_f32 import case, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,members,rows", [
    ((6, 256, 255, 33), 4, 71), ((6, 256, 255, 33), 4, 72), ((6, 256, 255, 33), 4, 73),
    ((6, 256, 255, 33), 4, 145), ((6, 256, 255, 33), 4, 216), ((6, 256, 255, 33), 4, 217),
    ((1, 1, 1), 1, 1), ((256, 3), 2, 9), ((3, 65, 129, 61, 2), 2, 25), ((5, 31, 64, 253, 4), 3, 17),
    ((4,) + (40,) * 15 + (3,), 2, 50), ((256,) * 4, 1, 8),
])
def test_gradients(env, sizes, members, rows):
    pic, torch = env
    m, nets, x, t, X, T = case(pic, torch, sizes, members, rows, rows + 3)
    g, loss = pic.pic_mlp_grad(m, X, T)
    for e, (W, b) in enumerate(nets):
        y, cache = mlp.forward(W, b, x.astype(float))
        dW, db = mlp.backward(W, cache, y, t.astype(float))
        gW, gb = unflat(g[e], sizes)
        for l in range(len(W)):
            assert np.abs(gW[l] - dW[l]).max() <= 1e-4 * np.abs(dW[l]).max(), (e, l)
            assert np.abs(gb[l] - db[l]).max() <= 1e-4 * np.abs(db[l]).max(), (e, l)
        assert abs(loss[e] - mlp.loss(y, t.astype(float))) <= 1e-5 * mlp.loss(y, t.astype(float))
