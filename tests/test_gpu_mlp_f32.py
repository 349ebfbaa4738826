"""FP32 network kernels at the edges of their tiles: layer products in 32 and 64 wide tiles
(ragged rows and widths, unaligned strides, sums longer and shorter than a stage) and whole
networks in one kernel (each width class, narrow outputs, ragged row tiles), against the
FP64 reference.

Tolerances: a sum of K products in FP32 errs by at most K 2^-24 of the sum of their
magnitudes and typically by sqrt(K) 2^-24; over at most five layers of K <= 300 that is
about 5 x 17 x 6e-8 = 5e-6 of the outputs' scale, asserted at 1e-5 (gradients pass the
layers twice and are compared entry by entry with their largest: 1e-4)."""
import numpy as np
import pytest

from oracle import mlp
from tests.mlp_util import flat, unflat, members

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic
    return pic, torch


def case(pic, torch, sizes, members_, rows, max_batch, seed=21):
    m = pic.pic_mlp_create(members_, sizes, max_batch)
    nets = [([w.astype(np.float32).astype(float) for w in W], [v.astype(np.float32).astype(float) for v in b])
            for W, b in members(members_, sizes, seed=seed)]
    pic.pic_mlp_params_set(m, np.stack([flat(W, b) for W, b in nets]))
    rng = np.random.default_rng(seed + 1)
    x = rng.uniform(-1, 1, (rows, sizes[0])).astype(np.float32)
    t = rng.normal(0, 0.5, (rows, sizes[-1])).astype(np.float32)
    return m, nets, x, t, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()


# the last column: the largest batch.  Few rows go layer by layer, many through the
# whole-network kernel; widths above 256 always layer by layer.
@pytest.mark.parametrize("sizes,members_,rows,max_batch", [
    ((6, 256, 256, 33), 2, 1, 256), ((6, 256, 256, 33), 2, 31, 16), ((6, 256, 256, 33), 5, 1025, 256),
    ((1, 1), 1, 1, 1), ((1, 1), 3, 200, 4), ((3, 64, 64, 64), 2, 257, 64), ((64, 16, 17, 1), 2, 600, 64),
    ((5, 100, 128, 33), 3, 130, 32), ((128, 128, 32), 2, 129, 32), ((7, 129, 200, 65), 2, 193, 64),
    ((256, 256), 2, 65, 8), ((6, 300, 33), 2, 77, 32), ((9, 257, 40), 1, 5, 8), ((6, 64, 33), 64, 700, 700),
])
def test_forward_edges(env, sizes, members_, rows, max_batch):
    pic, torch = env
    m, nets, x, _, X, _ = case(pic, torch, sizes, members_, rows, max_batch)
    Y = pic.pic_mlp_forward(m, X).cpu().numpy()
    for e, (W, b) in enumerate(nets):
        y = mlp.forward(W, b, x.astype(float))[0]
        assert np.abs(Y[e] - y).max() <= 1e-5 * max(1e-3, np.abs(y).max()), e


@pytest.mark.parametrize("sizes,members_,rows", [
    ((6, 33), 2, 31), ((6, 100, 33), 3, 33), ((4, 128, 128, 5), 2, 100), ((6, 257, 31, 2), 2, 65),
    ((3, 64, 64, 64, 64, 1), 4, 1), ((6, 256, 256, 33), 64, 64), ((6, 256, 256, 33), 2, 1500),
])
def test_gradient_edges(env, sizes, members_, rows):
    pic, torch = env
    m, nets, x, t, X, T = case(pic, torch, sizes, members_, rows, rows)
    g, loss = pic.pic_mlp_grad(m, X, T)
    for e, (W, b) in list(enumerate(nets))[::max(1, members_ - 1)]:
        y, cache = mlp.forward(W, b, x.astype(float))
        dW, db = mlp.backward(W, cache, y, t.astype(float))
        gW, gb = unflat(g[e], sizes)
        for l in range(len(W)):
            assert np.abs(gW[l] - dW[l]).max() <= 1e-4 * np.abs(dW[l]).max(), (e, l)
            assert np.abs(gb[l] - db[l]).max() <= 1e-4 * np.abs(db[l]).max(), (e, l)
        assert abs(loss[e] - mlp.loss(y, t.astype(float))) <= 1e-5 * mlp.loss(y, t.astype(float))


@pytest.mark.parametrize("sizes,batch", [((6, 33), 32), ((6, 100, 33), 31), ((6, 256, 256, 33), 128),
                                         ((5, 64, 64, 64, 7), 100)])
def test_adam_steps(env, sizes, batch):
    """One training row: every draw is that row, whatever the minibatch.  An Adam step moves
    a parameter by at most lr, by lr g / |g| early on: a gradient known to 1e-4 of its
    layer's largest leaves the direction of at most a few in 1e3 open, so the parameters
    agree within 0.05 lr in the mean square."""
    pic, torch = env
    m, nets, x, t, X, T = case(pic, torch, sizes, 2, 1, batch)
    lr, steps = 1e-3, 4
    pic.pic_mlp_train(m, X, T, batch=batch, steps=steps, lr=lr, seed=3)
    got = pic.pic_mlp_params_get(m)
    for e, (W, b) in enumerate(nets):
        p = W + b
        mom, var = [np.zeros_like(v) for v in p], [np.zeros_like(v) for v in p]
        for k in range(steps):
            y, cache = mlp.forward(W, b, x.astype(float))
            dW, db = mlp.backward(W, cache, y, t.astype(float))
            mlp.adam(p, dW + db, mom, var, k + 1, lr=lr)
        assert np.sqrt(np.mean((got[e] - flat(W, b)) ** 2)) <= 0.05 * lr, e
