"""The losses that training and gradient calls report, call after call: each starts from zero.

Tolerance: the outputs err by some 1e-5 of their scale at most (five layers of K <= 300 in
FP32: 5 x 17 x 6e-8), and the loss is a mean of squares of order one."""
import numpy as np
import pytest

from oracle import mlp
from tests.mlp_util import flat, members

pytestmark = pytest.mark.gpu
SIZES = (6, 128, 128, 33)


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic
    return pic, torch


def _nets(seed):
    return [([w.astype(np.float32).astype(float) for w in W], [v.astype(np.float32).astype(float) for v in b])
            for W, b in members(3, SIZES, seed=seed)]


def _params(nets):
    return np.stack([flat(W, b) for W, b in nets])


def test_losses_of_repeated_calls(env):
    """Each call's losses are its own: the sums start at zero every time."""
    pic, torch = env
    nets = _nets(9)
    rng = np.random.default_rng(4)
    for rows in (1, 40, 300):
        m = pic.pic_mlp_create(3, SIZES, rows)
        pic.pic_mlp_params_set(m, _params(nets))
        x = rng.uniform(-1, 1, (rows, SIZES[0])).astype(np.float32)
        t = rng.normal(0, 0.5, (rows, SIZES[-1])).astype(np.float32)
        X, T = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        want = [mlp.loss(mlp.forward(W, b, x.astype(float))[0], t.astype(float)) for W, b in nets]
        for _ in range(3):
            loss = pic.pic_mlp_grad(m, X, T)[1]
            assert np.abs(loss - want).max() <= 1e-5 * max(want)
        # one training row: every minibatch is that row, and the first step's loss is known
        X1, T1 = X[:1].contiguous(), T[:1].contiguous()
        want = [mlp.loss(mlp.forward(W, b, x[:1].astype(float))[0], t[:1].astype(float)) for W, b in nets]
        for _ in range(3):
            pic.pic_mlp_params_set(m, _params(nets))
            loss = pic.pic_mlp_train(m, X1, T1, batch=rows, steps=1, lr=1e-3, seed=1)
            assert np.abs(loss - want).max() <= 1e-5 * max(want)
