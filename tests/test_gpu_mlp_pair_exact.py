"""BF16 inference by pairs of SMs where its arithmetic is exact: inputs, biases and sums are
multiples of 16 up to 4096 (eight bits of mantissa), weights are 0 and +-1, and GELU of such
a number is the number itself above zero and 0 from zero down (tanh of 100 and more is 1).
Every output then has one right value, so a bias, a chunk of the weights, a padded row or a
column too many or too few shows as it is, at any width."""
import numpy as np
import pytest

from tests.mlp_util import flat

pytestmark = pytest.mark.gpu


def exact_net(rng, sizes):
    """Each unit takes one input of its own (all inputs are taken) minus another, and a bias."""
    Ws, bs = [], []
    for k, n in zip(sizes[:-1], sizes[1:]):
        W = np.zeros((n, k))
        take = np.concatenate([rng.permutation(k) for _ in range(-(-n // k))])[:n]
        W[np.arange(n), take] = 1.0
        less = rng.integers(0, k, n)
        W[np.arange(n), less] -= less != take
        Ws.append(W)
        bs.append(16.0 * rng.integers(-1, 3, n))
    return Ws, bs


def exact_forward(Ws, bs, x):
    top = np.abs(x).max()
    for l, (W, b) in enumerate(zip(Ws, bs)):
        x = x @ W.T + b
        top = max(top, np.abs(x).max())
        if l < len(Ws) - 1:
            x = np.maximum(x, 0.0)
    assert top <= 4096
    return x


@pytest.mark.parametrize("sizes,counts", [
    ((6, 256, 256, 33), (1, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1025)),
    ((130, 129, 127, 1), (1, 300)),
    ((256, 256, 256), (600,)),
    ((1, 1, 1), (513,)),
    ((3, 16, 5), (25601, 40000)),   # several tiles a pair, an odd last one
    ((17, 33, 31, 161, 65), (640,)),
    ((5,) + (48,) * 15 + (2,), (270,)),
])
@pytest.mark.parametrize("members", [1, 5])
def test_pair_exact(sizes, counts, members):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic
    rng = np.random.default_rng(77)
    m = pic.pic_mlp_create(members, sizes, 256)
    nets = [exact_net(rng, sizes) for _ in range(members)]
    pic.pic_mlp_params_set(m, np.stack([flat(W, b) for W, b in nets]))
    for n in counts:
        x = 16.0 * rng.integers(-3, 4, (n, sizes[0]))
        Y = pic.pic_mlp_forward(m, torch.tensor(x, dtype=torch.float32, device="cuda"), tensor_cores=True)
        for e, (W, b) in enumerate(nets):
            assert np.array_equal(Y[e].cpu().numpy(), exact_forward(W, b, x)), (n, e)
