"""FP32 inference reads what the network's parameters are when it runs: replayed from a
recorded graph after the parameters changed, and from two streams right after they were set.
Whole-network kernel (n above 1024) and layer by layer.

Tolerance: as for the FP32 kernels elsewhere, five layers of K <= 300 in FP32 err by some
5 x 17 x 6e-8 of the outputs' scale: 1e-5."""
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


def _check(Y, nets, x):
    for e, (W, b) in enumerate(nets):
        y = mlp.forward(W, b, x.astype(float))[0]
        assert np.abs(Y[e].cpu().numpy() - y).max() <= 1e-5 * np.abs(y).max(), e


@pytest.mark.parametrize("n", [100, 3000])
def test_replay_after_new_parameters(env, n):
    pic, torch = env
    m = pic.pic_mlp_create(3, SIZES, 128)
    first, second = _nets(5), _nets(50)
    pic.pic_mlp_params_set(m, _params(first))
    x = np.random.default_rng(1).uniform(-1, 1, (n, SIZES[0])).astype(np.float32)
    X = torch.from_numpy(x).cuda()
    Y = torch.zeros((3, n, SIZES[-1]), dtype=torch.float32, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        pic.pic_mlp_forward(m, X, out=Y)   # kernels are set up before the capture
        s.synchronize()
        _check(Y, first, x)
        with torch.cuda.graph(graph, stream=s):
            pic.pic_mlp_forward(m, X, out=Y)
    for nets in (first, second, first):
        pic.pic_mlp_params_set(m, _params(nets))
        Y.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        _check(Y, nets, x)
    # trained parameters are the ones read, too
    T = torch.zeros((n, SIZES[-1]), dtype=torch.float32, device="cuda")
    pic.pic_mlp_train(m, X, T, batch=64, steps=5, lr=1e-2, seed=3)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    p = pic.pic_mlp_params_get(m)
    assert np.abs(p - _params(first)).max() > 1e-3
    from tests.mlp_util import unflat
    _check(Y, [unflat(q, SIZES) for q in p], x)


def test_two_streams_after_new_parameters(env):
    pic, torch = env
    m = pic.pic_mlp_create(3, SIZES, 128)
    n = 20_000
    x = np.random.default_rng(2).uniform(-1, 1, (n, SIZES[0])).astype(np.float32)
    X = torch.from_numpy(x).cuda()
    streams = [torch.cuda.Stream() for _ in range(3)]
    Y = [torch.zeros((3, n, SIZES[-1]), dtype=torch.float32, device="cuda") for _ in streams]
    for seed in (7, 70, 700):
        nets = _nets(seed)
        pic.pic_mlp_params_set(m, _params(nets))
        for s, y in zip(streams, Y):
            with torch.cuda.stream(s):
                pic.pic_mlp_forward(m, X, out=y)
        torch.cuda.synchronize()
        for y in Y:
            _check(y, nets, x)
