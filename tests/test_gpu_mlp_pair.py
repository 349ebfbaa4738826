"""BF16 inference by pairs of SMs (two tiles of 256 samples a pair): sample counts around the
128-row halves and the 256-row tiles, and widths around the padding of a layer to 32 (half
in each SM), the 128-wide weight chunks and a first layer of several chunks."""
import numpy as np
import pytest

from oracle import mlp
from tests.mlp_util import flat, members

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic
    return pic


@pytest.mark.parametrize("sizes,counts", [
    ((6, 256, 256, 33), (127, 128, 129, 255, 256, 257, 384, 385, 511, 512, 513, 1025)),
    ((130, 129, 127, 1), (1, 300)),
    ((256, 256, 256), (600,)),
    ((1, 1, 1), (513,)),
    ((3, 16, 5), (25601, 40000)),   # several tiles a pair, an odd last one
    ((17, 33, 31, 161, 65), (640,)),
    ((5,) + (48,) * 15 + (2,), (270,)),
])
def test_pair_edges(pic, sizes, counts):
    import torch
    E = 2
    m = pic.pic_mlp_create(E, sizes, 256)
    nets = members(E, sizes, seed=51)
    pic.pic_mlp_params_set(m, np.stack([flat(W, b) for W, b in nets]))
    for n in counts:
        x = np.random.default_rng(52 + n).uniform(-1, 1, (n, sizes[0]))
        out = torch.full((E, n + 8, sizes[-1]), 7.0, dtype=torch.float32, device="cuda")
        flat_out = out.view(-1)[: E * n * sizes[-1]].view(E, n, sizes[-1])
        pic.pic_mlp_forward(m, torch.tensor(x, dtype=torch.float32, device="cuda"),
                            tensor_cores=True, out=flat_out)
        Y = flat_out.cpu().numpy()
        assert bool((out.view(-1)[E * n * sizes[-1]:] == 7.0).all())
        for e, (W, b) in enumerate(nets):
            y, _ = mlp.forward(W, b, x)
            # per layer an operand rounding and the BF16 GELU steps (about 2^-8 each, random
            # in sign over a row's products): 5 layers give the 1e-2 of the scale that the
            # other tests of this path allow, and more layers scale it
            scale = max(np.abs(y).max(), np.sqrt(np.mean(y ** 2)))
            assert np.abs(Y[e] - y).max() <= 3e-2 * max(1.0, (len(sizes) - 1) / 5) * scale, (n, e)
