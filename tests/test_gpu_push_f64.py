"""FP64 particle kernel against the oracle where its split of the work can go wrong: fewer
particles than a warp, one more than a warp or a block, and enough that every warp takes
several rounds and fills its ring of leaving particles more than once; slow particles (few
leave their triangle) and fast ones (most cross several edges).  1e-12 relative per step,
the bound of the FP64 build."""
import numpy as np
import pytest

import workloads as W
from oracle import OracleSim
from tests.test_gpu_parity import _gpu_particles, _oracle_step, _setup, pic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small_mesh():
    arrays = W.cavity_mesh(n_tri=400)
    return arrays, OracleSim(*arrays)


@pytest.mark.parametrize("pusher", ["boris", "vay"])
@pytest.mark.parametrize("n,sigma_u", [(1, 0.3), (31, 3.0), (33, 0.3), (65, 3.0), (2049, 3.0),
                                       (700_001, 0.02), (650_017, 1.0)])
def test_push_over_rounds(pic, small_mesh, n, sigma_u, pusher):  # noqa: F811
    arrays, oracle = small_mesh
    o, sim, mesh, cap = _setup(pic, arrays, oracle, pic.PIC_FP64, n, seed=60, sigma_u=sigma_u, pusher=pusher)
    pic.pic_step(sim, 1)
    _oracle_step(o, 1, cap)
    d = pic.pic_diagnostics(sim, fields=True)
    tri, lam, u = _gpu_particles(pic, sim, n)
    assert np.array_equal(tri, o.tri)
    live = o.tri >= 0
    assert np.abs(lam[live] - o.lam[live]).max(initial=0.0) < 1e-12
    assert np.abs(u[live] - o.u[live]).max(initial=0.0) < 1e-12 * np.abs(o.u).max()
    Q, _, Qa = pic.pic_charges_get(sim)
    # sums of n terms in another order: sqrt(n) 2^-53 of the largest
    tol = 1e-12 * max(1.0, np.sqrt(n) * 1e-3)
    for got, want in ((d["E"], o.E), (d["B"], o.B), (d["J"], o.J), (Q, o.Q)):
        assert np.abs(got - want).max() < tol * np.abs(want).max()
    assert np.abs(Qa - o.Qabs).max() < tol * max(np.abs(o.Q).max(), 1e-30)
    assert d["n_absorbed"] == o.counters[0] and d["n_crossings"] == o.counters[2]
