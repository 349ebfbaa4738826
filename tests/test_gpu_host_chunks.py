"""Host round trips in three chunks and in four (large states, few steps a call), and one
after the other: the same state, bit for bit, as the same steps on the device."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_chunk_counts():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic
    n = (3 << 20) + 517            # ragged chunks; 2 steps: four of them, 5 steps: three
    rng = np.random.default_rng(8)
    z, r = rng.uniform(0.3, 0.7, n), rng.uniform(0.1, 0.4, n)
    u = rng.normal(0, 0.02, (3, n))   # none reaches a wall
    mesh = pic.pic_mesh_create(*W.cavity_mesh(n_tri=2000), precision=pic.PIC_FP32)
    dt = 0.5 * pic.pic_spai_build(mesh)
    runs = []
    for calls in (None, (2, 5), (5, 2), (1, 1, 5)):
        sim = pic.pic_sim_create(mesh, dt, 0.3, n)
        pic.pic_sim_set_sort_interval(sim, 3)
        pic.pic_particles_inject(sim, z, r, u[0], u[1], u[2], -1.0, 1.0, 1e-9)
        if calls is None:
            pic.pic_step(sim, 7)
        else:
            host = torch.empty(pic.pic_particles_raw_size(sim, n), dtype=torch.uint8, pin_memory=True)
            pic.pic_particles_raw_get(sim, host.data_ptr(), n)
            torch.cuda.synchronize()
            for k in calls:
                pic.pic_step_host(sim, host.data_ptr(), n, k)
            torch.cuda.synchronize()
        d = pic.pic_diagnostics(sim, fields=True)
        g = pic.pic_particles_get(sim)
        at = np.argsort(g["pid"])
        assert d["n_absorbed"] == 0 and d["dce_nonzero"] == 0
        runs.append([g[k][at] for k in ("pid", "tri", "lam", "u")] + [d["E"], d["B"], d["J"]])
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)
