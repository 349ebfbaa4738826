"""Recorded values and births do not depend on the launch shapes: a run through the tuner,
which steps with every block size it may pick, against plain steps."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic as p
    return p


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_records_of_a_tuned_run(pic, precision):
    trial = 3
    steps = 2 * trial * 7   # the setting found, and two others of each of three knobs
    arrays = W.rect_mesh(1.0, 0.5, 3000, 17)
    mesh = pic.pic_mesh_create(*arrays, precision=pic.PIC_FP64 if precision == "fp64" else pic.PIC_FP32)
    dt = 0.5 * pic.pic_spai_build(mesh)
    info = pic.pic_mesh_info(mesh)
    face = np.arange(info["n_tris"])
    # particles feed the fields in the FP32 build only: its sums are exact whatever their order
    births = 700 if precision == "fp32" else 0
    runs = []
    for tuned in (False, True):
        sim = pic.pic_sim_create(mesh, dt, 0.0, 16 + births * steps)
        pic.pic_fields_set(sim, W.random_edge_values(info["n_edges"], 0.05, 41),
                           W.random_edge_values(info["n_tris"], 1e-3, 42))
        if births:
            pic.pic_sim_set_emitter(sim, 0.013, 0.0, 0.35, births, 0.1, 1e-2, 5, -1.0, 1.0, 1e-6)
        pic.pic_sim_set_probes(sim, face, face % 3, 1.0 + face * 1e-3, [1, 2, 1], capacity=steps, every=1)
        pic.pic_sim_set_ports(sim, [0.4321, 0.6113], [0.0, 0.1], [0.5, 0.37], capacity=steps)
        if tuned:
            pic.pic_sim_autotune(sim, trial)
        else:
            pic.pic_step(sim, steps)
        rec, dropped = pic.pic_probes_read(sim)
        ports, lost = pic.pic_ports_read(sim)
        assert rec.shape == (steps, 3) and ports.shape == (steps, 2) and dropped == lost == 0
        E, B = pic.pic_fields_get(sim)
        d = pic.pic_diagnostics(sim)
        assert d["n_emitted"] == births * steps and d["dce_nonzero"] == 0
        runs.append((rec, ports, E, B))
    for a, b in zip(*runs):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
