"""Work that rides along with a step's field kernels: births over many blocks of the face
kernel (fewer than a block's threads, one more than a block, more than all its blocks take
at once) and probes and ports together in the residual kernel, at every block size the
tuner may pick, with plain and replayed steps giving the same records."""
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
@pytest.mark.parametrize("per_step", [1, 255, 257, 1024 * 256 + 3])
def test_births_over_blocks(pic, precision, per_step):
    mesh = pic.pic_mesh_create(*W.cavity_mesh(n_tri=400), precision=pic.PIC_FP32 if precision == "fp32"
                               else pic.PIC_FP64)
    dt = 0.5 * pic.pic_spai_build(mesh)
    steps = 3
    # room for two steps' births and a part of the third's: the third makes none
    sim = pic.pic_sim_create(mesh, dt, 0.0, 3 * per_step - 1)
    pic.pic_sim_set_emitter(sim, 0.013, 0.0, 0.35, per_step, 1e-3, 1e-4, 5, -1.0, 1.0, 1e-9)
    pic.pic_step(sim, steps)
    d = pic.pic_diagnostics(sim)
    assert d["n_emitted"] == 2 * per_step and d["emit_dropped"] == per_step
    p = pic.pic_particles_get(sim)
    assert np.array_equal(np.sort(p["pid"]), np.arange(2 * per_step))
    assert np.all(p["tri"] >= 0) and d["n_absorbed"] == 0
    assert d["dce_nonzero"] == 0 if precision == "fp32" else d["dce_max"] < 1e-9 * per_step


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_probes_and_ports_together(pic, precision):
    arrays = W.rect_mesh(1.0, 0.5, 1200, 17)
    prec = pic.PIC_FP64 if precision == "fp64" else pic.PIC_FP32
    mesh = pic.pic_mesh_create(*arrays, precision=prec)
    dt = 0.5 * pic.pic_spai_build(mesh)
    info = pic.pic_mesh_info(mesh)
    face = np.arange(info["n_tris"])
    group = face % 3
    runs = []
    for graph in (False, True):
        sim = pic.pic_sim_create(mesh, dt, 0.0, 16)
        pic.pic_sim_set_sort_interval(sim, 2)
        pic.pic_sim_set_graph(sim, graph)
        pic.pic_fields_set(sim, W.random_edge_values(info["n_edges"], 0.05, 41),
                           W.random_edge_values(info["n_tris"], 1e-3, 42))
        pic.pic_sim_set_probes(sim, face, group, 1.0 + face * 1e-3, [1, 2, 1], capacity=8, every=3)
        pic.pic_sim_set_ports(sim, [0.4321, 0.6113], [0.0, 0.1], [0.5, 0.37], capacity=4, every=2)
        sums = []
        for k in range(14):
            pic.pic_step(sim, 1)
            if k % 3 == 0:
                B = pic.pic_fields_get(sim)[1]
                w = 1.0 + face * 1e-3
                sums.append([(w * B ** q)[group == g].sum() for g, q in enumerate((1, 2, 1))])
        rec, dropped = pic.pic_probes_read(sim)
        ports, lost = pic.pic_ports_read(sim)
        # 14 steps: probes at steps 0, 3, .. 12 (5 records), ports at 0, 2, .. 12 (7, room for 4)
        assert rec.shape == (5, 3) and dropped == 0 and ports.shape == (4, 2) and lost == 3
        # the probes' FP64 sums of 400 values against numpy's
        assert np.abs(rec - np.array(sums)).max() <= 1e-12 * np.abs(sums).max()
        runs.append((rec, ports))
    assert np.array_equal(runs[0][0], runs[1][0]) and np.array_equal(runs[0][1], runs[1][1])


@pytest.mark.parametrize("interval", [0, 2, 16])
@pytest.mark.parametrize("n0,per_step", [(0, 100), (0, 1500), (511, 513), (400_000, 2000), (300, 400_000)])
def test_every_slot_once_with_births(pic, n0, per_step, interval):
    """Slots that the last re-sort ordered and births since then are walked by different
    rules: with next to no charge and fields every particle flies straight, so a slot taken
    twice or not at all is off by a step.  Positions are fixed point at 2^-22 of a cell and
    the displacement is FP32: 1e-5 of a cell a step."""
    arrays = W.rect_mesh(1.0, 0.5, 800, 3)
    nodes, tris = arrays[0], arrays[1]
    mesh = pic.pic_mesh_create(*arrays, precision=pic.PIC_FP32)
    dt = 0.5 * pic.pic_spai_build(mesh)
    steps, u = 5, 0.1
    sim = pic.pic_sim_create(mesh, dt, 0.0, n0 + steps * per_step)
    pic.pic_sim_set_sort_interval(sim, interval)
    rng = np.random.default_rng(9)
    if n0:
        z0, r0 = rng.uniform(0.1, 0.5, n0), rng.uniform(0.05, 0.45, n0)
        pic.pic_particles_inject(sim, z0, r0, np.zeros(n0), np.zeros(n0), np.full(n0, u), -1.0, 1.0, 1e-15)
    pic.pic_sim_set_emitter(sim, 0.013, 0.0, 0.35, per_step, u, 0.0, 5, -1.0, 1.0, 1e-15)
    pic.pic_step(sim, steps)
    p = pic.pic_particles_get(sim)
    n = n0 + steps * per_step
    assert np.array_equal(np.sort(p["pid"]), np.arange(n)) and np.all(p["tri"] >= 0)
    z = np.zeros(n)
    z[p["pid"]] = (p["lam"] * nodes[tris[p["tri"]]][:, :, 0]).sum(1)
    v = u / np.sqrt(1.0 + u * u)
    born = np.where(np.arange(n) < n0, 0, (np.arange(n) - n0) // per_step)
    start = np.full(n, 0.013)
    if n0:
        start[:n0] = z0
    cell = 0.04
    assert np.abs(z - start - v * dt * (steps - born)).max() <= 1e-5 * cell * steps
