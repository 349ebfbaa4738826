"""Particles at places that the particle kernels meet rarely: landing exactly on the axis,
coordinates that rounding left just below zero, and steps too small for a normal FP32 number.
Force-free, so every particle ends at z + v_z dt, |rho + v_rho dt|."""
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


def _sim(pic, precision, cap, n_tri=400):
    arrays = W.cavity_mesh(n_tri=n_tri)
    mesh = pic.pic_mesh_create(*arrays, precision=pic.PIC_FP64 if precision == "fp64" else pic.PIC_FP32)
    dt = 0.5 * pic.pic_spai_build(mesh)
    sim = pic.pic_sim_create(mesh, dt, 0.0, cap)
    pic.pic_sim_set_sort_interval(sim, 0)
    return arrays, sim, dt


def _by_pid(p, n):
    """lam, u, tri by particle id; tri is -1 for a particle that is gone."""
    tri, lam, u = -np.ones(n, np.int64), np.zeros((n, 3)), np.zeros((n, 3))
    tri[p["pid"]], lam[p["pid"]], u[p["pid"]] = p["tri"], p["lam"], p["u"]
    return tri, lam, u


def _positions(arrays, tri, lam):
    return np.einsum("nk,nkd->nd", lam, np.asarray(arrays[0])[np.asarray(arrays[1])[tri]])


@pytest.mark.parametrize("pusher", ["boris", "vay"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_landing_on_the_axis(pic, precision, pusher):
    """Radially inward from rho = |v| dt: rho + v dt is zero or its rounding, and both have to
    end on the axis (FP32: within the 2^-22 of a cell that positions have, a few times; that
    rounding also spreads the landings, so more particles are needed for some exact ones)."""
    n = 3000 if precision == "fp64" else 40_000
    arrays, sim, dt = _sim(pic, precision, n)
    if pusher == "vay":
        pic.pic_sim_set_pusher(sim, pic.PIC_PUSHER_VAY)
    rng = np.random.default_rng(11)
    v = rng.uniform(0.05, 0.95, n)
    z = rng.uniform(0.1, 0.9, n)
    zero = np.zeros(n)
    pic.pic_particles_inject(sim, z, v * dt, -v / np.sqrt(1.0 - v * v), zero, zero, -1.0, 1.0, 1e-15)
    pic.pic_step(sim, 1)
    tri, lam, u = _by_pid(pic.pic_particles_get(sim), n)
    assert np.all(tri >= 0)
    x = _positions(arrays, tri, lam)
    cell = np.sqrt(0.5 / 400)
    tol = 1e-12 if precision == "fp64" else 8 * 2.0 ** -22 * cell
    assert np.abs(x[:, 1]).max() < tol
    assert np.abs(x[:, 0] - z).max() < tol
    d = pic.pic_diagnostics(sim)
    assert d["n_absorbed"] == 0
    assert d["dce_nonzero"] == 0 if precision == "fp32" else d["dce_max"] < 1e-12 * n


@pytest.mark.parametrize("speed", [1e-3, 1e-18, 1e-20, 1e-28])
def test_reflection_at_the_axis(pic, speed):
    """FP32 (whose coordinates on the axis are exact): from the axis across it at any speed
    (1e-18 and below: the square of the step, 1e-2 of that, is no normal number), u_rho comes
    out reversed."""
    n = 100
    arrays, sim, dt = _sim(pic, "fp32", n)
    z, zero = np.linspace(0.1, 0.9, n), np.zeros(n)
    pic.pic_particles_inject(sim, z, zero, np.full(n, -speed), zero, zero, -1.0, 1.0, 1e-15)
    pic.pic_step(sim, 1)
    tri, lam, u = _by_pid(pic.pic_particles_get(sim), n)
    assert np.all(tri >= 0)
    assert np.abs(u[:, 0] / speed - 1.0).max() < 1e-6 and np.all(u[:, 1:] == 0.0)
    assert np.abs(_positions(arrays, tri, lam)[:, 1] - speed * dt).max() < 1e-7


def _raw_state(pic, sim, precision, tri, l0, l1, u):
    """One slot per entry, written through the raw layout (pic_particles_raw_set)."""
    import torch
    n = len(tri)
    stride = (n + 31) // 32 * 32
    real = np.float64 if precision == "fp64" else np.float32
    lam = np.float64 if precision == "fp64" else np.int32
    buf = torch.zeros(pic.pic_particles_raw_size(sim, n), dtype=torch.uint8).pin_memory()
    raw, at = buf.numpy(), 0
    for a, t in ((tri, np.int32), (l0, lam), (l1, lam), (u[:, 0], real), (u[:, 1], real), (u[:, 2], real)):
        size = np.dtype(t).itemsize
        raw[at:at + size * n] = np.ascontiguousarray(a, t).view(np.uint8)
        at += size * stride
    pic.pic_particles_raw_set(sim, buf.data_ptr(), n)
    torch.cuda.synchronize()


def _gradients(arrays):
    """grad lambda_k (z, rho) of every triangle, in the mesh's counter-clockwise node order"""
    p = np.asarray(arrays[0])[np.asarray(arrays[1])]
    e = np.stack([p[:, (k + 2) % 3] - p[:, (k + 1) % 3] for k in range(3)], 1)
    twice = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - \
            (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
    return np.stack([-e[:, :, 1], e[:, :, 0]], 2) / twice[:, None, None], twice


@pytest.mark.parametrize("share", [0.0, 0.3, 0.7, 0.95])
@pytest.mark.parametrize("below", [1.1e-16, 1e-12])
def test_coordinate_below_zero_moving_inward(pic, below, share):
    """FP64: on every edge (walls and the axis among them), `below` outside of its triangle,
    at rest or moving inward by a share of that: the particle stays where it is."""
    arrays = W.cavity_mesh(n_tri=400)
    g, twice = _gradients(arrays)
    N2 = len(twice)
    assert np.all(twice > 0)   # the mesh keeps the node order of counter-clockwise triangles
    arrays, sim, dt = _sim(pic, "fp64", 3 * N2)
    tri = np.repeat(np.arange(N2), 3)
    k = np.tile(np.arange(3), N2)
    l = np.full((3 * N2, 3), 0.5)
    l[np.arange(3 * N2), k] = -below
    l[k == 2, 1] = 0.5 + max(below, 2.0 ** -53)   # l2 = 1 - l0 - l1
    gk = g[tri, k]
    v = share * below * gk / (gk ** 2).sum(1)[:, None] / dt
    u = np.stack([v[:, 1], np.zeros(3 * N2), v[:, 0]], 1)
    # one particle of each id through the ordinary way first: a species has to be known
    centre = np.asarray(arrays[0])[np.asarray(arrays[1])].mean(1)[tri]
    zero = np.zeros(3 * N2)
    pic.pic_particles_inject(sim, centre[:, 0], centre[:, 1], zero, zero, zero, -1.0, 1.0, 1e-15)
    ids = pic.pic_particles_get(sim)["pid"]
    _raw_state(pic, sim, "fp64", tri, l[:, 0], l[:, 1], u)
    pic.pic_step(sim, 1)
    got, lam, gu = _by_pid(pic.pic_particles_get(sim), 3 * N2)
    order = np.empty(3 * N2, np.int64)
    order[ids] = np.arange(3 * N2)   # slot of each id
    assert np.all(got >= 0) and np.all(np.isfinite(lam)) and np.all(np.isfinite(gu))
    was = _positions(arrays, tri, np.stack([l[:, 0], l[:, 1], 1 - l[:, 0] - l[:, 1]], 1))[order]
    assert np.abs(_positions(arrays, got, lam) - was).max() < 4 * below + 1e-14
    d = pic.pic_diagnostics(sim, fields=True)
    assert d["n_absorbed"] == 0 and np.all(np.isfinite(d["J"])) and np.all(np.isfinite(d["E"]))


@pytest.mark.parametrize("place", ["edge", "node"])
@pytest.mark.parametrize("step", [1e-37, 1e-38, 1e-41])
def test_step_below_the_normal_range(pic, step, place):
    """FP32: at coordinate 0 of a triangle away from the walls, moving outward by a step of
    `step` of that coordinate, a normal or a subnormal number: the particle stays where it is."""
    arrays = W.cavity_mesh(n_tri=400)
    g, _ = _gradients(arrays)
    nodes, tris = np.asarray(arrays[0]), np.asarray(arrays[1])
    wall = np.zeros(len(nodes), bool)
    wall[np.asarray(arrays[2]).ravel()] = True
    inner = np.flatnonzero(~wall[tris].any(1))
    n = 3 * len(inner)
    arrays, sim, dt = _sim(pic, "fp32", n)
    tri, k = np.repeat(inner, 3), np.tile(np.arange(3), len(inner))
    one, i = 1 << 22, np.arange(n)
    l = np.full((n, 3), one // 2)
    l[i, k] = 0
    if place == "node":   # node k+1, leaving through edge k
        l[i, (k + 1) % 3] = one
        l[i, (k + 2) % 3] = 0
    gk = g[tri, k]
    v = -step * gk / (gk ** 2).sum(1)[:, None] / dt
    u = np.stack([v[:, 1], np.zeros(n), v[:, 0]], 1)
    centre = nodes[tris].mean(1)[tri]
    zero = np.zeros(n)
    pic.pic_particles_inject(sim, centre[:, 0], centre[:, 1], zero, zero, zero, -1.0, 1.0, 1e-15)
    ids = pic.pic_particles_get(sim)["pid"]
    _raw_state(pic, sim, "fp32", tri, l[:, 0], l[:, 1], u)
    pic.pic_step(sim, 1)
    got, lam, _ = _by_pid(pic.pic_particles_get(sim), n)
    order = np.empty(n, np.int64)
    order[ids] = i
    assert np.all(got >= 0)
    was = _positions(arrays, tri, l / one)[order]
    assert np.abs(_positions(arrays, got, lam) - was).max() < 1e-6
    assert pic.pic_diagnostics(sim)["n_absorbed"] == 0
