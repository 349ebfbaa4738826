"""The work that this library's users have it do, as cases whose time can be taken.

A case is one call sequence through the binding (``paper_1701_03784_gb300.pic``), of one of
these kinds:

* ``cold``    field solver alone, one step and the fields read back, as a cold test's
              ring-down loop does it (FP64, no particles);
* ``cavity``  the normalised cavity with thermal electrons, many steps and the whole state
              read back (particles by id, fields, charges);
* ``diode``   emission and a gun field: one step, the electrodes' charges read, repeated;
* ``union``   surrogate data: instances of the ripple sweep as one simulation, CUDA-graph
              replay, output-port power recorded on the device;
* ``beam``    the backward-wave oscillator: steps between two looks at the fields;
* ``host``    the same with the particle state in page-locked host memory between steps;
* ``infer``   the surrogate ensemble's answers;
* ``train``   Adam steps of the ensemble, and the updated weights.

Outputs of the FP32 build are returned as FP32, the precision that it keeps them in (the
binding widens them to FP64 on the way out).  Meshes and their SPAI operators do not
depend on the inputs; a program builds them once, and so does this file.
"""
import functools
import math

import numpy as np
import torch

import workloads as W
from paper_1701_03784_gb300 import pic
from paper_1701_03784_gb300.batch import union
from paper_1701_03784_gb300.diode import classical_limit
from paper_1701_03784_gb300.ports import graded_layer, sigma_max_for
from paper_1701_03784_gb300.surrogate import SIZES
from workloads.bwo import BZ_BWO, C0, EPS0, ME, MU0, QE
from workloads.sweep import WEIGHT, surrogate_instance

CELL = dict(r0=15.0e-3, ripple=2.1e-3, period=7.5e-3)       # the cold test's cell
CAVITY = dict(a=0.5, L=1.0)
GAP, V_GAP, R_EMIT, R_TUBE = 1e-2, 1e5, 1e-2, 2e-2          # the diode
SIGMA_U = 0.01


def listed():
    return [
        # one step of a ring-down on a mesh of the staircasing study: nothing but latency
        dict(name="cold_test_step", kind="cold", n_tri=1960, steps=1),
        # the plain method's stated configuration: 2000 triangles, 10,000 electrons, FP64
        dict(name="cavity_fp64", kind="cavity", n_tri=2000, n=10_000, bits=64, steps=200),
        # the diode as stated: 20k triangles, 2000 births a step, the gap filled
        dict(name="diode_read", kind="diode", n_tri=20_000, per_step=2000, steps=4),
        # surrogate data: eight instances at 450 triangles per cm^2, 5% of their particles
        dict(name="surrogate_union", kind="union", instances=8, steps=64, every=8),
        # the single BWO as stated: 200k triangles, 16M particles
        dict(name="bwo_16m", kind="beam", n_tri=200_000, n=16_000_000, bits=32, fill="beam",
             pusher="boris", loss=False, sort=16, steps=32),
        # the whole mesh filled evenly, absorbing layers at both ends, the corrected pusher
        dict(name="filled_vay_5m", kind="beam", n_tri=50_000, n=5_000_001, bits=32,
             fill="even", pusher="vay", loss=True, sort=16, steps=16),
        # a sweep instance at its smallest beam, re-sorted as the autotuner picks
        dict(name="sweep_half_million", kind="beam", n_tri=47_001, n=500_000, bits=32,
             fill="beam", pusher="boris", loss=False, sort=32, steps=32),
        # the FP64 build that checks the FP32 one
        dict(name="bwo_fp64_1m", kind="beam", n_tri=200_000, n=1_000_000, bits=64, fill="beam",
             pusher="boris", loss=False, sort=16, steps=8),
        # end to end: the state goes up and comes back every step
        dict(name="host_state_8m", kind="host", n_tri=200_000, n=8_000_003, steps=4),
        # the ensemble asked for the answers of one batch of queries
        dict(name="infer_bf16_65536", kind="infer", members=5, hidden=256, layers=4,
             rows=65_536, tensor_cores=True),
        # the same in FP32 on a study's held-out rows and their neighbours, a ragged count
        dict(name="infer_fp32_10007", kind="infer", members=5, hidden=256, layers=4,
             rows=10_007, tensor_cores=False),
        # the ensemble's training at its own batch size
        dict(name="train_128", kind="train", members=5, hidden=256, layers=4, batch=128,
             rows=1024, steps=100),
    ]


def _between(rng, lo, hi):
    """A whole number, even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cold", "cavity", "diode", "union", "beam", "beam", "beam64", "host",
                       "infer", "infer", "train"])
    if kind == "cold":
        return dict(kind="cold", n_tri=_between(rng, 490, 7900), steps=rng.choice([1, 2, 5]))
    if kind == "cavity":
        return dict(kind="cavity", n_tri=_between(rng, 400, 4000), n=_between(rng, 100, 40_000),
                    bits=rng.choice([32, 64]), steps=rng.randint(20, 200))
    if kind == "diode":
        return dict(kind="diode", n_tri=_between(rng, 5000, 40_000),
                    per_step=_between(rng, 200, 3000), steps=rng.randint(1, 8))
    if kind == "union":
        return dict(kind="union", instances=rng.randint(1, 8), steps=rng.randint(33, 128),
                    every=rng.choice([4, 8]))
    if kind == "beam":
        n_tri = _between(rng, 20_000, 200_000)
        n = _between(rng, 200_000, 16_000_000)
        return dict(kind="beam", n_tri=n_tri, n=n, bits=32, fill=rng.choice(["beam", "even"]),
                    pusher=rng.choice(["boris", "vay"]), loss=rng.random() < 0.3,
                    sort=rng.choice([8, 16, 32]), steps=rng.randint(4, 16))
    if kind == "beam64":
        return dict(kind="beam", n_tri=_between(rng, 20_000, 200_000),
                    n=_between(rng, 50_000, 2_000_000), bits=64,
                    fill=rng.choice(["beam", "even"]), pusher=rng.choice(["boris", "vay"]),
                    loss=rng.random() < 0.3, sort=16, steps=rng.randint(1, 8))
    if kind == "host":
        return dict(kind="host", n_tri=_between(rng, 20_000, 200_000),
                    n=_between(rng, 500_000, 8_000_000), steps=rng.randint(2, 6))
    if kind == "infer":
        tc = rng.random() < 0.5
        return dict(kind="infer", members=rng.randint(1, 8), hidden=rng.choice([64, 100, 128, 256]),
                    layers=rng.randint(1, 5), rows=_between(rng, 1, 65_536 if tc else 16_384),
                    tensor_cores=tc)
    return dict(kind="train", members=rng.randint(1, 8), hidden=rng.choice([64, 100, 128, 256]),
                layers=rng.randint(1, 4), batch=rng.choice([32, 100, 128, 256]),
                rows=_between(rng, 200, 4000), steps=rng.randint(8, 30))


# ---- meshes, built once ---------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _mesh(kind, size, bits):
    """(mesh handle, nodes, tris, stable step, what else the kind needs)."""
    more = None
    units = dict(eps0=EPS0, mu0=MU0, c=C0)
    if kind == "cold":
        nodes, tris, be, bt = W.meshes.sws_cell_mesh(size, **CELL)
    elif kind == "cavity":
        nodes, tris, be, bt = W.cavity_mesh(CAVITY["a"], CAVITY["L"], size)
        units = dict(eps0=1.0, mu0=1.0, c=1.0)
    elif kind == "diode":
        nodes, tris, be, bt = W.diode_mesh(size, gap=GAP, radius=R_TUBE)
    elif kind == "union":
        ins = [surrogate_instance(i) for i in range(size)]
        more = union(ins)
        more["zp"] = np.array([s + x["z_end"] - 4.93e-3 for s, x in zip(more["shift"], ins)])
        more["rp"] = np.array([x["r_out"] for x in ins]) * (1.0 - 1e-9)
        nodes, tris, be, bt = (more[k] for k in ("nodes", "tris", "be", "bt"))
    else:
        nodes, tris, be, bt = W.bwo_mesh(size)
    mesh = pic.pic_mesh_create(nodes, tris, be, bt, precision=pic.PIC_FP64 if bits == 64
                               else pic.PIC_FP32, **units)
    return mesh, nodes, tris, (be, bt), pic.pic_spai_build(mesh, 2, 1e-4), more


def _rule_step(kind, n_tri):
    """Time step of the small meshes, about half the stable one: 0.12 cells a step."""
    if kind == "cavity":
        return 0.12 * math.sqrt(4.0 * CAVITY["a"] * CAVITY["L"] / (math.sqrt(3.0) * n_tri))
    area = CELL["r0"] * CELL["period"]
    return 0.12 * math.sqrt(4.0 * area / (math.sqrt(3.0) * n_tri)) / C0


class _Draws:
    """Seeded draws made on the GPU and handed over as host arrays (injection takes those)."""

    def __init__(self, seed):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.g = torch.Generator(device=self.dev).manual_seed(int(seed) % (1 << 62))

    def unit(self, *shape):
        return torch.rand(*shape, generator=self.g, device=self.dev, dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=self.dev, dtype=torch.float64)


def _thermal(d, n, sigma, drift):
    u = sigma * d.normal(3, n)
    u[2] += drift
    return list(u.cpu().numpy())


# ---- inputs -----------------------------------------------------------------------------------

def _cavity_inputs(case, seed, nodes, edges):
    """Edge field of the two modes at seeded amplitudes, and thermal electrons."""
    d = _Draws(seed)
    p0, p1 = W.cavity_modes(nodes, edges)
    amp = 0.5 + d.unit(2).cpu().numpy()
    n = case["n"]
    z = (1e-3 + (CAVITY["L"] - 2e-3) * d.unit(n)).cpu().numpy()
    rho = ((CAVITY["a"] - 1e-3) * d.unit(n).sqrt()).cpu().numpy()
    return amp[0] * p0 + amp[1] * p1, [z, rho] + _thermal(d, n, SIGMA_U, 0.0)


def _cold_inputs(seed, nodes, edges):
    amp = 0.5 + _Draws(seed).unit(2).cpu().numpy()
    return sum(a * W.tm0np_edge_dofs(nodes, edges, CELL["r0"], CELL["period"], 1, p)
               for p, a in enumerate(amp))


def _beam_inputs(case, seed, nodes, tris):
    """Annular 400 kV beam over the ripple section, or the whole mesh filled evenly."""
    d = _Draws(seed)
    n = case["n"]
    gamma = 1.0 + 400e3 / 510998.95
    uz = C0 * math.sqrt(gamma * gamma - 1.0)
    (zs0, zs1) = W.bwo_wall()[2]
    if case.get("fill", "beam") == "beam":
        z = zs0 + (zs1 - zs0) * d.unit(n)
        rho = (0.85e-2 ** 2 + (0.95e-2 ** 2 - 0.85e-2 ** 2) * d.unit(n)).sqrt()
    else:
        p = torch.from_numpy(nodes[tris]).to(d.dev)
        t = torch.arange(n, device=d.dev) % len(tris)
        s, r = d.unit(n).sqrt(), d.unit(n)
        lam = torch.stack([1.0 - s, s * (1.0 - r), s * r], 1) * (1.0 - 3e-6) + 1e-6
        zr = (lam[:, :, None] * p[t]).sum(1)
        z, rho = zr[:, 0].contiguous(), zr[:, 1].contiguous()
    vz = uz / gamma
    weight = 3e3 * (zs1 - zs0) / vz / (abs(QE) * n)
    edge = 1e-3 * (3e3 / vz) / (2 * math.pi * EPS0 * 0.9e-2) * 2e-4
    return [z.cpu().numpy(), rho.cpu().numpy()] + _thermal(d, n, 1e-3 * uz, uz), weight, edge, d


def _edge_field(d, n_edges, scale):
    return scale * (2.0 * d.unit(n_edges) - 1.0).cpu().numpy()


def _net_inputs(case, seed):
    """Member weights as the ensemble starts them, and query rows in [-1, 1]."""
    sizes = (SIZES[0],) + (case["hidden"],) * case["layers"] + (SIZES[-1],)
    d = _Draws(seed)
    params = []
    for k, n in zip(sizes[:-1], sizes[1:]):
        lim = 1.0 / math.sqrt(k)
        params.append(lim * (2.0 * d.unit(case["members"], n * k) - 1.0))
        params.append(0.05 * d.normal(case["members"], n))
    params = torch.cat(params, 1).float().double().cpu().numpy()
    X = (2.0 * d.unit(case["rows"], sizes[0]) - 1.0).float()
    # smooth targets of unit size with some scatter
    mix = d.normal(sizes[0], sizes[-1])
    T = (torch.sin(X.double() @ mix) + 0.02 * d.normal(case["rows"], sizes[-1])).float()
    return sizes, params, X, T


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("infer", "train"):
        sizes, params, X, T = _net_inputs(case, seed)
        net = pic.pic_mlp_create(case["members"], sizes, case.get("batch", 256))
        pic.pic_mlp_params_set(net, params)
        return dict(case=case, net=net, X=X, T=T, seed=seed % 1000)
    bits = 64 if kind == "cold" else case.get("bits", 32)
    size = case["instances"] if kind == "union" else case["n_tri"]
    mesh, nodes, tris, _, dt_max, more = _mesh("beam" if kind == "host" else kind, size, bits)
    info = pic.pic_mesh_info(mesh)
    no_b = np.zeros(info["n_tris"])
    st = dict(case=case, mesh=mesh, bits=bits, nodes=nodes, tris=tris)
    if kind == "cold":
        st["sim"] = pic.pic_sim_create(mesh, _rule_step(kind, size), 0.0, 16)
        pic.pic_fields_set(st["sim"], _cold_inputs(seed, nodes, pic.pic_mesh_edges(mesh)), no_b)
    elif kind == "cavity":
        E, parts = _cavity_inputs(case, seed, nodes, pic.pic_mesh_edges(mesh))
        sim = st["sim"] = pic.pic_sim_create(mesh, _rule_step(kind, size), 0.0, case["n"])
        pic.pic_sim_set_graph(sim, True)
        pic.pic_fields_set(sim, E, no_b)
        pic.pic_particles_inject(sim, *parts, -1.0, 1.0, W.cavity_weight(case["n"]))
    elif kind == "diode":
        z = nodes[:, 0]
        held = np.flatnonzero((z == 0.0) | (z == GAP))
        _, Es = pic.pic_static_potential(mesh, held, np.where(z[held] == 0.0, 0.0, V_GAP))
        dt = 0.5 * dt_max
        # space-charge-limited flow: a particle born t ago is at z = gap (t / T)^3
        v_end = math.sqrt(2.0 * V_GAP * abs(QE) / ME)
        transit = 3.0 * GAP / v_end
        n = int(case["per_step"] * transit / dt)
        d = _Draws(seed)
        s = (1e-3 + (1.0 - 2e-3) * d.unit(n)).cpu().numpy()
        rho = (0.999 * R_EMIT * d.unit(n).sqrt()).cpu().numpy()
        gamma = 1.0 + V_GAP * s ** 4 / 510998.95
        weight = classical_limit(V_GAP, GAP) * math.pi * R_EMIT ** 2 * dt / (case["per_step"] * abs(QE))
        room = (n + 4000 * case["per_step"] + 1023) // 1024 * 1024
        sim = st["sim"] = pic.pic_sim_create(mesh, dt, 0.0, room)
        pic.pic_sim_set_graph(sim, True)
        pic.pic_sim_set_static_field(sim, Es)
        pic.pic_particles_inject(sim, GAP * s ** 3, rho, np.zeros(n), np.zeros(n),
                                 C0 * np.sqrt(gamma * gamma - 1.0), QE, ME, weight)
        pic.pic_sim_set_emitter(sim, 1e-6 * GAP, 0.0, R_EMIT, case["per_step"], 0.0, 0.0,
                                int(seed), QE, ME, weight)
    elif kind == "union":
        d = _Draws(seed)
        n = len(more["z"])
        sim = st["sim"] = pic.pic_sim_create(mesh, 1e-13, 2.0, n + 1024)
        pic.pic_sim_set_graph(sim, True)
        pic.pic_fields_set(sim, _edge_field(d, info["n_edges"], 1.0), no_b)
        u = [x + 1e-3 * C0 * d.normal(n).cpu().numpy() for x in (more["ur"], more["up"], more["uz"])]
        pic.pic_particles_inject(sim, more["z"], more["r"], *u, QE, ME, WEIGHT)
        pic.pic_sim_set_ports(sim, more["zp"], 0.0, more["rp"], capacity=256, every=case["every"])
    else:
        parts, weight, edge, d = _beam_inputs(case, seed, nodes, tris)
        sim = st["sim"] = pic.pic_sim_create(mesh, 0.49 * dt_max, BZ_BWO, case["n"])
        pic.pic_sim_set_sort_interval(sim, case.get("sort", 32))
        if case.get("pusher") == "vay":
            pic.pic_sim_set_pusher(sim, pic.PIC_PUSHER_VAY)
        if case.get("loss"):
            z1 = float(nodes[:, 0].max())
            sig = sigma_max_for(1e-4, 1e-2, eps0=EPS0, c=C0)
            e = pic.pic_mesh_edges(mesh)
            lo = graded_layer(nodes, e, tris, 1e-2, 0.0, sig, eps0=EPS0, mu0=MU0)
            hi = graded_layer(nodes, e, tris, z1 - 1e-2, z1, sig, eps0=EPS0, mu0=MU0)
            pic.pic_sim_set_loss(sim, lo[0] + hi[0], lo[1] + hi[1])
        pic.pic_fields_set(sim, _edge_field(d, info["n_edges"], edge), no_b)
        pic.pic_particles_inject(sim, *parts, QE, ME, weight)
        if kind == "host":
            st["state"] = _host_state(sim, case["n"])
    return st


def _host_state(sim, n):
    """The raw state in a page-locked buffer, the slots of a triangle in the order of their
    coordinates (injection leaves them in none)."""
    buf = torch.empty(pic.pic_particles_raw_size(sim, n), dtype=torch.uint8).pin_memory()
    pic.pic_particles_raw_get(sim, buf.data_ptr(), n)
    torch.cuda.current_stream().synchronize()
    rows = buf.view(torch.int32).view(6, -1)[:, :n]
    dev = rows.cuda()
    key = ((dev[0].long() << 44) | (dev[1].long() << 22)) + dev[2].long()
    rows.copy_(dev[:, torch.argsort(key)])
    return buf


# ---- one pass ---------------------------------------------------------------------------------

def _kept(st, arrays):
    """Values of the FP32 build in the precision that it keeps."""
    return [a if st["bits"] == 64 else a.astype(np.float32) for a in arrays]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "infer":
        return pic.pic_mlp_forward(state["net"], state["X"], tensor_cores=case["tensor_cores"])
    if kind == "train":
        loss = pic.pic_mlp_train(state["net"], state["X"], state["T"], case["batch"],
                                 case["steps"], lr=1e-3, seed=state["seed"])
        return [pic.pic_mlp_params_get(state["net"]).astype(np.float32), loss.astype(np.float32)]
    sim = state["sim"]
    if kind == "cold":
        pic.pic_step(sim, case["steps"])
        return list(pic.pic_fields_get(sim))
    if kind == "diode":
        wall = 0.0
        for _ in range(case["steps"]):
            pic.pic_step(sim, 1)
            Q, _, Qa = pic.pic_charges_get(sim)
            wall = wall + Qa
        return _kept(state, [Q, wall, *pic.pic_fields_get(sim)])
    if kind == "union":
        pic.pic_step(sim, case["steps"])
        power, _ = pic.pic_ports_read(sim)
        return _kept(state, [power, *pic.pic_fields_get(sim), pic.pic_charges_get(sim)[0]])
    if kind == "host":
        buf, n = state["state"], case["n"]
        pic.pic_step_host(sim, buf.data_ptr(), n, case["steps"])
        E, B = pic.pic_fields_get(sim)      # waits for the last write-back
        u = buf.view(torch.float32).view(6, -1)[3:, :n]
        return [*u, *_kept(state, [E, B, pic.pic_charges_get(sim)[0]])]
    pic.pic_step(sim, case["steps"])
    d = pic.pic_diagnostics(sim, fields=True)
    out = _kept(state, [d["E"], d["B"], d["J"], pic.pic_charges_get(sim)[0]])
    if kind == "cavity":
        p = pic.pic_particles_get(sim)
        out.append(_by_id(state, p, case["n"]))
    else:
        out.append(np.array([d["kinetic_energy"], d["field_energy"]]))
    return out if state["bits"] == 64 else [np.float32(x) for x in out]


def _by_id(state, p, n):
    """(z, rho, u_rho, u_phi, u_z) of every particle by id; zeros once it is absorbed."""
    live = p["tri"] >= 0
    zr = (p["lam"][live][:, :, None] * state["nodes"][state["tris"][p["tri"][live]]]).sum(1)
    out = np.zeros((n, 5))
    out[p["pid"][live], :2] = zr
    out[p["pid"][live], 2:] = p["u"][live]
    return out


# ---- what a pass cannot do without ------------------------------------------------------------

def work(case):
    """Particle state in and out once a step (fields couple all particles between steps);
    per triangle and step the operators, fields and currents: 1.5 edges and half a node a
    triangle, 12.5 SPAI entries an edge.  Networks: weights, rows and results once (training:
    weights, moments and gradients once a step)."""
    kind = case["kind"]
    if kind in ("infer", "train"):
        h = case["hidden"]
        weights = SIZES[0] * h + h * h * (case["layers"] - 1) + h * SIZES[-1]
        if kind == "train":
            steps, rows = case["steps"], case["batch"]
            flops = 6.0 * rows * weights * case["members"] * steps
            return dict(bytes=4.0 * 7 * weights * case["members"] * steps, flops=flops)
        rows, wide = case["rows"], 2.0 if case["tensor_cores"] else 4.0
        return dict(bytes=4.0 * rows * (SIZES[0] + SIZES[-1] * case["members"])
                    + wide * weights * case["members"],
                    flops=2.0 * rows * weights * case["members"])
    real = 8.0 if case.get("bits") == 64 or kind == "cold" else 4.0
    n, tri = 0.0, 20_000.0 * case["instances"] if kind == "union" else float(case["n_tri"])
    if kind == "diode":
        n = 2000.0 * case["per_step"]
    elif kind == "union":
        n = 1e5 * case["instances"]
    elif kind != "cold":
        n = float(case["n"])
    per_tri = 1.5 * (12.5 * (real + 4) + 2 * real + 32) + 18 * real + 24
    return dict(bytes=case["steps"] * (n * 2 * (4 + 5 * real) + tri * per_tri),
                flops=case["steps"] * (220.0 * n + 100.0 * tri))


# ---- the same in 64 bits ----------------------------------------------------------------------

def exact(case, seed):
    """Networks by torch in FP64; the two small simulations by numpy from the paper's
    equations, the SPAI operator included.  The large ones would take minutes."""
    kind = case["kind"]
    if kind in ("infer", "train"):
        return _exact_net(case, seed)
    if kind not in ("cold", "cavity"):
        return None
    n_tri = case["n_tri"]
    if kind == "cold":
        m = _Plain(*W.meshes.sws_cell_mesh(n_tri, **CELL), EPS0, MU0)
        E, parts, qm, q_src = _cold_inputs(seed, m.nodes, m.edges), None, 0.0, 0.0
    else:
        m = _Plain(*W.cavity_mesh(CAVITY["a"], CAVITY["L"], n_tri), 1.0, 1.0)
        E, parts = _cavity_inputs(case, seed, m.nodes, m.edges)
        qm, q_src = -1.0, -W.cavity_weight(case["n"]) / (2.0 * math.pi)
    sim = _PlainSim(m, E, parts, qm, q_src, _rule_step(kind, n_tri))
    for _ in range(case["steps"]):
        sim.step()
    if kind == "cold":
        return [sim.E, sim.B]
    return [sim.E, sim.B, sim.J, sim.charge(), sim.by_id()]


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _exact_net(case, seed):
    sizes, params, X, T = _net_inputs(case, seed)
    X, T = X.double(), T.double()
    p = torch.from_numpy(params).to(X.device)

    def forward(p, x):          # x: members x rows x inputs
        at = 0
        for i, (k, n) in enumerate(zip(sizes[:-1], sizes[1:])):
            w = p[:, at:at + n * k].reshape(-1, n, k)
            b = p[:, at + n * k:at + n * k + n]
            at += n * k + n
            x = x @ w.transpose(1, 2) + b[:, None, :]
            if i + 2 < len(sizes):
                x = _gelu(x)
        return x

    if case["kind"] == "infer":
        return torch.cat([forward(p, c.expand(len(p), -1, -1)) for c in X.split(8192)], 1)
    mom, var = torch.zeros_like(p), torch.zeros_like(p)
    for step in range(case["steps"]):
        rows = torch.from_numpy(_minibatch(case, seed % 1000, step)).to(X.device)
        q = p.clone().requires_grad_(True)
        loss = ((forward(q, X[rows]) - T[rows]) ** 2).mean((1, 2))
        loss.sum().backward()
        mom = 0.9 * mom + 0.1 * q.grad
        var = 0.999 * var + 0.001 * q.grad ** 2
        a, b = 1.0 - 0.9 ** (step + 1), 1.0 - 0.999 ** (step + 1)
        p = p - 1e-3 * (mom / a) / ((var / b).sqrt() + 1e-8)
    return [p, loss.detach()]


def _minibatch(case, seed, step):
    """Rows that each member draws at a step: splitmix64 of (seed, member, step, row)."""
    def mix(x):
        x = x + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return x ^ (x >> np.uint64(31))
    member = np.arange(case["members"], dtype=np.uint64)[:, None] << np.uint64(48)
    row = np.arange(case["batch"], dtype=np.uint64)[None, :]
    h = mix(np.uint64(seed) ^ mix(member ^ np.uint64(step << 20) ^ row))
    return (h % np.uint64(case["rows"])).astype(np.int64)


class _Plain:
    """Mesh operators in numpy: incidence, Hodge matrices, approximate inverse."""

    def __init__(self, nodes, tris, be, bt, eps0, mu0):
        p = nodes[tris]
        s2 = ((p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1])
              - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1]))
        tris = np.where((s2 < 0)[:, None], tris[:, [0, 2, 1]], tris).astype(np.int64)
        self.nodes, self.tris, self.c = nodes, tris, 1.0 / math.sqrt(eps0 * mu0)
        p = nodes[tris]
        self.area = 0.5 * np.abs(s2)
        nxt, prv = [1, 2, 0], [2, 0, 1]
        self.grad = np.stack([p[:, nxt, 1] - p[:, prv, 1], p[:, prv, 0] - p[:, nxt, 0]], 2)
        self.grad /= 2.0 * self.area[:, None, None]
        # local edge k runs from local node k+1 to k+2; edges from the lower to the higher node
        a, b = tris[:, nxt], tris[:, prv]
        key = np.minimum(a, b) * len(nodes) + np.maximum(a, b)
        keys, inv = np.unique(key.ravel(), return_inverse=True)
        self.tri_edge = inv.reshape(-1, 3)
        self.sign = np.where(a < b, 1.0, -1.0)
        self.edges = np.stack([keys // len(nodes), keys % len(nodes)], 1)
        n1 = len(keys)
        by = np.argsort(self.tri_edge.ravel(), kind="stable")
        first = np.searchsorted(self.tri_edge.ravel()[by], np.arange(n1))
        count = np.bincount(self.tri_edge.ravel(), minlength=n1)
        self.nbr = np.full(3 * len(tris), -1)
        both = first[count == 2]
        self.nbr[by[both]], self.nbr[by[both + 1]] = by[both + 1] // 3, by[both] // 3
        self.nbr = self.nbr.reshape(-1, 3)
        tag = np.zeros(n1, np.int64)
        tag[np.searchsorted(keys, be.min(1) * len(nodes) + be.max(1).astype(np.int64))] = bt
        self.tag = tag[self.tri_edge]
        self.free = np.flatnonzero(tag != W.BC_PEC)
        self.mu_inv = p[:, :, 1].mean(1) / (mu0 * self.area)
        self._operator(eps0)

    def _operator(self, eps0):
        """M: per column the least-squares inverse of star_eps over the free edges within two
        triangles, entries under 1e-4 of its largest dropped, then symmetrised."""
        tris, n1 = self.tris, len(self.edges)
        # Whitney forms at the six points of a degree-4 rule (the integrand is cubic)
        w4 = [(0.223381589678011, 0.445948490915965), (0.109951743655322, 0.091576213509771)]
        T = np.zeros((len(tris), 3, 3))
        for w, x in w4:
            for k in range(3):
                lam = np.full(3, x)
                lam[k] = 1.0 - 2.0 * x
                f = np.stack([self.sign[:, e, None] * (lam[(e + 1) % 3] * self.grad[:, (e + 2) % 3]
                                                       - lam[(e + 2) % 3] * self.grad[:, (e + 1) % 3])
                              for e in range(3)], 1)
                rho = self.nodes[tris][:, :, 1] @ lam
                T += (w * eps0 * self.area * rho)[:, None, None] * (f @ f.transpose(0, 2, 1))
        near = [set() for _ in range(n1)]
        entries = [dict() for _ in range(n1)]
        for t, e3 in enumerate(self.tri_edge.tolist()):
            for i, e in enumerate(e3):
                near[e].update(e3)
                for j, e2 in enumerate(e3):
                    entries[e][e2] = entries[e].get(e2, 0.0) + T[t, i, j]
        is_free = np.zeros(n1, bool)
        is_free[self.free] = True
        rows, cols, vals = [], [], []
        for e in self.free.tolist():
            S = sorted(x for x in set().union(*(near[y] for y in near[e])) if is_free[x])
            R = sorted(x for x in set().union(*(entries[y].keys() for y in S)) if is_free[x])
            at = {x: i for i, x in enumerate(R)}
            A = np.zeros((len(R), len(S)))
            for j, y in enumerate(S):
                for x, v in entries[y].items():
                    if is_free[x]:
                        A[at[x], j] = v
            rhs = np.zeros(len(R))
            rhs[at[e]] = 1.0
            # scaled: the entries' sizes depend on the units
            s = np.abs(A).max()
            m = np.linalg.lstsq(A / s, rhs, rcond=None)[0] / s
            keep = np.abs(m) >= 1e-4 * np.abs(m).max()
            rows.append(np.array(S)[keep])
            cols.append(np.full(int(keep.sum()), e))
            vals.append(m[keep])
        rows, cols, vals = (np.concatenate(x) for x in (rows, cols, vals))
        self.M = (np.concatenate([rows, cols]), np.concatenate([cols, rows]),
                  0.5 * np.concatenate([vals, vals]))

    def times(self, r):
        i, j, v = self.M
        return np.bincount(i, v * r[j], len(self.edges))

    def locate(self, z, rho):
        """(triangle, barycentric coordinates) of every point."""
        tri, lam = np.zeros(len(z), np.int64), np.zeros((len(z), 3))
        p0 = self.nodes[self.tris[:, 0]]
        for i in range(0, len(z), 512):
            q = np.stack([z[i:i + 512], rho[i:i + 512]], 1)
            l = np.einsum("tkd,ptd->ptk", self.grad, q[:, None, :] - p0[None])
            l[:, :, 0] += 1.0
            t = l.min(2).argmax(1)
            tri[i:i + 512], lam[i:i + 512] = t, l[np.arange(len(q)), t]
        return tri, lam


class _PlainSim:
    """One cycle of the method: B, particles (Boris, rotate-back, walk, currents), E."""

    def __init__(self, m, E, parts, qm, q_src, dt):
        self.m, self.dt, self.qm, self.q_src = m, dt, qm, q_src
        self.E, self.B, self.J = np.zeros(len(m.edges)), np.zeros(len(m.tris)), np.zeros(len(m.edges))
        self.E[m.free] = E[m.free]
        self.parts = parts is not None
        if self.parts:
            self.tri, self.lam = m.locate(parts[0], parts[1])
            self.u = np.stack(parts[2:], 1)

    def step(self):
        m, dt = self.m, self.dt
        B = self.B - dt * (m.sign * self.E[m.tri_edge]).sum(1)
        self.J = np.zeros(len(m.edges))
        if self.parts:
            self._push(0.5 * (B + self.B))
        self.B = B
        r = np.bincount(m.tri_edge.ravel(), (m.sign * (m.mu_inv * B)[:, None]).ravel(), len(m.edges)) - self.J
        self.E[m.free] += dt * m.times(r)[m.free]

    def _push(self, Bavg):
        m, dt, c2 = self.m, self.dt, self.m.c ** 2
        live = np.flatnonzero(self.tri >= 0)
        t, l, u = self.tri[live], self.lam[live], self.u[live]
        e = m.sign[t] * self.E[m.tri_edge[t]]
        g = m.grad[t]
        w = [l[:, (k + 1) % 3, None] * g[:, (k + 2) % 3] - l[:, (k + 2) % 3, None] * g[:, (k + 1) % 3]
             for k in range(3)]
        Ef = sum(e[:, k, None] * w[k] for k in range(3))
        h = 0.5 * self.qm * dt
        kick = h * np.stack([Ef[:, 1], 0.0 * Ef[:, 0], Ef[:, 0]], 1)
        um = u + kick
        tv = np.zeros_like(um)
        tv[:, 1] = h * Bavg[t] / m.area[t] / np.sqrt(1.0 + (um * um).sum(1) / c2)
        up = um + np.cross(um, tv)
        u = um + np.cross(up, 2.0 * tv / (1.0 + (tv * tv).sum(1, keepdims=True))) + kick
        v = u / np.sqrt(1.0 + (u * u).sum(1, keepdims=True) / c2)
        rho = (l * m.nodes[m.tris[t]][:, :, 1]).sum(1)
        x, y = rho + v[:, 0] * dt, v[:, 1] * dt
        rn = np.hypot(x, y)
        self.u[live] = np.stack([(x * u[:, 0] + y * u[:, 1]) / rn, (x * u[:, 1] - y * u[:, 0]) / rn, u[:, 2]], 1)
        self._walk(live, t, l, np.stack([v[:, 2] * dt, rn - rho], 1))

    def _walk(self, who, t, l, d):
        """Straight meridian segments, cut at every edge that they cross."""
        m = self.m
        entered = np.full(len(who), -1)
        rows = lambda n: np.arange(n)  # noqa: E731
        for _ in range(16):
            if not len(who):
                return
            le = l + np.einsum("pkd,pd->pk", m.grad[t], d)
            out = (le < 0.0) & (entered[:, None] != rows(3))
            with np.errstate(divide="ignore", invalid="ignore"):
                s = np.where(out, l / (l - le), 2.0)
            k, cut = s.argmin(1), out.any(1)
            s = np.where(cut, s[rows(len(k)), k], 1.0)
            end = np.where(cut[:, None], l + s[:, None] * (le - l), le)
            end[cut, k[cut]] = 0.0
            end /= end.sum(1, keepdims=True)
            for q in range(3):
                a, b = (q + 1) % 3, (q + 2) % 3
                cur = m.sign[t, q] * (l[:, a] * end[:, b] - l[:, b] * end[:, a])
                self.J += self.q_src / self.dt * np.bincount(m.tri_edge[t, q], cur, len(m.edges))
            axis = cut & (m.tag[t, k] == W.BC_AXIS)
            stay = ~cut | axis
            self.tri[who[stay]], self.lam[who[stay]] = t[stay], end[stay]
            nb = m.nbr[t, k]
            self.tri[who[~stay & (nb < 0)]] = -1
            go = np.flatnonzero(~stay & (nb >= 0))
            k, nb, old, point = k[go], nb[go], t[go], end[go]
            # the two shared nodes keep their coordinates
            l = np.zeros((len(go), 3))
            for q in range(3):
                for j in range(3):
                    l[:, q] += np.where(m.tris[nb, q] == m.tris[old, j], point[:, j], 0.0)
            entered = (m.nbr[nb] == old[:, None]).argmax(1)
            d = (d * (1.0 - s)[:, None])[go]
            who, t = who[go], nb
        self.tri[who] = -1

    def charge(self):
        live = self.tri >= 0
        return self.q_src * np.bincount(self.m.tris[self.tri[live]].ravel(), self.lam[live].ravel(),
                                        len(self.m.nodes))

    def by_id(self):
        live = self.tri >= 0
        out = np.zeros((len(self.tri), 5))
        out[live, :2] = (self.lam[live][:, :, None] * self.m.nodes[self.m.tris[self.tri[live]]]).sum(1)
        out[live, 2:] = self.u[live]
        return out
