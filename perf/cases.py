"""What the performance of this framework is measured on.

A case is one pass of a user's program through the library's public entry
points: a few PIC steps of one simulation and a read-back of its potential and
charge densities (`step`), the same for a batch of independent simulations
(`batch`), a field solve for given loads (`solve`), or frozen-field steps with a
read-back of every particle by id (`track`).  The set-ups are those of
paper_2011_10214_gb300.workloads (its sphere, eighth-sphere, crater and lunar
configurations at their own or other sizes) with the library's default solver
settings; read-backs go to device arrays through the C ABI, as a host program
that keeps its diagnostics on the GPU does.

listed, draw, prepare, run, work, tolerance and exact are described where they
are defined.
"""
import ctypes as C
import math
import random

import torch

from paper_2011_10214_gb300 import capi
from paper_2011_10214_gb300 import workloads as wl

DEV = "cuda"


# ---- the cases ---------------------------------------------------------------

def listed():
    return [
        # the smallest run: the 16^3 validation sphere in plain FP64, latency only
        dict(name="step_sphere16_fp64", kind="step", setup="sphere", precision="fp64", nx=16, ppc=16, radius=2.0,
             eps=4.0, edge=4, refine=1, steps=4),
        # the same problem in the speed mode
        dict(name="step_sphere16", kind="step", setup="sphere", precision="mixed", nx=16, ppc=16, radius=2.0, eps=4.0,
             edge=4, refine=1, steps=8),
        # an odd-sized box (37 cells a side, bins and solver tiles ragged), as a served request is
        dict(name="step_sphere37", kind="step", setup="sphere", precision="mixed", nx=37, ppc=27, radius=4.7, eps=7.5,
             edge=4, refine=1, steps=4),
        # the headline workload: 64^3 cells, 32.6M particles
        dict(name="step_sphere64", kind="step", setup="sphere", precision="mixed", nx=64, ppc=64, radius=6.0, eps=4.0,
             edge=4, refine=1, steps=2),
        # the FP64 contract on a mid-size run, particles bound by the FP64 pipe
        dict(name="step_sphere40_fp64", kind="step", setup="sphere", precision="fp64", nx=40, ppc=32, radius=4.0,
             eps=4.0, edge=4, refine=1, steps=1),
        # the paper's eighth-sphere validation: reflecting symmetry planes, mass ratio 1836
        dict(name="step_oml50", kind="step", setup="oml", precision="mixed", nx=50, ppc=125, radius=0.401, eps=4.0,
             edge=4, refine=1, steps=2),
        # the lunar crater at half resolution: layered ground, half crater, photoelectrons, mostly Neumann
        dict(name="step_lunar100", kind="step", setup="lunar", precision="mixed", nx=100, ppc=64, radius=0.0, eps=4.0,
             edge=4, refine=1, steps=1),
        # the largest: 160 x 160 x 80 crater, 390M particles, photoelectrons
        dict(name="step_crater160", kind="step", setup="crater", precision="mixed", nx=160, ppc=125, radius=0.0,
             eps=4.0, edge=4, refine=1, steps=1),
        # hybrid grid: the field mesh refined twice per axis
        dict(name="step_sphere32_h2", kind="step", setup="sphere", precision="mixed", nx=32, ppc=64, radius=3.0,
             eps=4.0, edge=4, refine=2, steps=2),
        # many independent problems at once, drawn as a server's requests are
        dict(name="batch24", kind="batch", members=24, mix=1, precision="mixed", steps=2),
        # a field solver's caller: loads that change from call to call, 64^3
        dict(name="solve_sphere64", kind="solve", precision="mixed", nx=64, ny=64, nz=64, radius=6.0, eps=4.0,
             neumann=0),
        # particle tracking in a given field: closed reflecting box, every particle read back by id
        dict(name="track25", kind="track", precision="mixed", nx=25, ny=23, nz=27, ppc=64, steps=4),
    ]


def draw(rng):
    """One more case: the kinds in the proportions of use, sizes over the ranges
    of the listed ones (spread over their logarithm)."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["step"] * 7 + ["batch", "solve", "solve", "track"])
    if kind == "step":
        setup = rng.choice(["sphere"] * 4 + ["oml", "crater", "lunar"])
        c = dict(kind="step", setup=setup, precision="mixed", ppc=log_int(8, 125), eps=round(rng.uniform(2.0, 10.0), 2),
                 radius=0.0, edge=4, refine=1, steps=rng.choice([1, 2, 4]))
        if setup in ("sphere", "oml"):
            c["nx"] = log_int(13, 97)
            c["radius"] = round(rng.uniform(0.08, 0.28) * c["nx"] * (0.5 if setup == "sphere" else 0.1), 3)
            if setup == "sphere" and c["nx"] <= 41:
                c["precision"] = rng.choice(["mixed", "mixed", "fp64"])
                c["refine"] = rng.choice([1, 1, 2]) if c["precision"] == "mixed" else 1
        else:
            c["nx"] = log_int(40, 150)
        if c["precision"] == "mixed" and c["ppc"] <= 48:
            c["edge"] = rng.choice([4, 4, 8])
        return c
    if kind == "batch":
        return dict(kind="batch", members=log_int(3, 32), mix=rng.randrange(1 << 20), precision="mixed",
                    steps=rng.choice([1, 2]))
    if kind == "solve":
        nx, ny, nz = (log_int(13, 110) for _ in range(3))
        return dict(kind="solve", precision=rng.choice(["mixed", "mixed", "fp64"]), nx=nx, ny=ny, nz=nz,
                    radius=round(rng.uniform(0.1, 0.3) * 0.5 * min(nx, ny, nz), 3), eps=round(rng.uniform(2.0, 10.0), 2),
                    neumann=rng.choice([0, 0, 1, 4, 21]))
    return dict(kind="track", precision=rng.choice(["fp64", "mixed"]), nx=log_int(9, 49), ny=log_int(9, 49),
                nz=log_int(9, 49), ppc=log_int(4, 64), steps=rng.choice([1, 4]))


PRECISION = {"fp64": capi.FP64, "mixed": capi.MIXED}


def _config(c):
    """The workload dict (paper_2011_10214_gb300.workloads) of a step case."""
    n, ppc = c["nx"], c["ppc"]
    if c["setup"] == "sphere":
        cfg = wl.sphere_config(n, c["radius"], ppc, 1, eps_in=c["eps"])
    elif c["setup"] == "oml":
        cfg = wl.oml_eighth_config(n=n, radius=c["radius"], ppc=ppc, eps_in=c["eps"])
    elif c["setup"] == "crater":
        s = n / 160.0
        cfg = wl.crater_config(nx=n, ny=n, nz=max(n // 2, 8), z_ground=20.0 * s, rim_radius=30.0 * s, depth=10.0 * s,
                               ppc=ppc)
        cfg["object"]["eps_in"] = c["eps"]
    else:
        s = n / 200.0
        cfg = wl.lunar_config(nx=n, ny=max(n // 2, 8), nz=max(n // 2, 8), z_ground=9.5 * s, z_bed=4.5 * s,
                              r_inner=10.5 * s, r_top=20.2 * s, r_outer=30.9 * s, height=2.7 * s, depth=4.0 * s,
                              ppc=ppc)
        cfg["object"]["eps_in"] = c["eps"]
    cfg["ife_refine"] = c["refine"]
    return cfg


def _mix(c):
    """The members of a batch: boxes of 16 to 48 cells a side, radii 1 to 8
    Debye lengths, permittivities 2 to 10, 16 to 64 particles per cell."""
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["members"]):
        n, ppc = rng.randint(16, 48), rng.randint(16, 64)
        out.append(wl.sphere_config(n, min(rng.uniform(1.0, 8.0), 0.15 * n), ppc, 1, eps_in=rng.uniform(2.0, 10.0)))
    return out


# ---- what a program has in hand -------------------------------------------------

def _densities_scale(cfg):
    """Charge density per unit of a species' node charge (2^32 units a particle)."""
    species = cfg["species"] + ([cfg["photo"]] if cfg.get("photo") else [])
    return [(sp["q"] * (sp["weight"] if "weight" in sp else wl.macro_weight(cfg, sp))) / (2.0 ** 32 * cfg["h"] ** 3)
            for sp in species]


def _start(cfg, precision, seed, edge=4):
    """A simulation after its initial solve and leapfrog start."""
    cfg = dict(cfg, seed=wl.SEED_BASE + seed)
    sim = capi.from_config(cfg, precision=PRECISION[precision], bin_edge=edge)
    sim.solve()
    sim.leapfrog_init()
    return sim


def _readers(sim, cfg):
    """Device buffers for a simulation's potential, charges and surface counts."""
    sz = sim.sizes()
    return dict(phi=torch.empty(sz["nnodes"], dtype=torch.float64, device=DEV),
                W=torch.empty((sim.nspecies, sz["nnodes"]), dtype=torch.int64, device=DEV),
                surf=torch.zeros((sim.nspecies, sz["n_cut_cells"]), dtype=torch.int64, device=DEV),
                scale=torch.tensor(_densities_scale(cfg), dtype=torch.float64, device=DEV)[:, None])


def prepare(case, seed):
    """A running simulation (after its start and two steps), a batch of them, a
    solver with its ring of loads, or a box of particles in a given field."""
    kind = case["kind"]
    if kind == "step":
        cfg = _config(case)
        sim = _start(cfg, case["precision"], seed, case["edge"])
        sim.step(2)
        return dict(kind=kind, sim=sim, steps=case["steps"], out=_readers(sim, cfg))
    if kind == "batch":
        cfgs = _mix(case)
        sims = [_start(cfg, case["precision"], seed + 1000 * i) for i, cfg in enumerate(cfgs)]
        batch = capi.Batch(sims)
        batch.step(2)
        return dict(kind=kind, batch=batch, sims=sims, steps=case["steps"],
                    phi=torch.empty(sum(s.sizes()["nnodes"] for s in sims), dtype=torch.float64, device=DEV),
                    W=torch.empty(2 * sum(s.sizes()["nnodes"] for s in sims), dtype=torch.int64, device=DEV))
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    nn = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    if kind == "solve":
        sim = capi.Simulation(n, SOLVE_H, 0.05, precision=PRECISION[case["precision"]], pcg_max_iter=SOLVE_CAP)
        sim.set_field_bc(_solve_bc(case))
        sim.set_object(capi.OBJ_SPHERE, [*(0.5 * SOLVE_H * v for v in n), case["radius"]], case["eps"], 1.0)
        loads, q = _solve_loads(case, seed), _solve_jump(sim.sizes()["n_interface_tets"])
        for F in loads[-2:]:   # the caller's earlier loads
            sim.solve_field(F, q)
        return dict(kind=kind, sim=sim, loads=loads, q=q, calls=0, phi=torch.empty(nn, dtype=torch.float64, device=DEV),
                    E=torch.empty((nn, 3), dtype=torch.float32, device=DEV))
    x, v, E = _track_inputs(case, g)
    sim = capi.Simulation(n, 1.0, TRACK_DT, precision=PRECISION[case["precision"]], track_ids=True)
    sim.set_object(capi.OBJ_NONE, [], 1.0, 1.0)
    s = sim.add_species(-1.0, 1.0, 1.0)
    sim.set_particle_bc(s, ["reflect"] * 6)
    ids = torch.arange(x.shape[1], device=DEV)
    sim.load_particles(s, *x, *v, ids)
    sim.set_external_E(E)
    k = x.shape[1]
    return dict(kind=kind, sim=sim, steps=case["steps"], n=k, ids=torch.empty(k, dtype=torch.int64, device=DEV),
                flat=torch.empty((6, k), dtype=torch.float64, device=DEV),
                W=torch.empty(nn, dtype=torch.int64, device=DEV))


SOLVE_H = 0.5
SOLVE_CAP = 1000   # iterations: a caller of the solver alone wants its tolerance met
RING = 32   # loads of a solve case: a closed ring, neighbours as alike as a PIC run's consecutive steps
TRACK_DT = 0.05


def _solve_bc(case):
    """Field boundary: bit f of `neumann` makes face f zero-Neumann, else a Dirichlet value of its own."""
    return [("N",) if case["neumann"] >> f & 1 else ("D", 0.1 * f) for f in range(6)]


def _solve_loads(case, seed):
    """Loads of a plasma: the shot noise of 64 particles a cell and species on a smooth net charge."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ax = [torch.linspace(0, math.pi, m + 1, dtype=torch.float64, device=DEV).sin() for m in (nx, ny, nz)]
    h3 = SOLVE_H ** 3
    smooth = 0.05 * h3 * (ax[2][:, None, None] * ax[1][None, :, None] * ax[0][None, None, :]).reshape(-1)
    noise = 0.1 * h3 * torch.randn((2, smooth.numel()), dtype=torch.float64, device=DEV, generator=g)
    t = [2 * math.pi * k / RING for k in range(RING)]
    return [smooth + math.cos(a) * noise[0] + math.sin(a) * noise[1] for a in t]


def _solve_jump(nit):
    """The flux jump of a charged surface, varying over its interface tets."""
    return -0.4 + 0.2 * torch.sin(0.37 * torch.arange(nit, dtype=torch.float64, device=DEV))


def _track_inputs(case, g):
    """Positions in cell units, velocities and the field of a track case."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    k = nx * ny * nz * case["ppc"]
    x = torch.rand((3, k), dtype=torch.float64, device=DEV, generator=g)
    x *= torch.tensor([[nx], [ny], [nz]], dtype=torch.float64, device=DEV)
    v = torch.randn((3, k), dtype=torch.float64, device=DEV, generator=g)
    E = 0.5 * torch.randn(((nx + 1) * (ny + 1) * (nz + 1), 3), dtype=torch.float64, device=DEV, generator=g)
    return x, v, E


# ---- one pass ----------------------------------------------------------------------

def _ok(status, what):
    if status != 0:
        raise RuntimeError(f"{what}: status {status}")


def _read(fn, sim, *args):
    _ok(fn(sim._c, *args), fn.__name__)


def run(state):
    """One pass; see the kinds in the module's docstring."""
    kind = state["kind"]
    lib = capi.lib
    if kind == "step":
        sim, out = state["sim"], state["out"]
        st = sim.step(state["steps"])
        _read(lib.pifepic_get_potential, sim, out["phi"].data_ptr(), capi.DEVICE)
        for s in range(sim.nspecies):
            _read(lib.pifepic_get_node_charge, sim, s, out["W"][s].data_ptr(), capi.DEVICE)
            if out["surf"].shape[1]:
                _read(lib.pifepic_get_surface_charge, sim, s, out["surf"][s].data_ptr(), capi.DEVICE)
        # species apart: their sum is small where the plasma is neutral
        return dict(phi=out["phi"], rho=out["W"] * out["scale"], surface=out["surf"].double(),
                    alive=torch.tensor(st["count"], dtype=torch.float64), potential=st["surface_potential"])
    if kind == "batch":
        st = state["batch"].step(state["steps"])
        p = w = 0
        for sim in state["sims"]:
            nn = (sim.n[0] + 1) * (sim.n[1] + 1) * (sim.n[2] + 1)
            _read(lib.pifepic_get_potential, sim, state["phi"].data_ptr() + 8 * p, capi.DEVICE)
            p += nn
            for s in range(sim.nspecies):
                _read(lib.pifepic_get_node_charge, sim, s, state["W"].data_ptr() + 8 * w, capi.DEVICE)
                w += nn
        return dict(phi=state["phi"], W=state["W"].double(),
                    alive=torch.tensor([n for x in st for n in x["count"]], dtype=torch.float64))
    sim = state["sim"]
    if kind == "solve":
        F = state["loads"][state["calls"] % RING]
        state["calls"] += 1
        sim.solve_field(F, state["q"])
        _read(lib.pifepic_get_potential, sim, state["phi"].data_ptr(), capi.DEVICE)
        _read(lib.pifepic_get_node_E_f32, sim, state["E"].data_ptr(), capi.DEVICE)
        return dict(phi=state["phi"], E=state["E"])
    sim.step(state["steps"])
    flat, ids, got = state["flat"], state["ids"], C.c_int64()
    _read(lib.pifepic_get_particles, sim, 0, state["n"], *(flat[d].data_ptr() for d in range(6)), ids.data_ptr(),
          C.byref(got), capi.DEVICE)
    _read(lib.pifepic_get_node_charge, sim, 0, state["W"].data_ptr(), capi.DEVICE)
    by_id = torch.empty_like(flat)
    by_id[:, ids] = flat
    return dict(x=by_id[:3], v=by_id[3:], W=state["W"].double())


# ---- what a pass cannot do without -----------------------------------------------------

def _particles(cfg):
    """Particles of a loaded configuration: the cells in the plasma, roughly."""
    n = cfg["n"]
    cells = n[0] * n[1] * n[2]
    ob = cfg["object"]
    if ob["kind"] == "sphere":
        part = 0.125 if cfg.get("particle_bc") else 1.0
        cells -= part * 4.0 / 3.0 * math.pi * (ob["radius"] / cfg["h"]) ** 3
    elif "z_ground" in ob:
        cells -= n[0] * n[1] * ob["z_ground"] / cfg["h"]
    return sum(sp["ppc"] for sp in cfg["species"]) * cells


def _step_work(cfg, fp64, refine):
    """One PIC step: every particle's state read and written once (48 or 28
    bytes), each species' node charges written and read once (8 bytes), the
    potential read and written and the node field written.  Operations: about 75
    for the gather, 15 for kick, drift and tests, 30 for the deposit, a particle;
    60 a node for one residual and the node field."""
    n = cfg["n"]
    nodes = (n[0] * refine + 1) * (n[1] * refine + 1) * (n[2] * refine + 1)
    p = _particles(cfg)
    ns = len(cfg["species"]) + (1 if cfg.get("photo") else 0)
    b = p * 2 * (48 if fp64 else 28) + nodes * (16 * ns + 16 + (24 if fp64 else 12))
    return b, 120.0 * p + 60.0 * nodes


def work(case):
    kind = case["kind"]
    if kind == "step":
        b, f = _step_work(_config(case), case["precision"] == "fp64", case["refine"])
        nodes = math.prod(v * case["refine"] + 1 for v in _config(case)["n"])
        return dict(bytes=case["steps"] * b + 40.0 * nodes, flops=case["steps"] * f)
    if kind == "batch":
        w = [_step_work(c, False, 1) for c in _mix(case)]
        return dict(bytes=case["steps"] * sum(x[0] for x in w), flops=case["steps"] * sum(x[1] for x in w))
    nn = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    if kind == "solve":   # the load read, the potential and the node field written; one residual's operations
        return dict(bytes=nn * (8.0 + 8.0 + 12.0), flops=60.0 * nn)
    p = case["nx"] * case["ny"] * case["nz"] * case["ppc"]
    size = 48 if case["precision"] == "fp64" else 28
    # the state in and out per step, and the read-back by id
    return dict(bytes=p * (2.0 * size * case["steps"] + 2 * 56.0) + nn * 8.0, flops=120.0 * p * case["steps"])


def tolerance(case):
    kind = case["kind"]
    if kind == "track":
        # FP64: rounding of the same operations in another order; MIXED: offsets and velocities of 24 bits
        return dict(rel=1e-12, max=1e-9) if case["precision"] == "fp64" else dict(rel=3e-6, max=1e-4)
    if kind == "solve":
        # seen: 2e-6 (2-norm) and 5e-6 (largest) from solves stopped at 1e-10, 1.2e-5 in the FP32 field
        return dict(rel=1e-5, max=1e-4)
    # a solve stops at a relative residual of 1e-6; the potential of solvers that stop there (Jacobi, multigrid, plain
    # FP64) was seen up to 8e-5 (2-norm) and 2e-4 (largest) from one stopped at 1e-10, charges and counts far less
    return dict(rel=4e-4, max=1e-3)


# ---- the same in 64 bits ------------------------------------------------------------------

def exact(case, seed):
    """Plain torch in 64 bits for the kinds whose result is a function of the
    inputs made here; a running simulation's particles come from the library's
    own random streams."""
    if case["kind"] == "track":
        return _exact_track(case, seed)
    if case["kind"] == "solve":
        return dict(phi=_exact_solve(case, seed), E=None)
    return None


def _corners(n, x):
    """Node indices (8, k) and trilinear weights of positions in cell units."""
    c = x.floor()
    f = x - c
    i, j, k = (c[d].long() for d in range(3))
    idx, w = [], []
    for l in range(8):
        a, b, d = l & 1, l >> 1 & 1, l >> 2 & 1
        idx.append((i + a) + (n[0] + 1) * ((j + b) + (n[1] + 1) * (k + d)))
        w.append((f[0] if a else 1 - f[0]) * (f[1] if b else 1 - f[1]) * (f[2] if d else 1 - f[2]))
    return idx, w


def _exact_track(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    x, v, E = _track_inputs(case, g)
    n = (case["nx"], case["ny"], case["nz"])
    for _ in range(case["steps"]):
        idx, w = _corners(n, x)
        for d in range(3):
            v[d] -= TRACK_DT * sum(wl_ * E[i, d] for i, wl_ in zip(idx, w))
        x = x + TRACK_DT * v
        for d in range(3):
            lo, hi = x[d] < 0, x[d] >= n[d]
            x[d] = torch.where(lo, -x[d], torch.where(hi, 2.0 * n[d] - x[d], x[d]))
            v[d] = torch.where(lo | hi, -v[d], v[d])
    idx, w = _corners(n, x)
    W = torch.zeros((n[0] + 1) * (n[1] + 1) * (n[2] + 1), dtype=torch.float64, device=DEV)
    for i, a in zip(idx, w):
        W.index_add_(0, i, a * 2.0 ** 32)
    return dict(x=x, v=v, W=W)


def _tets(case):
    """The 5-tet split of every cell: (5 ncells, 4) nodes in (cell, tet) order and (5 ncells, 4, 3) vertex offsets."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    off = torch.tensor([[l & 1, l >> 1 & 1, l >> 2 & 1] for l in range(8)], device=DEV)
    table = []
    for parity in range(2):
        even = [l for l in range(8) if bin(l).count("1") % 2 == parity]
        odd = [l for l in range(8) if bin(l).count("1") % 2 != parity]
        table.append([even] + [[o, o ^ 1, o ^ 2, o ^ 4] for o in odd])
    table = torch.tensor(table, device=DEV)
    k, j, i = torch.meshgrid(torch.arange(nz, device=DEV), torch.arange(ny, device=DEV),
                             torch.arange(nx, device=DEV), indexing="ij")
    cell = torch.stack([i, j, k], -1).reshape(-1, 3)
    local = table[cell.sum(1) % 2].reshape(-1, 4)                     # (5 ncells, 4)
    at = cell.repeat_interleave(5, 0)[:, None, :] + off[local]
    nodes = at[..., 0] + (nx + 1) * (at[..., 1] + (ny + 1) * at[..., 2])
    return nodes, at.double() * SOLVE_H


def _p1(X):
    """Basis gradients (m, 4, 3) and volumes of tets with vertices X (m, 4, 3)."""
    M = torch.cat([torch.ones_like(X[..., :1]), X], -1)
    inv = torch.linalg.inv(M)
    return inv[:, 1:, :].transpose(1, 2), torch.linalg.det(M).abs() / 6


def _ife(X, L, em, ep):
    """Stiffness (m, 4, 4) and unit flux-jump load (m, 4) of interface tets: the
    linear immersed basis, continuous across the cut plane, with the flux jump
    [eps dn psi] = q, on exact sub-volumes."""
    m = X.shape[0]
    minus = L < 0
    o = X[:, :1].clone()
    X = X - o
    g, V = _p1(X)
    n = torch.einsum("mv,mvd->md", L, g)
    gl = n.norm(dim=1, keepdim=True)
    n = n / gl
    d = L / gl                                                         # signed distances of the vertices
    # columns 0..3: nodal basis, 4: unit jump (zero at the nodes); psi+ = a + b.x
    A = torch.zeros((m, 4, 4), dtype=torch.float64, device=DEV)
    A[:, :, 0] = 1
    A[:, :, 1:] = X + (minus * d * ((ep - em) / em))[..., None] * n[:, None, :]
    R = torch.zeros((m, 4, 5), dtype=torch.float64, device=DEV)
    R[:, :, :4] = torch.eye(4, dtype=torch.float64, device=DEV)
    R[:, :, 4] = minus * d / em
    S = torch.linalg.solve(A, R)
    bp = S[:, 1:, :]                                                   # (m, 3, 5)
    beta = (ep - em) / em * torch.einsum("md,mdc->mc", n, bp)
    beta[:, 4] -= 1.0 / em
    bm = bp + n[:, :, None] * beta[:, None, :]
    # minus vertices first; the cut polygon and the minus side's volume
    order = torch.argsort(L, dim=1, stable=True)
    Xs = torch.gather(X, 1, order[..., None].expand(-1, -1, 3))
    Ls = torch.gather(L, 1, order)
    count = minus.sum(1)

    def cut(u, w):
        t = Ls[:, u] / (Ls[:, u] - Ls[:, w])
        return Xs[:, u] + t[:, None] * (Xs[:, w] - Xs[:, u])

    def vol(a, b, c, e):
        return torch.linalg.det(torch.stack([b - a, c - a, e - a], 1)).abs() / 6
    one, two = (count == 1)[:, None], (count == 2)[:, None]
    c01, c02, c03, c12, c13, c23 = cut(0, 1), cut(0, 2), cut(0, 3), cut(1, 2), cut(1, 3), cut(2, 3)
    # polygon p0 p1 p2 (p3): a triangle around the single vertex, or a quadrilateral
    p0 = torch.where(one, c01, torch.where(two, c02, c03))
    p1 = torch.where(one, c02, torch.where(two, c03, c13))
    p2 = torch.where(one, c03, torch.where(two, c13, c23))
    p3 = torch.where(two, c12, p2)
    v1 = vol(Xs[:, 0], c01, c02, c03)
    v3 = V - vol(Xs[:, 3], c03, c13, c23)
    # two and two: the wedge with edge 0-1 and the quadrilateral, as three tets
    v2 = vol(Xs[:, 0], c02, c03, c13) + vol(Xs[:, 0], c02, c13, c12) + vol(Xs[:, 0], Xs[:, 1], c12, c13)
    vm = torch.where(count == 1, v1, torch.where(count == 2, v2, v3))
    vp = V - vm
    K = ep * vp[:, None, None] * (bp.transpose(1, 2) @ bp) + em * vm[:, None, None] * (bm.transpose(1, 2) @ bm)
    gamma = torch.zeros((m, 4), dtype=torch.float64, device=DEV)
    for a, b, c in ((p0, p1, p2), (p0, p2, p3)):
        area = torch.linalg.cross(b - a, c - a).norm(dim=1) / 2
        gamma += area[:, None] * (S[:, 0, :4] + torch.einsum("md,mdc->mc", (a + b + c) / 3, bp[:, :, :4]))
    return K[:, :4, :4], -gamma - K[:, 4, :4]


def _exact_solve(case, seed):
    """The immersed-finite-element potential of the first load, by conjugate gradients to round-off."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nodes, X = _tets(case)
    N = (nx + 1) * (ny + 1) * (nz + 1)
    ids = torch.arange(N, device=DEV)
    at = torch.stack([ids % (nx + 1), ids // (nx + 1) % (ny + 1), ids // ((nx + 1) * (ny + 1))], 1)
    centre = torch.tensor([0.5 * nx, 0.5 * ny, 0.5 * nz], dtype=torch.float64, device=DEV)
    L = ((at - centre) ** 2).sum(1) - (case["radius"] / SOLVE_H) ** 2
    em, ep = case["eps"], 1.0
    inside = (L[nodes] < 0).sum(1)
    whole = (inside == 0) | (inside == 4)
    b = _solve_loads(case, seed)[0]
    rows, cols, vals = [], [], []
    g, V = _p1(X[whole] - X[whole][:, :1])
    K = (torch.where(inside[whole] == 4, em, ep) * V)[:, None, None] * (g @ g.transpose(1, 2))
    Ki, ci = _ife(X[~whole], L[nodes[~whole]], em, ep)
    b.index_add_(0, nodes[~whole].reshape(-1), (_solve_jump(Ki.shape[0])[:, None] * ci).reshape(-1))
    for nd, k in ((nodes[whole], K), (nodes[~whole], Ki)):
        rows.append(nd[:, :, None].expand(-1, 4, 4).reshape(-1))
        cols.append(nd[:, None, :].expand(-1, 4, 4).reshape(-1))
        vals.append(k.reshape(-1))
    A = torch.sparse_coo_tensor(torch.stack([torch.cat(rows), torch.cat(cols)]), torch.cat(vals),
                                (N, N)).coalesce().to_sparse_csr()
    free = torch.ones(N, dtype=torch.bool, device=DEV)
    phi = torch.zeros(N, dtype=torch.float64, device=DEV)
    for f, bc in enumerate(_solve_bc(case)):
        face = (at[:, f // 2] == (nx, ny, nz)[f // 2] * (f & 1)) & free
        if bc[0] == "D":
            phi[face] = bc[1]
            free &= ~face
    mask = free.double()
    r = mask * (b - A @ phi)
    diag = torch.zeros(N, dtype=torch.float64, device=DEV)
    i = torch.cat(rows)
    same = i == torch.cat(cols)
    diag.index_add_(0, i[same], torch.cat(vals)[same])
    z = r / diag
    p, rz, stop = z.clone(), r @ z, 1e-28 * (r @ r)
    for it in range(4000):
        q = mask * (A @ p)
        a = rz / (p @ q)
        phi += a * p
        r -= a * q
        if it % 20 == 0 and r @ r <= stop:
            break
        z = r / diag
        new = r @ z
        p = z + (new / rz) * p
        rz = new
    return phi
