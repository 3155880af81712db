"""Routes inside the FP64 kernels that must give what the plain route gives.

The push takes a particle's cell, floor and weights from the bits of its
position and puts the leavers of a bin aside, 256 at a time; the PCG sums its
dot products in fixed point where the previous totals give a scale, and by
partial sums where they do not."""
import numpy as np
import pytest

from paper_2011_10214_gb300 import workloads as wl
from tests.pairs import add_species_both, by_id, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["sphere16", "ragged"])
@pytest.mark.parametrize("n,vth", [(1, 0.1), (255, 30.0), (257, 30.0), (1500, 5.0), (4000, 30.0)])
def test_push_bit_exact_at_cell_edges_and_with_many_leavers(case, n, vth):
    """One bin at the mesh's corner, full of positions on cell faces, at -0,
    just below a face and denormal, up to all of them leaving at once."""
    gpu, orc = make_pair(case, dt=0.3)
    add_species_both(gpu, orc, -1.0, 1.0, 0.01)
    g = np.random.default_rng(n)
    X = g.uniform(0.0, 3.999, (3, n))
    edge = np.array([-0.0, 0.0, 5e-324, 1e-310, 1.0, 2.0, 3.0, np.nextafter(1.0, 0.0), np.nextafter(4.0, 0.0)])
    pick = g.integers(0, 4, (3, n)) == 0
    X[pick] = edge[g.integers(0, len(edge), int(pick.sum()))]
    V = g.normal(0, vth, (3, n))
    V[:, ::5] = 0.0
    ids = np.arange(n, dtype=np.int64)
    gpu.load_particles(0, X[0], X[1], X[2], V[0], V[1], V[2], ids)
    orc.load_particles(0, X[0], X[1], X[2], V[0], V[1], V[2], ids)
    E = wl.random_node_field(orc.mesh.nnodes, 3, scale=0.3)
    gpu.set_external_E(E); orc.set_external_E(E)
    for _ in range(3):
        sg, so = gpu.step(1), orc.step()
        assert sg["absorbed"][0] == so["absorbed"][0] and sg["pushed"][0] == so["pushed"][0]
        a, b = by_id(gpu.particles(0)), by_id(orc.P[0])
        assert np.array_equal(a["id"], b["id"])
        for k in ("x", "y", "z", "vx", "vy", "vz"):
            assert np.array_equal(a[k], b[k]), k
        assert np.array_equal(gpu.node_charge(0), orc.W[0])
    gpu.close()


@pytest.mark.parametrize("n", [(5, 4, 3), (16, 16, 16), (33, 20, 27)])
def test_solve_sums_in_fixed_point_and_by_partials_agree(n):
    """Loads 2^-350 times as large put every total out of the fixed-point range:
    the same solve by partial sums.  Both stop at |r| <= 1e-13 |b|, so they agree
    to 2e-13 times the operator's condition (below 1e3 on these meshes)."""
    from paper_2011_10214_gb300 import capi
    scale = 2.0 ** -350
    g = np.random.default_rng(sum(n))
    nodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    F = g.normal(0, 1, nodes)
    phi = []
    for s in (1.0, scale):
        sim = capi.Simulation(n, 0.5, 0.1, precision=0, pcg_tol=1e-13, pcg_max_iter=2000)
        sim.set_field_bc([("D", 0.0)] * 6)
        sim.set_object(capi.OBJ_NONE, [], 1.0, 1.0)
        iters, relres = sim.solve_field(F * s)
        assert 0 < iters < 2000 and relres <= 1e-13
        phi.append(sim.potential() / s)
        sim.close()
    assert np.abs(phi[0]).max() > 0
    assert np.abs(phi[0] - phi[1]).max() <= 2e-10 * np.abs(phi[0]).max()


def test_sums_out_of_range_inside_a_solve():
    """A load that is one eigenvector of D^-1 A and, 1e-5 as large, all the others: the first
    iteration takes the totals down by 1e8 or more, far below the 1/128 of the last ones that
    the fixed-point sums reach, so they are redone by partial sums there and in fixed point
    again after it.  Both sides stop at |r| <= 1e-12 |b| (condition below 100 here)."""
    from oracle.field import FieldSystem
    from oracle.geometry import Mesh, NoObject
    from paper_2011_10214_gb300 import capi
    n = (9, 7, 8)
    bc = [("D", 0.0)] * 6
    m = Mesh(*n, 0.5)
    fs = FieldSystem(m, NoObject(), bc)
    A = fs.A_ff.toarray()
    d = np.sqrt(A.diagonal())
    _, V = np.linalg.eigh(A / np.outer(d, d))            # D^-1/2 A D^-1/2; r = D^1/2 v is D times an eigenvector
    c = np.full(len(d), 1e-5)
    c[len(d) // 3] = 1.0
    F = np.zeros(m.nnodes)
    F[fs.free] = d * (V @ c)
    one, _, rr = fs.solve(F, np.zeros(0), tol=1e-3, maxit=5)
    assert rr < 1e-3                                     # (one step: |r|^2 down by more than 1e6)
    phi, it, _ = fs.solve(F, np.zeros(0), tol=1e-12, maxit=500)
    assert it > 10
    sim = capi.Simulation(n, 0.5, 0.1, precision=0, pcg_tol=1e-12, pcg_max_iter=500)
    sim.set_field_bc(bc)
    sim.set_object(capi.OBJ_NONE, [], 1.0, 1.0)
    git, relres = sim.solve_field(F)
    assert abs(git - it) <= 2 and relres <= 1e-12
    assert np.abs(sim.potential() - phi).max() <= 1e-10 * np.abs(phi).max()
    sim.close()
