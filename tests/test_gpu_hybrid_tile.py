"""Hybrid grid, the IFE mesh twice as fine: bins of 4 cells deposit into a tile
of IFE nodes in shared memory, bins of 8 straight onto the nodes.  Both add the
same integers, so the node charges are the same bit for bit."""
import numpy as np
import pytest

from paper_2011_10214_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,npart", [((3, 2, 2), 40), ((13, 9, 7), 5000), ((8, 8, 8), 60000), ((17, 4, 5), 33)])
def test_tile_and_direct_deposits_agree(n, npart):
    from paper_2011_10214_gb300 import capi
    x, y, z, vx, vy, vz = wl.random_particles(n, npart, npart, vth=0.3)
    X = np.stack([x, y, z])
    # on and just below cell and half-cell faces, where the IFE cell changes
    g = np.random.default_rng(npart)
    pick = g.integers(0, 4, X.shape) == 0
    X[pick] = np.floor(X[pick]) + g.choice([0.0, 0.5, 1 - 2.0 ** -24, 0.5 - 2.0 ** -25, 2.0 ** -30], int(pick.sum()))
    charges = []
    for edge in (4, 8):
        sim = capi.Simulation(n, 0.5, 0.2, precision=1, track_ids=True, ife_refine=2)
        sim.set_bin_edge(edge)
        sim.set_field_bc([("D", 0.0)] * 6)
        sim.set_object(capi.OBJ_NONE, [], 1.0, 1.0)
        sim.add_species(-1.0, 1.0, 0.01)
        sim.load_particles(0, *X, vx, vy, vz, np.arange(npart, dtype=np.int64))
        sim.set_external_E(wl.random_node_field((2 * n[0] + 1) * (2 * n[1] + 1) * (2 * n[2] + 1), 3, scale=0.3))
        out = []
        for _ in range(3):
            sim.step(1)
            out.append(sim.node_charge(0))
        charges.append(out)
        sim.close()
    for a, b in zip(*charges):
        assert a.any() and np.array_equal(a, b)
