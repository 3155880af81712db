"""Routes inside the FP64 kernels that must give what the plain route gives.

The PCG sums its dot products in fixed point where the previous totals give a
scale, and by partial sums where they do not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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
