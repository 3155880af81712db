"""Statistics of a step: one launch over the interface tets, the cut cells and
the bins of up to eight contexts, packed by the last block to arrive.  Batches
of one context, of a full group of eight, and of a group and one more, whose
members differ in every extent, must report each member's own numbers: those of
the call that follows with no step in it, the particles the context holds, and
the charge of its surface accumulators."""
import numpy as np
import pytest

from paper_2011_10214_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("members", [1, 8, 9])
def test_batch_statistics_are_each_members_own(members, precision):
    from paper_2011_10214_gb300 import capi
    cfgs = [wl.sphere_config(8 + 2 * i, 0.15 * (8 + 2 * i), 2 + i, 4, eps_in=4.0, seed_offset=i) for i in range(members)]
    sims = []
    for cfg in cfgs:
        s = capi.from_config(cfg, precision=precision, track_ids=False)
        s.solve()
        s.leapfrog_init()
        sims.append(s)
    b = capi.Batch(sims)
    first = b.step(2)
    second = b.step(3)
    b.close()
    for s, cfg, a, z in zip(sims, cfgs, first, second):
        now = s.step(0)
        nsp = len(cfg["species"])
        assert a["steps"] == 2 and z["steps"] == 5
        for q in range(nsp):
            held = len(s.particles(q)["x"])
            assert z["count"][q] == held and now["count"][q] == held
            assert now["pushed"][q] == 0 and now["injected"][q] == 0
            assert z["count"][q] - a["count"][q] == (z["injected"][q] - z["absorbed"][q] - z["collected"][q]
                                                     - z["dropped"][q])
            assert z["pushed"][q] > 0
        # the same sums in another grid's order: FP64 round-off of a few thousand terms
        assert np.isclose(now["surface_charge"], z["surface_charge"], rtol=1e-12, atol=0)
        assert np.isclose(now["surface_potential"], z["surface_potential"], rtol=1e-11, atol=1e-14)
        assert now["pcg_iters_total"] == 0 and z["pcg_iters_total"] >= 3
        s.close()
