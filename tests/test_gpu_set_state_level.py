"""sww_set_state_level on a handle that has stepped: the levels above the given one start
empty, whatever an earlier state left there, so the run equals that of a fresh handle bit
for bit (a closure mark of the earlier state's last mask used to make points live)."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", ["lists", "dense"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_used_handle_equals_fresh_one(precision, mask):
    import paper_1404_0405_gb300 as sww
    make = lambda: sww.Model(3, 7, patch=4, eps=3e-3, precision=precision, mask=mask)

    def run(m, seed, level):
        xyz, en = m.grid(level)
        m.set_state(*workloads.Workload("jet", seed=seed).fields(xyz, *lib_edge_geometry(xyz, en)), level=level)
        m.adapt()
        m.step(-1.0, 3, True)

    used, fresh = make(), make()
    run(used, 1, 7)
    run(used, 2, 5)
    run(fresh, 2, 5)
    assert used.stats()["live_nodes"] == fresh.stats()["live_nodes"]
    for j in range(3, 8):
        for q in (sww.NODE_FLAGS, sww.EDGE_FLAGS):
            assert np.array_equal(used.get(j, q) & 7, fresh.get(j, q) & 7), (j, q)
        for a, b in zip(used.get_state(j), fresh.get_state(j)):
            assert np.array_equal(a, b), j
