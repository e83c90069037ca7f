"""A new state on a handle whose last mask had applied a proposal: no proposal belongs to it, so
none of its patches counts as over-refined at its first adaptation."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [5, 4])
def test_earlier_proposal_is_forgotten(level):
    import paper_1404_0405_gb300 as sww
    m = sww.Model(2, 5, patch=4, eps=1e-2)

    def state(seed, j):
        xyz, en = m.grid(j)
        m.set_state(*workloads.Workload("jet", seed=seed).fields(xyz, *lib_edge_geometry(xyz, en)), level=j)

    state(1, 5)
    m.adapt()
    for j in (4, 5):
        m.propose(j, np.ones(m.sizes(j)[3] + 1, np.uint8))
    m.adapt()
    assert m.patch_data(5, sww.P_PROPOSAL).all()
    state(2, level)
    m.learn_stats(reset=True)
    m.adapt()
    got = m.learn_stats()
    assert got["over"] == 0 and got["proposed"] == 0
