"""Live edges of a mask with a learned proposal: an edge is live only when one of its ends is.
A proposed patch lies at the rim of the mask's candidates, and the closure marks parents
beyond them that do not become live; an edge to such a parent is a ghost at most."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


def _eager_proposal(sww):
    """A perceptron that proposes every patch with a neighbour whose coefficients reach a third of
    a threshold."""
    W1 = np.zeros((sww.MLP_FEATURES, sww.MLP_HIDDEN))
    w2 = np.zeros(sww.MLP_HIDDEN)
    W1[4, 0] = W1[5, 1] = 1.0
    w2[:2] = 4.0
    return np.concatenate([W1.ravel(), np.zeros(sww.MLP_HIDDEN), w2, [-1.6]]).astype(np.float32)


@pytest.mark.parametrize("nu", [0.0, 2.0e5])
@pytest.mark.parametrize("mask", ["lists", "dense"])
@pytest.mark.parametrize("patch,jmax", [(8, 6), (8, 7), (16, 7)])
def test_live_edge_has_a_live_end(patch, jmax, mask, nu):
    import paper_1404_0405_gb300 as sww
    m = sww.Model(3, jmax, patch=patch, eps=1e-2, precision="fp32", mask=mask, nu=nu)
    xyz, en = m.grid(jmax)
    m.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)))
    m.adapt()
    m.set_learned(2, _eager_proposal(sww), 0.5)
    ends = {j: m.grid(j)[1] for j in range(3, jmax + 1)}
    for _ in range(4):
        m.step(-1.0, 1, True)
        for j, e in ends.items():
            n, f = m.mask(j)
            orphans = ((f & 1) > 0) & ((n[e[:, 0]] | n[e[:, 1]]) & 1 == 0)
            assert not orphans.any(), f"level {j}: {orphans.sum()} live edges without a live end"
    assert m.learn_stats()["proposed"] > 20
