"""Which launches of an adaptive step the tracing hook counts under which kernel class, for a
handle alone: a launch per level of the ghosts, the restriction, its divergence, the partial
transform and the inverse transform (two: even nodes and edges, odd nodes), with the four
stages as one launch each or as their phases."""
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("persistent", [True, False])
def test_launches_by_class(persistent, precision):
    import paper_1404_0405_gb300 as sww
    jmin, jmax = 3, 6
    m = sww.Model(jmin, jmax, patch=8, eps=1e-2, precision=precision, persistent=persistent)
    xyz, en = m.grid(jmax)
    m.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)))
    m.adapt()
    top = max(j for j, n in m.stats()["active_patches"].items() if n > 0)
    m.profile(sww.KERNEL_CLASSES)
    m.step(-1.0, 1, True)
    n = {k: v[1] for k, v in m.profile_read().items()}
    m.profile([])
    down, up = top - jmin, min(top + 1, jmax) - jmin   # levels of a stage and of the inverse transform
    phased = 0 if persistent else 4
    assert down > 0
    assert n["stage"] == 4 - phased
    assert n["restrict"] == n["node"] == phased * down
    assert n["fill"] == phased * down + down + up
    assert n["partial"] == down and n["inverse"] == 2 * up
    assert n["coeff"] == 1 and n["mask"] > 10 and n["dt"] == 2
    assert n["update"] == phased and n["trend"] == phased
