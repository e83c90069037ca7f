"""A whole step in one cooperative launch (time step, stages, partial transform,
coefficients) and the inverse transform in another, against one launch per phase: the
same bodies in the same order, so state, masks, step and time agree bit for bit, with the
CFL step and with a given one, adaptive and on a fixed mask, on one level and on several,
for both schemes, and with more items than threads (the lists' later items)."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


def _run(persistent, precision, jmin, jmax, dt, adapt, rk, eps):
    import paper_1404_0405_gb300 as sww
    m = sww.Model(jmin, jmax, patch=8, eps=eps, persistent=persistent, precision=precision, rk=rk)
    xyz, en = m.grid(jmax)
    m.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)))
    if jmax > jmin:
        m.adapt()
    m.step(dt, 3, adapt)
    st = m.stats()
    out = [st["t"], st["dt"], st["eps_h"], st["eps_u"]]
    for j in range(jmin, jmax + 1):
        out += [m.get(j, q) for q in (sww.NODE_FLAGS, sww.EDGE_FLAGS, sww.DH, sww.U)]
    m.close()
    return out


@pytest.mark.parametrize("dt", [-1.0, 20.0])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("jmin,jmax,adapt,rk,eps", [(3, 3, False, "rk4", 1e-2), (3, 6, True, "rk4", 1e-2),
                                                    (3, 6, False, "ssp43", 1e-2), (3, 7, True, "ssp43", 1e-4)])
def test_step_launch_matches_phase_launches(jmin, jmax, adapt, rk, eps, precision, dt):
    a = _run(True, precision, jmin, jmax, dt, adapt, rk, eps)
    b = _run(False, precision, jmin, jmax, dt, adapt, rk, eps)
    for x, y in zip(a, b):
        assert np.array_equal(x, y, equal_nan=True)
