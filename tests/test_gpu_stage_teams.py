"""The persistent stage with its teams of threads per patch against one launch per
phase, for every patch side (4: teams of 128 threads, 8: of 256, 16: of 512) and both
precisions, from grids with fewer patches than teams up, and for the viscous form, whose
patches all take the tabulated path.  The bodies and their order are the same, so the
inviscid results agree bit for bit; the compiler may contract the viscous terms
differently in the two kernels, so those are compared to rounding (1e-12 of the field's
maximum in FP64, 2e-6 in FP32)."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


def _run(persistent, precision, patch, jmin, jmax, nu):
    import paper_1404_0405_gb300 as sww
    m = sww.Model(jmin, jmax, patch=patch, eps=1e-2, persistent=persistent, precision=precision, nu=nu)
    xyz, en = m.grid(jmax)
    m.set_state(*workloads.Workload("jet", seed=9).fields(xyz, *lib_edge_geometry(xyz, en)))
    if jmax > jmin:
        m.adapt()
    m.step(-1.0, 2, jmax > jmin)
    return [(m.get(j, sww.NODE_FLAGS), m.get(j, sww.EDGE_FLAGS), m.get(j, sww.DH), m.get(j, sww.U))
            for j in range(jmin, jmax + 1)]


@pytest.mark.parametrize("nu", [0.0, 2.0e5])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("patch,jmin,jmax", [(4, 2, 2), (4, 3, 5), (8, 3, 6), (8, 5, 5), (16, 4, 6)])
def test_teams_match_phase_launches(patch, jmin, jmax, precision, nu):
    a = _run(True, precision, patch, jmin, jmax, nu)
    b = _run(False, precision, patch, jmin, jmax, nu)
    tol = 1e-12 if precision == "fp64" else 2e-6
    for (nf, ef, dh, u), (nf2, ef2, dh2, u2) in zip(a, b):
        if nu == 0.0:
            assert np.array_equal(nf, nf2) and np.array_equal(ef, ef2)
            assert np.array_equal(dh, dh2) and np.array_equal(u, u2)
        else:
            for x, y in ((dh, dh2), (u, u2)):
                assert np.abs(x - y).max() <= tol * np.abs(y).max()
