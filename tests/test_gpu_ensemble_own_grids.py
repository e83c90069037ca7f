"""The batched step (persistent = 3) of members that do not share a grid, the coarsest first:
bit for bit the members stepped alone."""
import numpy as np
import pytest

from test_gpu_ensemble import _fields, _snapshot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("jmaxes", [(3, 5), (4, 3, 6)])
def test_coarse_lead_matches_single_runs(jmaxes, precision):
    import paper_1404_0405_gb300 as sww
    ens, alone = [], []
    for seed, jmax in enumerate(jmaxes):
        for group in (ens, alone):
            m = sww.Model(2, jmax, patch=4, eps=3e-3, precision=precision, persistent="phased")
            m.set_state(*_fields(m, seed))
            m.adapt()
            group.append(m)
    sww.step_ensemble(ens, -1.0, 3, True)
    for m in alone:
        m.step(-1.0, 3, True)
    for a, b in zip(ens, alone):
        fa, sa = _snapshot(sww, a)
        fb, sb = _snapshot(sww, b)
        assert sa == sb
        for k in fa:
            assert np.array_equal(fa[k], fb[k]), k
