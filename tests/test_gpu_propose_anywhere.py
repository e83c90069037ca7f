"""Proposals by sww_propose anywhere on the grid, most of them away from the active patches:
the candidate-list mask against the oracle's mask with the same extra nodes, bit for bit, and
the fields, on every patch side; and against the dense mask over steps of a state that was set
below Jmax (levels whose storage holds no earlier values)."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry
from test_gpu_learn import _patch_nodes
from test_gpu_parity import Pair

pytestmark = pytest.mark.gpu


def _proposals(m, rng):
    """A tenth of the inactive patches of every level that the next mask covers."""
    act = m.stats()["active_patches"]
    out = {}
    for j in range(m.jmin + 1, m.jmax + 1):
        if act[j - 1] == 0:
            continue
        n = m.sizes(j)[3]
        off = np.ones(n, bool)
        off[m.patches(j)] = False
        out[j] = np.append(off & (rng.random(n) < 0.1), False).astype(np.uint8)
    return out


@pytest.mark.parametrize("patch", [4, 8, 16])
def test_list_mask_matches_oracle(patch):
    P = Pair(3, 6, kind="jet", seed=3, patch=patch)
    P.adapt()
    rng = np.random.default_rng(2)
    for _ in range(2):
        sent = _proposals(P.lib, rng)
        assert any(f.any() for f in sent.values())
        for j, f in sent.items():
            P.lib.propose(j, f)
        P.ora.adapt(extra={j: P.maps[j].nodes_to_ora(_patch_nodes(P.lib, j, f).astype(np.uint8)) > 0
                           for j, f in sent.items()})
        P.lib.adapt()
        P.check_masks()
        P.check_fields()


@pytest.mark.parametrize("precision,nu", [("fp64", 0.0), ("fp32", 0.0), ("fp64", 2.0e5)])
@pytest.mark.parametrize("patch", [4, 8, 16])
def test_list_mask_matches_dense_mask(patch, precision, nu):
    import paper_1404_0405_gb300 as sww
    runs = []
    for mask in ("lists", "dense"):
        m = sww.Model(3, 6, patch=patch, eps=1e-2, precision=precision, mask=mask, nu=nu)
        xyz, en = m.grid(5)
        m.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)), level=5)
        m.adapt()
        runs.append(m)
    rng = np.random.default_rng(1)
    for _ in range(3):
        sent = _proposals(runs[0], rng)
        for m in runs:
            for j, f in sent.items():
                m.propose(j, f)
            m.step(-1.0, 1, True)
        for j in range(3, 7):
            (na, ea), (nb, eb) = (m.mask(j) for m in runs)
            assert np.array_equal(na & 7, nb & 7) and np.array_equal(ea & 7, eb & 7), j
            for q, f in ((sww.DH, na), (sww.U, ea)):
                x, y = (m.get(j, q)[(f & 3) > 0] for m in runs)
                assert np.array_equal(x, y), (j, q)
