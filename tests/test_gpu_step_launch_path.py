"""Which path a step takes: alone and below the switch to a launch per phase it is a cooperative
launch (a handle that never uses it launches far more kernels), and with more live points than
the cooperative grid has threads, so that its lists' later items are met, both paths agree bit
for bit."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu

THREADS = 512 * 152      # of a cooperative launch: one block of 512 an SM
SWITCH = 1 << 17         # live nodes from which an FP32 step is a launch per phase


@pytest.mark.parametrize("eps", [1e-2, 1e-3])
def test_cooperative_step_beyond_one_item_a_thread(eps):
    import paper_1404_0405_gb300 as sww
    outs, launches = [], []
    for persistent in (True, False):
        m = sww.Model(3, 7, patch=8, eps=eps, persistent=persistent, precision="fp32")
        xyz, en = m.grid(7)
        m.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)))
        m.adapt()
        points = sum(int((f & 1).sum()) for j in range(3, 8) for f in m.mask(j))
        assert points > THREADS and m.live_nodes() < SWITCH
        own = m.stats()["kernel_launches"]
        own = m.stats()["kernel_launches"] - own      # those of stats() itself
        before = m.stats()["kernel_launches"]
        m.step(-1.0, 3, True)
        launches.append(m.stats()["kernel_launches"] - before - own)
        assert m.live_nodes() < SWITCH
        outs.append([m.get(j, q) for j in range(3, 8) for q in (sww.NODE_FLAGS, sww.EDGE_FLAGS, sww.DH, sww.U)])
    # a stage of a launch per phase: ghosts, two of the trend, restriction and divergence, update
    assert launches[1] - launches[0] >= 3 * 4 * 6
    for x, y in zip(*outs):
        assert np.array_equal(x, y)
