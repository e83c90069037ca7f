"""Reads and writes of an FP32 handle whose state came from sww_load take no device memory (they
cannot run out of it), and give what the saved handle gives."""
import numpy as np
import pytest

import workloads
from lib_mapping import lib_edge_geometry

pytestmark = pytest.mark.gpu


def test_reads_take_no_device_memory(tmp_path):
    import torch
    import paper_1404_0405_gb300 as sww
    a = sww.Model(3, 7, patch=8, eps=1e-2, precision="fp32")
    xyz, en = a.grid(7)
    a.set_state(*workloads.Workload("jet", seed=3).fields(xyz, *lib_edge_geometry(xyz, en)))
    a.adapt()
    a.step(-1.0, 1, True)
    a.save(str(tmp_path / "state"))
    b = sww.Model(3, 7, patch=8, eps=1e-2, precision="fp32", share=a)
    b.load(str(tmp_path / "state"))

    def use(m):
        m.forward()
        c = [m.coeffs(j) for j in range(4, 8)]
        out = [*m.get_state(7), *m.get_state(5), m.get(7, sww.DH), m.get(3, sww.U)]
        for j, x in zip(range(4, 8), c):
            m.set_coeffs(j, *x)
        m.set_level(7, out[4], m.get(7, sww.U))
        return out + [m.get(7, sww.DH), m.get(7, sww.U)]

    want = use(a)   # every kernel of these calls is loaded now
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    got = use(b)
    assert torch.cuda.mem_get_info()[0] == free
    for x, y in zip(want, got):
        assert np.array_equal(x, y)
