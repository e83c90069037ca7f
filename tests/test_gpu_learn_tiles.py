"""The perceptron's training and evaluation kernels at the edges of their tiles (64
samples a warp, a warp a tile, a block an SM) and with features that are not 16-byte
aligned, against the FP64 oracle (oracle/mlp.py).

Tolerance: a gradient entry is a sum of n FP32 products added in chains of at most 32
and then per warp, so its error is below 64 * 2^-24 of the sum of the terms'
magnitudes, 4e-6 of it; 1e-5 of the largest entry is asked, as for the other sizes."""
import numpy as np
import pytest

from oracle import mlp
from test_gpu_learn import _problem, _torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 31, 32, 33, 63, 64, 65, 127, 64 * 152, 64 * 152 + 1, 64 * 152 * 20 + 5])
def test_tile_edges_match_oracle(n, shift):
    import paper_1404_0405_gb300 as sww
    torch, dev = _torch()
    X, y, params = _problem(n, n + shift)
    buf = torch.empty(n * mlp.F + shift, device=dev)
    Xd = buf[shift:].view(n, mlp.F)   # shift 1: rows start 4 bytes past a 16-byte boundary
    Xd.copy_(torch.from_numpy(X))
    pd = torch.from_numpy(params).to(dev)
    work = torch.full((sww.MLP_WORK,), float("nan"), device=dev)
    out = torch.empty(sww.MLP_PARAMS + 1, device=dev)
    sww.mlp_loss_grad(Xd, torch.from_numpy(y).to(dev), pd, 2.5, work, out)
    got = out.cpu().numpy().astype(np.float64)
    W1, b1, w2, b2 = mlp.unpack(params)
    L, *grads = mlp.loss_grad(X, y, W1, b1, w2, b2, 2.5)
    want = mlp.flat(*grads)
    assert abs(got[-1] / L - 1) < 1e-5
    assert np.max(np.abs(got[:-1] - want)) < 1e-5 * max(np.max(np.abs(want)), 1e-3)
    p = torch.empty(n, device=dev)
    sww.mlp_predict(Xd, pd, p)
    assert np.max(np.abs(p.cpu().numpy() - mlp.predict(X, params))) < 1e-5
