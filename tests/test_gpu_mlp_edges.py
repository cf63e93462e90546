"""The network's row kernel (clusters of eight rows) and gradient kernel (passes of 256 rows) at the
edges of their tiles, against the float64 oracle: one row, around eight rows and around 256 rows.

Tolerance: float32 sums of at most 300 terms in order, a few layers deep, 2e-4 of each tensor's largest
magnitude (300 x 2^-24 = 1.8e-5 per sum)."""
import numpy as np
import pytest
import torch

import oracle.mlp as M

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def setup(solver, seed):
    p = M.init_params(seed)
    rng = np.random.default_rng(seed + 100)
    for k in ("b1", "b2", "b3"):
        p[k] = rng.normal(scale=0.1, size=p[k].shape)
    p32 = M.unflatten(M.flatten(p).astype(np.float32).astype(np.float64))
    solver.mlp_set_params(M.flatten(p32).astype(np.float32))
    return p32


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 15, 255, 256, 257, 300])
def test_forward_and_gradients(solver, rows):
    p = setup(solver, rows)
    rng = np.random.default_rng(rows)
    x = rng.normal(size=(rows, M.N_IN)).astype(np.float32)
    t = rng.normal(size=(rows, M.N_OUT)).astype(np.float32)
    xd, td = torch.from_numpy(x).to(DEV), torch.from_numpy(t).to(DEV)
    y = solver.mlp_forward(xd).cpu().numpy()
    yref, _ = M.forward(p, x.astype(np.float64))
    assert y.shape == (rows, M.N_OUT)
    assert np.max(np.abs(y - yref)) <= 2e-4 * max(1.0, np.max(np.abs(yref)))
    g, loss = solver.mlp_gradients(xd, td)
    L, gref = M.gradients(p, x.astype(np.float64), t.astype(np.float64), [1.0, 0.1])
    assert loss == pytest.approx(L, rel=1e-4)
    g = M.unflatten(g.cpu().numpy().astype(np.float64))
    for k in gref:
        assert np.max(np.abs(g[k] - gref[k])) <= 2e-4 * max(np.max(np.abs(gref[k])), 1e-3), k
