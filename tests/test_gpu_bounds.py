"""Bounds of one matrix: one cluster launch up to 256 rows, two launches above. Both give, bit for bit,
the row sums rounded once and what the density solver finds for the same matrix, on any row stride, and
flag a non-finite entry in any row."""
import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [2, 7, 8, 9, 127, 255, 256, 257, 511, 512, 513, 520, 777])
def test_bounds_at_the_edges_of_the_one_launch_form(solver, n):
    h = synth.random_symmetric(n, 40 + n)
    big = torch.full((n, n + 5), float("nan"), dtype=torch.float64, device=DEV)
    big[:, :n] = torch.from_numpy(h).to(DEV)
    d = big[:, :n]
    b = solver.spectral_bounds(d).cpu().numpy()
    r = np.array([math.fsum(np.abs(np.delete(h[i], i))) for i in range(n)])
    assert b[0] == np.min(np.diag(h) - r) and b[1] == np.max(np.diag(h) + r) and b[2] == 0.0
    _, res = solver.density_matrix(d, n / 2, solver.params(4, 1.0, mu=0.0, precision="fp64", mu_mode="fixed"))
    assert res["emin"] == b[0] and res["emax"] == b[1]
    for row, col, bad in ((0, n - 1, math.nan), (n - 1, 0, math.inf), (n - 1, n - 1, -math.inf)):
        keep = d[row, col].item()
        d[row, col] = bad
        assert solver.spectral_bounds(d)[2].item() == 1.0
        d[row, col] = keep
