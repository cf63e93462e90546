"""Float64 calls without a matrix product (one term; one or two moments): no digits are formed, and the
results are those of the formulas: P = c_0 I exactly, tau_0 = n, tau_1 = tr X, tau_2 = 2 ||X||_F^2 - n
(sums of at most n^2 float64 terms: n 2^-53 relative to the sum of their magnitudes)."""
import numpy as np
import pytest
import torch

import paper_2306_12616_gb300 as fo
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [1, 130])
def test_one_term_forms_no_digits(solver, n):
    h = torch.from_numpy(synth.random_symmetric(n, 3)).to(DEV)
    kw = dict(mu=0.1, precision="fp64", mu_mode="fixed", bounds=(-5.0, 5.0))
    p, r = solver.density_matrix(h, n / 2, solver.params(1, 0.5, **kw))
    _, s = solver.density_matrix(h, n / 2, solver.params(1, 0.5, flags=fo.FO_FLAG_FP64_FMA, **kw))
    assert r["n_gemm"] == 0 and r["n_launches"] == s["n_launches"]
    c0 = float(solver.chebyshev_coeffs(0.5, 0.1, -5.0, 5.0, 1)[0])
    assert torch.equal(p, c0 * torch.eye(n, dtype=torch.float64, device=DEV))


@pytest.mark.parametrize("count", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 130, 500])
def test_first_moments(solver, n, count):
    h = synth.random_symmetric(n, 7)
    b = torch.tensor([-30.0, 31.0, 0.0], dtype=torch.float64, device=DEV)
    tau = solver.moments(torch.from_numpy(h).to(DEV), b, count).cpu().numpy()
    x = (2.0 * h - np.eye(n)) / 61.0
    ref = np.array([n, np.trace(x), 2.0 * (x * x).sum() - n])[:count]
    size = np.array([n, np.abs(np.diag(x)).sum(), 2.0 * (x * x).sum() + n])[:count]
    assert np.all(np.abs(tau - ref) <= 4.0 * max(n, 4) * 2.0 ** -53 * np.maximum(size, 1e-300))
