"""Sizes past the registers and shared memory that the Lanczos update and the mu search hold: more than
2048 rows, more than 4096 quadrature nodes (4 per term; up to 1089 terms, k = 33), and the sizes around both lines.

Tolerances: Lanczos bounds 1e-8 of the width against the oracle's (both float64, different summation
orders); the oracle's trace at the mu found, 1e-8 N (see the test)."""
import numpy as np
import pytest
import torch

import oracle as O
import oracle.lanczos as L
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [2047, 2048, 2049, 2500])
def test_lanczos_bounds_past_the_rows_kept_in_registers(solver, n):
    h = np.ascontiguousarray(synth.tight_binding(2500, 900 + n)[:n, :n])   # (the generator wants multiples of 4)
    prm = solver.params(4, 0.1, precision="bf16x3", mu_mode="fixed", mu=0.0, lanczos_steps=24)
    _, r = solver.density_matrix(torch.from_numpy(h).to(DEV), 0.0, prm)
    lo, hi = L.lanczos_bounds(h, steps=24)
    assert abs(r["emin"] - lo) <= 1e-8 * (hi - lo) and abs(r["emax"] - hi) <= 1e-8 * (hi - lo)


@pytest.mark.parametrize("n_terms", [1023, 1024, 1025, 1089])
def test_mu_search_past_the_nodes_held_in_shared_memory(solver, n_terms):
    n, kT = 160, 0.05
    h = synth.tight_binding(n, 21)
    _, r = solver.density_matrix(torch.from_numpy(h).to(DEV), n / 2,
                                 solver.params(n_terms, kT, precision="fp64", mu_mode="bisect"))
    ga, gb = O.gershgorin_bounds(h)
    taus = O.moments_eig(O.spectrum_scaled(np.linalg.eigvalsh(h), ga, gb), n_terms)
    f = lambda mu: O.poly_trace(mu, taus, kT, ga, gb, n_terms) - n / 2
    # the trace at the found mu, to the search's own 1e-12 N_e plus the moments' rounding (1e-9 per
    # matrix row, as the float64 moments are compared elsewhere, times sum |c_n| < 10)
    assert r["status"] == 0 and abs(f(r["mu"])) <= 1e-8 * n
    assert abs(r["trace"] - n / 2) <= 1e-8
