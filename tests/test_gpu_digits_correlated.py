"""Digit products of matrices with equal and repeated entries, whose digits are as far from independent
as they can be: every left-out digit pair of a sum then has the same sign and size.

Tolerance. The pairs of order 8 and above and the rounding of the operands' digits change an entry
of a product by at most (7 + 2 + 1) K 2^-64 of the scales' 2^(eA + eB) (seven pairs of order 8 with |d| <=
2^7, the higher orders below a seventh of them, 2^(e-64) per operand entry); eA, eB <= 1 for members
of an enclosed spectrum, so below 40 K 2^-64 = K 2^-58.7 per entry, sqrt(n) times that in
||.||_F/sqrt(n) for an all-equal error. A recurrence of k and m steps amplifies the errors of its
products by at most its length squared: (k + m)^2 (sqrt(n) 2^-53 + n sqrt(n) 2^-58.7)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2306_12616_gb300 as fo

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def matrix(kind, n):
    i = np.arange(n)
    if kind == "constant":
        return np.full((n, n), 0.7)
    if kind == "blocks":   # blocks of 16 equal entries, the k extent of one digit block
        b = np.random.default_rng(4).normal(size=((n + 15) // 16,) * 2)
        return np.kron((b + b.T) / 2, np.ones((16, 16)))[:n, :n].copy()
    if kind == "circulant":   # every row the same entries
        v = np.random.default_rng(5).normal(size=n)
        v = (v + v[(-i) % n]) / 2
        return v[(i[:, None] - i[None, :]) % n]
    s = np.where((i // 3) % 2 == 0, 1.0, -1.0)   # one magnitude, two signs
    return 1.0 / 3.0 * s[:, None] * s[None, :]


@pytest.mark.parametrize("n", [129, 1000])
@pytest.mark.parametrize("kind", ["constant", "blocks", "circulant", "signs"])
def test_correlated_digits(solver, kind, n):
    h = matrix(kind, n)
    assert np.array_equal(h, h.T)
    ea, eb = O.gershgorin_bounds(h)
    terms, kT, mu = 100, 0.03 * (eb - ea), 0.45 * ea + 0.55 * eb
    hd = torch.from_numpy(h).to(DEV)
    kw = dict(mu=mu, precision="fp64", mu_mode="fixed")
    p, r = solver.density_matrix(hd, n / 2, solver.params(terms, kT, **kw))
    q, s = solver.density_matrix(hd, n / 2, solver.params(terms, kT, flags=fo.FO_FLAG_FP64_FMA, **kw))
    c = O.chebyshev_coeffs(kT, mu, r["emin"], r["emax"], terms)
    ref = O.poly_eig(h, c, r["emin"], r["emax"])
    k, m = O.plan_km(terms)
    tol = (k + m) ** 2 * (math.sqrt(n) * 2.0 ** -53 + n * math.sqrt(n) * 2.0 ** -58.7)
    err = [float(np.linalg.norm(x.cpu().numpy() - ref)) / math.sqrt(n) for x in (p, q)]
    print(kind, n, err, tol)
    assert err[0] <= tol and float((p - q).norm()) / math.sqrt(n) <= 2.0 * tol
