"""FO_FLAG_FP64_FMA: float64 products by FMAs, whose error is relative entry by entry, where the digit
products' is relative to the largest entries.

Two 4 x 4 fragments coupled by c: every term of an entry of T_n's coupling block has exactly one
odd number of factors c, so the block is c times a polynomial of order-one numbers, and each FMA
sum rounds relative to its own terms. Reference: the same polynomial (the library's c_n, given
bounds) in 60-digit decimals.

Tolerance. Entry-wise, one product of n terms rounds by at most (n + 2) 2^-53 of the sum of its terms'
magnitudes; the recurrences of k and m steps amplify a rounding at most by their lengths squared,
and the terms' magnitudes exceed the block's largest entry by at most 8 (a product of two 4-term
rows of entries below 1, twice). So the block's error is below 8 (k + m)^2 (n + 2) 2^-53 of its
largest entry: 8.9e-13 for n = 8 and 24 terms, which digit products miss by far from c = 1e-8 on."""
from decimal import Decimal, getcontext
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2306_12616_gb300 as fo

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TERMS, KT, MU, BOUNDS = 24, 0.3, 0.1, (-3.0, 3.0)


def fragments(c):
    rng = np.random.default_rng(17)
    h = np.zeros((8, 8))
    for o in (0, 4):
        a = rng.uniform(-0.5, 0.5, (4, 4))
        h[o:o + 4, o:o + 4] = a + a.T
    b = c * rng.uniform(0.25, 1.0, (4, 4)) * rng.choice([-1.0, 1.0], (4, 4))
    h[:4, 4:] = b
    h[4:, :4] = b.T
    return h


def reference(h, c, ea, eb):
    getcontext().prec = 60
    n, D = h.shape[0], Decimal
    w, s = D(eb) - D(ea), D(ea) + D(eb)
    x = [[(2 * D(float(h[i, j])) - (s if i == j else 0)) / w for j in range(n)] for i in range(n)]
    eye = [[D(int(i == j)) for j in range(n)] for i in range(n)]

    def mul(a, b):
        return [[sum((a[i][k] * b[k][j] for k in range(n)), D(0)) for j in range(n)] for i in range(n)]

    t0, t1 = eye, x
    p = [[D(float(c[0])) * t0[i][j] + D(float(c[1])) * t1[i][j] for j in range(n)] for i in range(n)]
    for q in range(2, len(c)):
        y = mul(x, t1)
        t0, t1 = t1, [[2 * y[i][j] - t0[i][j] for j in range(n)] for i in range(n)]
        p = [[p[i][j] + D(float(c[q])) * t1[i][j] for j in range(n)] for i in range(n)]
    return p


def call(solver, hs, flags):
    prm = solver.params(TERMS, KT, mu=MU, precision="fp64", mu_mode="fixed", bounds=BOUNDS, flags=flags)
    return solver.density_matrix_batched([torch.from_numpy(h).to(DEV) for h in hs], [4.0] * len(hs), prm)


@pytest.mark.parametrize("graph", [0, fo.FO_FLAG_GRAPH])
def test_weak_coupling_keeps_its_relative_accuracy(solver, graph):
    hs = [fragments(c) for c in (1e-4, 1e-8, 1e-12, 1e-16)]
    c = solver.chebyshev_coeffs(KT, MU, *BOUNDS, TERMS).cpu().numpy()
    k, m = O.plan_km(TERMS)
    tol = 8.0 * (k + m) ** 2 * 10 * 2.0 ** -53
    # a first call without the flag: its plan must not serve the call with it
    call(solver, hs, graph)
    for _ in range(2):
        ps, rs = call(solver, hs, graph | fo.FO_FLAG_FP64_FMA)
        for h, p in zip(hs, ps):
            ref, p = reference(h, c, *BOUNDS), p.cpu().numpy()
            big = max(abs(ref[i][j]) for i in range(4) for j in range(4, 8))
            err = max(abs(Decimal(float(p[i, j])) - ref[i][j]) for i in range(4) for j in range(4, 8))
            assert float(err / big) <= tol
            assert np.array_equal(p, p.T)


def test_default_is_as_accurate_norm_wise(solver):
    hs = [fragments(c) for c in (1e-4, 1e-8, 1e-12, 1e-16)]
    c = solver.chebyshev_coeffs(KT, MU, *BOUNDS, TERMS).cpu().numpy()
    k, m = O.plan_km(TERMS)
    ps, _ = call(solver, hs, 0)
    for h, p in zip(hs, ps):
        ref = np.array([[float(v) for v in row] for row in reference(h, c, *BOUNDS)])
        assert np.linalg.norm(p.cpu().numpy() - ref) <= (k + m) ** 2 * math.sqrt(8) * math.sqrt(8) * 2.0 ** -53


def test_searched_mu_and_features(solver):
    """The other calls that take the flag: mu by bisection and the learned model's training pairs."""
    import synth
    n, terms = 200, 64
    h = torch.from_numpy(synth.tight_binding(n, 3)).to(DEV)
    kw = dict(precision="fp64", mu_mode="bisect")
    p, r = solver.density_matrix(h, n / 2, solver.params(terms, 0.2, **kw))
    q, s = solver.density_matrix(h, n / 2, solver.params(terms, 0.2, flags=fo.FO_FLAG_FP64_FMA, **kw))
    assert s["n_gemm"] == r["n_gemm"] and s["n_launches"] < r["n_launches"]   # one launch per product
    assert abs(r["mu"] - s["mu"]) <= 1e-9
    assert float((p - q).norm()) / math.sqrt(n) <= 2.0 * (16 ** 2) * math.sqrt(n) * 2.0 ** -53 + 1e-9
    f, t, _ = solver.learned_features([h], [n / 2], solver.params(terms, 0.2, **kw))
    g, u, _ = solver.learned_features([h], [n / 2], solver.params(terms, 0.2, flags=fo.FO_FLAG_FP64_FMA, **kw))
    assert float((f - g).abs().max()) <= 1e-6 and float((t - u).abs().max()) <= 1e-6
