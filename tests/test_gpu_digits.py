"""Float64 products on the tensor cores as exact products of 8-bit digits (csrc/gemm_digits.cu):
tile edges, k ranges, scales far from 1, infinities and NaN, batches, and the FMA kernel where the
digit buffers do not fit.

Tolerances. A product of the digits differs from the exact one by 2^-59 sqrt(K/1000) of the scale
bounds plus one float64 rounding, no more than a float64 sum; the recurrences of k and m steps
amplify a rounding at most by their lengths squared, so ||dP||_F/sqrt(n) <= (k + m)^2 sqrt(n) 2^-53
(2^-53 = 1.2e-16) bounds the Chebyshev form."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2306_12616_gb300 as fo
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def to_dev(h):
    return torch.from_numpy(h).to(DEV)


def bound(n, terms):
    k, m = O.plan_km(terms)
    return (k + m) ** 2 * math.sqrt(n) * 2.0 ** -53


@pytest.mark.parametrize("n,terms", [(1, 4), (2, 9), (15, 30), (16, 30), (17, 30), (31, 50), (127, 64), (128, 64),
                                     (129, 64), (257, 100), (383, 100), (640, 40)])
def test_edges(solver, n, terms):
    h = synth.random_symmetric(n, 31 + n)
    ea, eb = O.gershgorin_bounds(h)
    if n == 1:
        ea, eb = ea - 1.0, eb + 1.0
    kT, mu = 0.03 * (eb - ea), 0.3 * ea + 0.7 * eb
    p, r = solver.density_matrix(to_dev(h), n / 2, solver.params(terms, kT, mu=mu, precision="fp64",
                                                                 mu_mode="fixed"))
    c = O.chebyshev_coeffs(kT, mu, r["emin"], r["emax"], terms)
    ref = O.poly_eig(h, c, r["emin"], r["emax"])
    p = p.cpu().numpy()
    assert np.array_equal(p, p.T)
    assert np.linalg.norm(p - ref) / math.sqrt(n) <= bound(n, terms)


@pytest.mark.parametrize("shrink", [0.2, 0.6])
def test_bounds_inside_the_spectrum(solver, shrink):
    """Given bounds narrower than the spectrum: T_n grows like cosh(n arccosh x), the digits' scales
    follow it. Reference: the same polynomial from the eigenvalues; the rounding of either side is
    relative to sum_n |c_n| max |T_n|."""
    n, terms = 150, 16
    h = synth.tight_binding(152, 5)[:n, :n].copy()
    w, u = np.linalg.eigh(h)
    mid, half = 0.5 * (w[0] + w[-1]), 0.5 * (w[-1] - w[0]) * shrink
    ea, eb = mid - half, mid + half
    p, r = solver.density_matrix(to_dev(h), n / 2, solver.params(terms, 5.0, mu=mid, precision="fp64", mu_mode="fixed",
                                                                 bounds=(ea, eb)))
    # the call's own coefficients: their rounding (1e-17) times T_15 (1e14) would swamp the products'
    c = solver.chebyshev_coeffs(5.0, mid, ea, eb, terms).cpu().numpy()
    x = (w - mid) / half
    t = np.polynomial.chebyshev.chebvander(x, terms - 1)
    ref = (u * (t @ c)) @ u.T
    scale = float(np.abs(c) @ np.abs(t).max(0))
    assert np.abs(t).max() > 1e6   # the members do grow
    assert np.linalg.norm(p.cpu().numpy() - ref) / math.sqrt(n) <= 50.0 * bound(n, terms) * scale


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_entries_reach_p(solver, bad):
    n = 140
    h = synth.random_symmetric(n, 9)
    h[3, 70] = h[70, 3] = bad
    out = torch.zeros((n, n + 3), dtype=torch.float64, device=DEV)
    prm = solver.params(25, 0.1, mu=0.0, precision="fp64", mu_mode="fixed", bounds=(-4.0, 4.0))
    solver.density_matrix(to_dev(h), n / 2, prm, out=out[:, :n])
    assert not torch.isfinite(out[:, :n]).any()
    assert float(out[:, n:].abs().max()) == 0.0
    # the plan's buffers hold no trace of it afterwards
    h = synth.random_symmetric(n, 10)
    p, _ = solver.density_matrix(to_dev(h), n / 2, prm)
    c = O.chebyshev_coeffs(0.1, 0.0, -4.0, 4.0, 25)
    assert np.linalg.norm(p.cpu().numpy() - O.poly_eig(h, c, -4.0, 4.0)) / math.sqrt(n) <= bound(n, 25)


def test_batch_agrees_with_single_calls(solver):
    """Sums of digit products are exact whatever the split of k, which depends on the plan; only
    the scale of a result's digits is a bound that depends on it (by a power of two), which moves
    the last bits. 18 padded sizes are two launch groups."""
    ns = [40 + 128 * i for i in range(17, -1, -1)][8:] + [129, 260, 100, 17, 1]
    ns += [50 + 128 * i for i in range(10, 18)]
    hs = [to_dev(synth.random_symmetric(n, 60 + n)) for n in ns]
    prm = solver.params(9, 0.2, mu=0.1, precision="fp64", mu_mode="fixed")
    ps, _ = solver.density_matrix_batched(hs, [n / 2 for n in ns], prm)
    for h, p, n in zip(hs, ps, ns):
        q, _ = solver.density_matrix(h, n / 2, prm)
        assert float((p - q).norm()) / math.sqrt(n) <= 2.0 * bound(n, 9), n


def test_close_to_the_fma_kernel(solver):
    """Staged chains run the float64 FMA kernel: the same polynomial by another chain."""
    n, terms = 300, 64
    h = to_dev(synth.tight_binding(n, 12))
    kw = dict(mu=-6.0, precision="fp64", mu_mode="fixed")
    p, _ = solver.density_matrix(h, n / 2, solver.params(terms, 0.2, **kw))
    q, _ = solver.density_matrix(h, n / 2, solver.params(terms, 0.2, flags=fo.FO_FLAG_STAGED, **kw))
    assert float((p - q).norm()) / math.sqrt(n) <= 2.0 * bound(n, terms)


def test_fma_kernel_where_the_digit_buffers_do_not_fit():
    """N = 2000, 400 terms: 58 slots of 33.6 MB (1.95 GB) without the digit buffers, 2.2 GB with
    them; 2.07 GB are left free."""
    n = 2000
    h = to_dev(synth.tight_binding(n, 4))
    torch.cuda.empty_cache()
    s = fo.Solver(0)
    hog = None
    try:
        s.spectral_bounds(h)   # the library's own start-up allocations
        out = torch.empty((n, n), dtype=torch.float64, device=DEV)
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(free - int(2.07e9), dtype=torch.uint8, device=DEV)
        s.profile_enable(True)
        prm = s.params(400, 0.1, mu=-6.0, precision="fp64", mu_mode="bisect")
        p, r = s.density_matrix(h, n / 2, prm, out=out)
        assert s.profile_read()["products"]["launches"] == r["n_gemm"]
        del hog
        hog = None
        torch.cuda.empty_cache()
        s2 = fo.Solver(0)
        q, r2 = s2.density_matrix(h, n / 2, prm)
        s2.close()
        assert abs(r["mu"] - r2["mu"]) <= 1e-9 and float((p - q).norm()) / math.sqrt(n) <= bound(n, 400)
    finally:
        del hog
        s.close()
        torch.cuda.empty_cache()
