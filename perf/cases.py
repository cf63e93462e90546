"""The solver's workloads, as calls of its public entry points, for timing and for comparing results.

Every case is a plain dict; its "kind" names the entry point and the Hamiltonian family:

* ``bounds``: spectral bounds of one dense Hamiltonian (``Solver.spectral_bounds``);
* ``density``: density matrices of one or several Hamiltonians in one call (``density_matrix``,
  ``density_matrix_batched``, or with ``host`` the host-buffer entry point);
* ``batch``: many Hamiltonians of different sizes in one call, replayed as a CUDA graph;
* ``features``: training pairs of the learned chemical potential (``learned_features``);
* ``train``: training of its network on such pairs (``mlp_init``, ``mlp_train``, ``mlp_get_params``).

The Hamiltonians are the families the solver is documented on (random symmetric, tight-binding,
metallic), drawn on the GPU from the seed alone. One solver per process, as a program that
computes density matrices keeps it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_12616_gb300 import FO_FLAG_GRAPH, FO_MLP_PARAMS, Solver

DEV = "cuda:0"
ONSITE_EV = (-10.0, -5.0, -5.0, -5.0)
METALLIC_FILL = (0.74, 0.81)
HIDDEN, INPUTS, OUTPUTS, MOMENTS = 256, 68, 2, 64
BATCH_KT = (0.05, 0.2)


def listed() -> list[dict]:
    return [
        # the smallest call: an enclosure of the spectrum of a small matrix, launch latency only
        {"name": "bounds_n256", "kind": "bounds", "family": "tb", "n": 256},
        # plain float64, one small random Hamiltonian (kT given as a share of the width)
        {"name": "fp64_random_n256", "kind": "density", "family": "random", "sizes": "256", "terms": 256,
         "kt": 0.05, "precision": "fp64", "lanczos": 0, "host": False},
        # plain float64 at the sizes of a dense electronic-structure step
        {"name": "fp64_tb_n1000", "kind": "density", "family": "tb", "sizes": "1000", "terms": 400, "kt": 0.1,
         "precision": "fp64", "lanczos": 0, "host": False},
        {"name": "fp64_tb_n2000", "kind": "density", "family": "tb", "sizes": "2000", "terms": 400, "kt": 0.1,
         "precision": "fp64", "lanczos": 0, "host": False},
        # split precision, the smallest molecule: a chain of tiny products, latency and launches
        {"name": "bf16x3_tb_n64", "kind": "density", "family": "tb", "sizes": "64", "terms": 300, "kt": 0.1,
         "precision": "bf16x3", "lanczos": 0, "host": False},
        # one self-consistent-field step of a mid-sized system
        {"name": "bf16x3_tb_n1000", "kind": "density", "family": "tb", "sizes": "1000", "terms": 400, "kt": 0.1,
         "precision": "bf16x3", "lanczos": 0, "host": False},
        # the headline workload: three sizes in one call
        {"name": "bf16x3_tb_1k_2k_5k", "kind": "density", "family": "tb", "sizes": "1000,2000,5000", "terms": 400,
         "kt": 0.1, "precision": "bf16x3", "lanczos": 0, "host": False},
        # an odd size, two-plane float16, tight (Lanczos) bounds
        {"name": "fp16x2_lanczos_n1501", "kind": "density", "family": "tb", "sizes": "1501", "terms": 400, "kt": 0.1,
         "precision": "fp16x2", "lanczos": 40, "host": False},
        # H in pinned host memory, P back to the host
        {"name": "bf16x3_host_n2000", "kind": "density", "family": "tb", "sizes": "2000", "terms": 400, "kt": 0.1,
         "precision": "bf16x3", "lanczos": 0, "host": True},
        # replicas of a molecular-dynamics run: 512 uneven sizes, one graph replay per call
        {"name": "bf16x3_batch512", "kind": "batch", "family": "tb", "count": 512, "lo": 64, "hi": 1024,
         "sizes_seed": 4000, "terms": 300, "precision": "bf16x3"},
        # training pairs of the learned chemical potential: 64 metallic systems, 1000 terms
        {"name": "features_metallic_64", "kind": "features", "family": "metallic", "count": 64, "n": 1024,
         "terms": 1000, "kt": 0.01, "precision": "bf16x3"},
        # the network trained on 20000 pairs (two of its epochs)
        {"name": "mlp_train_20k", "kind": "train", "rows": 20000, "epochs": 2, "batch": 256},
    ]


def _log_uniform(rng, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case of the same ranges."""
    kind = rng.choice(("bounds", "density64", "density", "density", "host", "batch", "features", "train"))
    if kind == "bounds":
        return {"kind": "bounds", "family": rng.choice(("tb", "random")), "n": _log_uniform(rng, 64, 6000)}
    if kind == "density64":
        family = rng.choice(("tb", "random"))
        return {"kind": "density", "family": family, "sizes": str(_log_uniform(rng, 64, 1900)),
                "terms": rng.randint(64, 400), "kt": rng.uniform(0.05, 0.2), "precision": "fp64",
                "lanczos": 0, "host": False}
    if kind in ("density", "host"):
        sizes = [_log_uniform(rng, 64, 3000) for _ in range(rng.choice((1, 1, 2, 3)))]
        return {"kind": "density", "family": "tb", "sizes": ",".join(str(n) for n in sizes),
                "terms": rng.randint(100, 500), "kt": rng.uniform(0.05, 0.2),
                "precision": rng.choice(("bf16x3", "bf16x3", "fp16x2")),
                "lanczos": rng.choice((0, 0, 40)), "host": kind == "host"}
    if kind == "batch":
        lo = _log_uniform(rng, 64, 256)
        return {"kind": "batch", "family": "tb", "count": rng.randint(8, 400), "lo": lo,
                "hi": _log_uniform(rng, 2 * lo, 1000), "sizes_seed": rng.randint(1, 1 << 20),
                "terms": rng.randint(100, 400), "precision": "bf16x3"}
    if kind == "features":
        return {"kind": "features", "family": "metallic", "count": rng.randint(4, 48), "n": rng.randint(200, 1000),
                "terms": rng.randint(300, 1000), "kt": rng.uniform(0.01, 0.05), "precision": "bf16x3"}
    return {"kind": "train", "rows": _log_uniform(rng, 500, 19000), "epochs": rng.randint(1, 2),
            "batch": rng.choice((32, 64, 100, 128, 256, 512))}


# ------------------------------------------------------------------ inputs

def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _tight_binding(n: int, g: torch.Generator, metallic: bool = False) -> torch.Tensor:
    """ceil(n/4) atoms at 0.1 per cubic angstrom in a periodic cube, four orbitals each, hopping
    -2 exp(-r / 1.5) times a random sign per orbital pair, cut at 6; the first n orbitals."""
    f64 = dict(device=DEV, dtype=torch.float64)
    na = (n + 3) // 4
    box = (na / 0.1) ** (1.0 / 3.0)
    pos = torch.rand((na, 3), generator=g, **f64) * box
    d = pos[:, None, :] - pos[None, :, :]
    d = d - box * torch.round(d / box)
    r = (d * d).sum(-1).sqrt()
    hop = torch.where(r < 6.0, -2.0 * torch.exp(-r / 1.5), torch.zeros((), **f64))
    hop.fill_diagonal_(0.0)
    h = hop.repeat_interleave(4, 0).repeat_interleave(4, 1)
    sign = torch.randint(0, 2, (4 * na, 4 * na), generator=g, device=DEV).to(torch.float64) * 2.0 - 1.0
    sign = torch.triu(sign, 1)
    h = h * (sign + sign.T)
    diag = torch.tensor(ONSITE_EV, **f64).repeat(na) + 0.1 * torch.randn(4 * na, generator=g, **f64)
    if metallic:
        idx = torch.randperm(4 * na, generator=g, device=DEV)[:na]
        diag[idx] = 0.02 * torch.randn(na, generator=g, **f64)
    h.diagonal().copy_(diag)
    return h[:n, :n]


def _random(n: int, g: torch.Generator) -> torch.Tensor:
    a = torch.randn((n, n), generator=g, device=DEV, dtype=torch.float64)
    h = (a + a.T) / (2.0 * math.sqrt(n))
    h.diagonal().add_(torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0)
    return h


def _hamiltonian(family: str, n: int, g: torch.Generator) -> torch.Tensor:
    return _random(n, g) if family == "random" else _tight_binding(n, g, family == "metallic")


def _sizes(case: dict) -> list[int]:
    if case["kind"] == "batch":
        rng = np.random.default_rng(case["sizes_seed"])
        n = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["count"]))
        return [int(x) for x in np.clip(np.round(n), case["lo"], case["hi"])]
    if case["kind"] == "features":
        return [case["n"]] * case["count"]
    if case["kind"] == "bounds":
        return [case["n"]]
    return [int(x) for x in case["sizes"].split(",")]


def _inputs(case: dict, seed: int) -> dict:
    """Hamiltonians (views of one flat buffer), electron counts and temperatures."""
    sizes, g = _sizes(case), _gen(seed)
    flat = torch.empty(sum(n * n for n in sizes), dtype=torch.float64, device=DEV)
    hs, o = [], 0
    for n in sizes:
        h = flat[o:o + n * n].view(n, n)
        h.copy_(_hamiltonian(case["family"], n, g))
        hs.append(h)
        o += n * n
    rng = np.random.default_rng(seed)
    if case["kind"] == "features":
        n_e = [float(x) for x in rng.uniform(*METALLIC_FILL, len(sizes)) * case["n"]]
    else:
        n_e = [float(n // 2) for n in sizes]
    kts = None
    if case["kind"] == "batch":
        kts = [float(x) for x in rng.uniform(*BATCH_KT, len(sizes))]
    elif case["kind"] != "bounds":
        kt = case["kt"]
        if case["family"] == "random":   # a share of the width of the spectrum's enclosure
            lo, hi = _gershgorin(hs[0])
            kt *= hi - lo
        kts = [kt] * len(sizes)
    return {"hs": hs, "flat": flat, "n_e": n_e, "kt": kts}


def _pairs(case: dict, seed: int) -> tuple[torch.Tensor, torch.Tensor]:
    """Training pairs with the scales of method-generated ones: decaying moments, filling,
    temperature and bounds; targets a smooth function of them plus scatter."""
    g, rows = _gen(seed), case["rows"]
    f64 = dict(device=DEV, dtype=torch.float64)
    j = torch.arange(1, MOMENTS + 1, **f64)
    c = torch.randn((rows, 4), generator=g, **f64)
    m = torch.exp(-j / 12.0)[None, :] * (c[:, :1] * torch.cos(0.35 * j) + c[:, 1:2] * torch.sin(0.8 * j)
                                         + 0.2 * c[:, 2:3]) * 0.2
    fill = 0.74 + 0.07 * torch.rand((rows, 1), generator=g, **f64)
    ktx = 1e-4 + 1e-4 * torch.rand((rows, 1), generator=g, **f64)
    ea = -0.8 + 0.03 * torch.randn((rows, 1), generator=g, **f64)
    eb = 0.7 + 0.03 * torch.randn((rows, 1), generator=g, **f64)
    feat = torch.cat((m, fill, ktx, ea, eb), 1)
    mu_x = 0.3 * torch.tanh(3.0 * m[:, 0] - m[:, 3]) + (fill[:, 0] - 0.77) + 0.002 * c[:, 3]
    order = 0.9 + 0.05 * torch.tanh(2.0 * m[:, 1]) + 200.0 * (ktx[:, 0] - 1.5e-4)
    return feat.float().contiguous(), torch.stack((mu_x, order), 1).float().contiguous()


_SOLVER = None


def _solver() -> Solver:
    global _SOLVER
    if _SOLVER is None:
        _SOLVER = Solver(0)
    return _SOLVER


def prepare(case: dict, seed: int) -> dict:
    s = {"kind": case["kind"], "solver": _solver()}
    if case["kind"] == "train":
        s["feat"], s["target"] = _pairs(case, seed)
        s["epochs"], s["batch"], s["seed"] = case["epochs"], case["batch"], seed
        return s
    s.update(_inputs(case, seed))
    if case["kind"] == "bounds":
        return s
    s["params"] = Solver.params(case["terms"], s["kt"][0], precision=case["precision"], mu_mode="bisect",
                                lanczos_steps=case.get("lanczos", 0),
                                flags=FO_FLAG_GRAPH if case["kind"] == "batch" else 0)
    if case["kind"] == "features":
        return s
    s["host"] = case.get("host", False)
    if s["host"]:
        s["hs"] = [h.cpu().pin_memory() for h in s["hs"]]
        del s["flat"]
        s["p"] = torch.empty(sum(h.numel() for h in s["hs"]), dtype=torch.float64).pin_memory()
    else:
        s["p"] = torch.empty_like(s["flat"])
    outs, o = [], 0
    for h in s["hs"]:
        outs.append(s["p"][o:o + h.numel()].view(h.shape))
        o += h.numel()
    s["outs"] = outs
    return s


def run(s: dict):
    solver, kind = s["solver"], s["kind"]
    if kind == "bounds":
        return solver.spectral_bounds(s["hs"][0])
    if kind == "train":
        solver.mlp_init(s["seed"])
        losses = solver.mlp_train(s["feat"], s["target"], epochs=s["epochs"], batch=s["batch"], lr=1e-3,
                                  seed=s["seed"])
        weights, norm = solver.mlp_get_params()
        return {"losses": np.array(losses, dtype=np.float32), "weights": weights, "norm": norm}
    if kind == "features":
        feat, target, res = solver.learned_features(s["hs"], s["n_e"], s["params"], kT=s["kt"])
        return {"features": feat, "targets": target}
    if s["host"]:
        res = solver.density_matrix_batched_host(s["hs"], s["n_e"], s["params"], s["outs"], kT=s["kt"])
    elif len(s["hs"]) == 1:
        _, r = solver.density_matrix(s["hs"][0], s["n_e"][0], s["params"], out=s["outs"][0])
        res = [r]
    else:
        _, res = solver.density_matrix_batched(s["hs"], s["n_e"], s["params"], kT=s["kt"], outs=s["outs"])
    return {"P": s["p"], "mu": np.array([r["mu"] for r in res]), "trace": np.array([r["trace"] for r in res])}


# ------------------------------------------------------------------ what a pass cannot do without

def _products(terms: int) -> int:
    """Matrix products of one density matrix: baby, giant and Clenshaw steps."""
    k = math.ceil(math.sqrt(terms))
    m = -(-terms // k)
    return (k - 1) + max(0, m - 2) + max(0, m - 1)


def work(case: dict) -> dict:
    if case["kind"] == "train":
        rows, steps = case["rows"] * case["epochs"], -(-case["rows"] // case["batch"]) * case["epochs"]
        return {"bytes": case["rows"] * 4.0 * (INPUTS + OUTPUTS) + 4.0 * 2 * FO_MLP_PARAMS,
                "flops": 6.0 * FO_MLP_PARAMS * rows + 12.0 * FO_MLP_PARAMS * steps}
    sizes = _sizes(case)
    area = float(sum(n * n for n in sizes))
    if case["kind"] == "bounds":
        return {"bytes": 8.0 * area + 24.0, "flops": area}
    split = {"fp64": 1, "bf16x3": 6, "fp16x2": 3}[case["precision"]]
    terms = case["terms"]
    volume = float(sum(n * n * (n + 1.0) for n in sizes))   # a symmetric product, upper triangle
    if case["kind"] == "features":
        k = math.ceil(math.sqrt(terms))
        products = (k - 1) + max(0, -(-terms // k) - 2)
        return {"bytes": 8.0 * area + 4.0 * len(sizes) * (INPUTS + OUTPUTS), "flops": split * products * volume}
    return {"bytes": 16.0 * area, "flops": split * _products(terms) * volume}


# ------------------------------------------------------------------ the same in 64 bits

def _gershgorin(h: torch.Tensor) -> tuple[float, float]:
    d = h.diagonal()
    r = h.abs().sum(1) - d.abs()
    return float((d - r).min()), float((d + r).max())


def _splitmix(seed: int, count: int) -> np.ndarray:
    """The first `count` outputs of splitmix64 started at `seed`."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _unit(z: np.ndarray) -> np.ndarray:
    return (z >> np.uint64(11)).astype(np.float64) * (1.0 / 9007199254740992.0)


def _lanczos(h: torch.Tensor, steps: int) -> tuple[float, float]:
    """Extreme Ritz values of `steps` Lanczos steps, widened by their residuals and 1 % of the
    width, inside the Gershgorin interval."""
    n = h.shape[0]
    q = torch.from_numpy(_unit(_splitmix(0x4C414E43, n)) - 0.5).to(h.device)
    q = q / q.norm()
    qp, alpha, beta = torch.zeros_like(q), [], [0.0]
    for j in range(min(steps, n)):
        w = h @ q - beta[j] * qp
        a = float(w @ q)
        w = w - a * q
        b = float(w.norm())
        alpha.append(a)
        beta.append(b)
        if not b > 1e-12 * (abs(a) + beta[j]):
            break
        qp, q = q, w / b
    k = len(alpha)
    t = np.diag(alpha) + np.diag(beta[1:k], 1) + np.diag(beta[1:k], -1)
    ev, vec = np.linalg.eigh(t)
    width = ev[-1] - ev[0]
    lo = ev[0] - beta[k] * abs(vec[-1, 0]) - 0.01 * width
    hi = ev[-1] + beta[k] * abs(vec[-1, -1]) + 0.01 * width
    ga, gb = _gershgorin(h)
    return max(lo, ga), min(hi, gb)


def _expansion(x: torch.Tensor, ea: float, eb: float, n_e: float, kt: float, terms: int):
    """(mu, coefficients, T_n(x)) of the Chebyshev interpolation of the Fermi function whose
    trace over the scaled eigenvalues x is n_e."""
    nodes = max(2048, 4 * terms)
    theta = math.pi * (torch.arange(nodes, dtype=torch.float64, device=x.device) + 0.5) / nodes
    e = 0.5 * (ea + eb) + 0.5 * (eb - ea) * torch.cos(theta)
    num = torch.arange(terms, dtype=torch.float64, device=x.device)
    dct = torch.cos(num[:, None] * theta[None, :]) * (2.0 / nodes)
    dct[0] *= 0.5
    cheb = torch.cos(num[None, :] * torch.arccos(x.clamp(-1.0, 1.0))[:, None])
    e_h, w_h = e.cpu().numpy(), (cheb.sum(0) @ dct).cpu().numpy()

    def fermi(mu):
        return 0.5 - 0.5 * np.tanh((e_h - mu) / (2.0 * kt))

    lo, hi = ea - 80.0 * kt, eb + 80.0 * kt
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if mid <= lo or mid >= hi:
            break
        if float(w_h @ fermi(mid)) < n_e:
            lo = mid
        else:
            hi = mid
    mu = 0.5 * (lo + hi)
    return mu, dct @ torch.from_numpy(fermi(mu)).to(x.device), cheb


def _exact_density(case: dict, seed: int):
    inp = _inputs(case, seed)
    out, mus, o = torch.empty_like(inp["flat"]), [], 0
    for h, n_e, kt in zip(inp["hs"], inp["n_e"], inp["kt"]):
        ea, eb = _lanczos(h, case["lanczos"]) if case.get("lanczos") else _gershgorin(h)
        lam, u = torch.linalg.eigh(h)
        mu, c, cheb = _expansion((2.0 * lam - (ea + eb)) / (eb - ea), ea, eb, n_e, kt, case["terms"])
        n = h.shape[0]
        out[o:o + n * n].view(n, n).copy_((u * (cheb @ c)) @ u.T)
        mus.append(mu)
        o += n * n
    return {"P": out.cpu() if case.get("host") else out, "mu": np.array(mus), "trace": np.array(inp["n_e"])}


def _exact_features(case: dict, seed: int):
    inp = _inputs(case, seed)
    k, terms = math.ceil(math.sqrt(case["terms"])), case["terms"]
    feat, target = [], []
    for h, n_e, kt in zip(inp["hs"], inp["n_e"], inp["kt"]):
        ea, eb = _gershgorin(h)
        n = h.shape[0]
        lam = torch.linalg.eigvalsh(h)
        mu, c, cheb = _expansion((2.0 * lam - (ea + eb)) / (eb - ea), ea, eb, n_e, kt, terms)
        tau = (cheb.sum(0) / n).cpu().numpy()
        row = [float(tau[j]) if j <= min(2 * k, terms - 1) else 0.0 for j in range(1, MOMENTS + 1)]
        feat.append(row + [n_e / n, 2.0 * kt / (eb - ea), ea / 100.0, eb / 100.0])
        tail, length, ch = 0.0, terms, c.abs().cpu().numpy()
        for j in range(terms - 1, 0, -1):
            tail += ch[j]
            if tail > 2.5e-7:
                break
            length = j
        target.append([(2.0 * mu - (ea + eb)) / (eb - ea), math.log2(max(length, 1)) / math.log2(terms)])
    return {"features": torch.tensor(feat, dtype=torch.float64, device=DEV),
            "targets": torch.tensor(target, dtype=torch.float64, device=DEV)}


def _exact_train(case: dict, seed: int):
    feat, target = (v.double() for v in _pairs(case, seed))
    rows, batch = case["rows"], min(case["batch"], case["rows"])
    shapes = ((HIDDEN, INPUTS), (HIDDEN,), (HIDDEN, HIDDEN), (HIDDEN,), (OUTPUTS, HIDDEN), (OUTPUTS,))
    drawn = _unit(_splitmix(seed, sum(s[0] * s[1] for s in shapes if len(s) == 2)))
    prm, o = [], 0
    for s in shapes:
        if len(s) == 2:
            a = math.sqrt(6.0 / (s[0] + s[1]))
            w = ((2.0 * drawn[o:o + s[0] * s[1]] - 1.0) * a).astype(np.float32).reshape(s)
            o += s[0] * s[1]
        else:
            w = np.zeros(s, dtype=np.float32)
        prm.append(torch.from_numpy(w).to(DEV).double().requires_grad_(True))
    stats = []
    for v in (feat, target):
        mean = v.mean(0)
        stats.append((mean, torch.maximum(v.var(0, correction=0).sqrt(), 1e-6 * mean.abs().clamp(min=1.0))))
    x = (feat - stats[0][0]) / stats[0][1]
    t = (target - stats[1][0]) / stats[1][1]
    weight = torch.tensor([1.0, 0.1], dtype=torch.float64, device=DEV)
    mom = [(torch.zeros_like(p), torch.zeros_like(p)) for p in prm]
    picks = _splitmix(seed ^ 0x5DEECE66D, (rows - 1) * case["epochs"])
    losses, step, at = [], 0, 0
    for _ in range(case["epochs"]):
        perm = np.arange(rows)
        for q in range(rows - 1, 0, -1):
            r = int(picks[at] % np.uint64(q + 1))
            at += 1
            perm[q], perm[r] = perm[r], perm[q]
        order, mean_loss = torch.from_numpy(perm).to(DEV), []
        for b in range(0, rows, batch):
            idx = order[b:b + batch]
            z1 = x[idx] @ prm[0].T + prm[1]
            z2 = torch.nn.functional.silu(z1) @ prm[2].T + prm[3]
            y = torch.nn.functional.silu(z2) @ prm[4].T + prm[5]
            loss = ((y - t[idx]).square() * weight).sum() / len(idx)
            grads = torch.autograd.grad(loss, prm)
            mean_loss.append(loss.detach())
            step += 1
            with torch.no_grad():
                for p, gr, (m, v) in zip(prm, grads, mom):
                    m.mul_(0.9).add_(gr, alpha=0.1)
                    v.mul_(0.999).addcmul_(gr, gr, value=0.001)
                    p -= 1e-3 * (m / (1.0 - 0.9 ** step)) / ((v / (1.0 - 0.999 ** step)).sqrt() + 1e-8)
        losses.append(float(torch.stack(mean_loss).mean()))
    norm = torch.cat((stats[0][0], stats[0][1], stats[1][0], stats[1][1]))
    return {"losses": np.array(losses), "weights": torch.cat([p.detach().reshape(-1) for p in prm]).cpu(),
            "norm": norm.cpu()}


def exact(case: dict, seed: int):
    if case["kind"] == "bounds":
        lo, hi = _gershgorin(_inputs(case, seed)["hs"][0])
        return torch.tensor([lo, hi, 0.0], dtype=torch.float64, device=DEV)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "features":
        return _exact_features(case, seed)
    return _exact_density(case, seed)
