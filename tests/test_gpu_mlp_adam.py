"""The second Adam step, bit for bit: m = fma(b1, m, (1 - b1) g) and v = fma(b2, v, ((1 - b2) g) g) in
float32, from the gradients of the same kernels at the parameters before and after the first step
(whose moments are zero, so that only the second shows which product of a sum is rounded). Float32
sums, fused products, divisions and square roots are exact restatements; the bias corrections hold a
powf, which may be some units in the last place off: one pair of them has to serve every parameter."""
import numpy as np
import pytest
import torch

import paper_2306_12616_gb300 as fo

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
F = np.float32


def fma(a, b, c):
    """Float32 fused multiply-add: the exact product and a float64 sum rounded to odd, then to float32."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    s = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(F)


def order(n, epochs, seed):
    """The rows of every epoch: Fisher-Yates on splitmix64."""
    x, out = (seed ^ 0x5DEECE66D) & (2 ** 64 - 1), []
    for _ in range(epochs):
        perm = list(range(n))
        for q in range(n - 1, 0, -1):
            x = (x + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
            z = x
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
            r = (z ^ (z >> 31)) % (q + 1)
            perm[q], perm[r] = perm[r], perm[q]
        out.append(perm)
    return out


@pytest.mark.parametrize("rows", [9, 300])
def test_second_step_bits(solver, rows):
    seed, lr = 11, 1e-3
    g = torch.Generator().manual_seed(rows)
    x, t = torch.randn(rows, 68, generator=g), torch.randn(rows, 2, generator=g)
    params = []
    for epochs in (0, 1, 2):
        solver.mlp_init(4)
        if epochs:
            solver.mlp_train(x.to(DEV), t.to(DEV), epochs, rows, lr, seed)
        p, norm = solver.mlp_get_params()
        params.append(p)
    nrm = torch.from_numpy(norm)
    xs, ts = (x - nrm[:68]) / nrm[68:136], (t - nrm[136:138]) / nrm[138:140]
    grads = []
    for p, perm in zip(params, order(rows, 2, seed)):
        solver.mlp_set_params(p)
        grads.append(solver.mlp_gradients(xs[perm].contiguous().to(DEV), ts[perm].contiguous().to(DEV))[0].cpu().numpy())
    b1, b2, one = F(0.9), F(0.999), F(1.0)
    m = v = np.zeros_like(grads[0])
    full = np.ones_like(m)
    for gr in grads:
        m = fma(b1 * full, m, (one - b1) * gr)
        v = fma(b2 * full, v, (one - b2) * gr * gr)

    def corrections(b):   # 1 - powf(b, 2), powf within four units in the last place
        near = F(float(b) ** 2)
        return [one - F(near + k * np.spacing(near)) for k in range(-4, 5)]

    best = fo.FO_MLP_PARAMS
    for c1 in corrections(b1):
        mh = m / c1
        for c2 in corrections(b2):
            p2 = params[1] - F(lr) * mh / (np.sqrt(v / c2) + F(1e-8))
            best = min(best, int((p2 != params[2]).sum()))
    assert best == 0
