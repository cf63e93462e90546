"""The split of the Frobenius products over blocks (csrc/gramsplit.h, compiled for the host): float32
plans keep blocks of 64 chunks; a float64 plan aims at about 300 blocks over its whole batch, not per
instance, since a block's final reduction costs as much as two chunks. On the GPU: the moments of
batches between the two ends of the rule against single calls (mu by bisection on them; both
sides' sums round at 2^-53 of tau's scale n, hence mu at |F| <= 1e-12 N_e over the density of states)."""
import math
import shutil
import subprocess

import pytest

import test_exactsum as T

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "gramsplit.h"
int main(int argc, char** argv) {
    std::vector<int64_t> np;
    for (int i = 2; i < argc; ++i) np.push_back(std::atoll(argv[i]));
    std::printf("%d\n", fo::gram_chunks(np.data(), (int)np.size(), argv[1][0] == '8'));
}
"""


def chunks(np):   # of 64 float64, on or above the diagonal
    return sum(r // 64 * -1 + np // 64 for r in range(np))


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("gram")
    (d / "g.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", T.CSRC, str(d / "g.cpp"), "-o", str(d / "g")], check=True)
    return lambda prec, sizes: int(subprocess.run([str(d / "g"), prec, *map(str, sizes)], check=True,
                                                  capture_output=True, text=True).stdout)


@pytest.mark.parametrize("sizes", [[128], [256], [384], [1024], [2048], [65536], [256] * 4, [256] * 16, [256] * 64,
                                   [128] * 512, [1024, 512, 256, 128], [2048] + [128] * 40])
def test_blocks_of_a_batch(rule, sizes):
    assert rule("4", sizes) == 64
    per = rule("8", sizes)
    assert 2 <= per <= 64
    total = sum(chunks(s) for s in sizes) if max(sizes) < 65536 else 64 * 1024 * 1025 // 2
    # the smallest blocks that leave about 300 of them, as far as the limits allow
    if per < 64:
        assert total / (per + 1) < 300
    if per > 2:
        assert total / per >= 300


@pytest.mark.gpu
@pytest.mark.parametrize("sizes", [[250] * 4, [256] * 12, [1000, 500, 130, 64, 20, 3], [100] * 70])
def test_float64_batch_moments(solver, sizes):
    import torch
    import synth
    hs = [torch.from_numpy(synth.random_symmetric(n, 11 + i)).to("cuda:0") for i, n in enumerate(sizes)]
    prm = solver.params(60, 0.3, precision="fp64", mu_mode="bisect")
    ps, rs = solver.density_matrix_batched(hs, [n / 2 for n in sizes], prm)
    for h, p, r, n in list(zip(hs, ps, rs, sizes))[:8]:
        q, s = solver.density_matrix(h, n / 2, prm)
        assert abs(r["mu"] - s["mu"]) <= 1e-9
        assert float((p - q).norm()) / math.sqrt(n) <= 1e-9
