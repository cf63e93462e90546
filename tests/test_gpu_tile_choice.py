"""The tile the autotuner chooses (among them the 128-wide one with 16 drain warps, which only it can
choose) against a forced one: every configuration adds the same products in the same order, so
P and the results are bit-identical, at the edges of tiles, k-blocks and row passes."""
import numpy as np
import pytest
import torch

import paper_2306_12616_gb300 as fo
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("prec", ["bf16x3", "fp16x2", "bf16x1"])
@pytest.mark.parametrize("n", [4, 64, 128, 132, 500, 1000])
def test_chosen_tile_equals_forced(prec, n):
    h = torch.from_numpy(synth.tight_binding(n, 60 + n)).to(DEV)
    s = fo.Solver(0)   # a context of its own: the choice is made anew
    try:
        p, r = s.density_matrix(h, n / 2, s.params(100, 0.1, precision=prec))
        q, rq = s.density_matrix(h, n / 2, s.params(100, 0.1, precision=prec, tile_n=128, tile_ctas=1, tile_drain=8,
                                                    tile_store=1))
    finally:
        s.close()
    assert torch.equal(p, q)
    assert all(r[k] == rq[k] for k in ("mu", "trace", "trace_raw", "frob2", "n_gemm", "status"))
    assert (r["tile_n"], r["tile_ctas"], r["tile_drain"]) in {(256, 1, 8), (256, 1, 16), (128, 1, 8), (128, 2, 8),
                                                              (128, 1, 16)}
    print(prec, n, r["tile_n"], r["tile_ctas"], r["tile_drain"], r["tile_store"])
