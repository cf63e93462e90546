"""Forced tiles: 128-wide tiles with 16 drain warps, in every precision and both plane storages, at the
edges of tiles, k-blocks and row passes, against those with 8 (the same products added in the same
order: P and the results are bit-identical), the tile a call reports asked for again, and the
combinations 16 drain warps are not built for."""
import pytest
import torch

import paper_2306_12616_gb300 as fo
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SAME = ("mu", "trace", "trace_raw", "trace_gamma", "trace_proj", "frob2", "n_gemm", "status")


def hamiltonian(n):
    return torch.from_numpy(synth.tight_binding((n + 3) // 4 * 4, 40 + n)[:n, :n].copy()).to(DEV)


@pytest.mark.parametrize("store", [1, 2])
@pytest.mark.parametrize("prec", ["bf16x3", "fp16x2", "bf16x1"])
@pytest.mark.parametrize("n", [1, 31, 64, 127, 128, 129, 160, 257, 500, 1000])
def test_sixteen_drain_warps_on_128_wide_tiles(solver, prec, n, store):
    h = hamiltonian(n)
    kw = dict(precision=prec, tile_n=128, tile_ctas=1, tile_store=store)
    got = [solver.density_matrix(h, n / 2, solver.params(100, 0.1, tile_drain=d, **kw)) for d in (8, 16)]
    (p, r), (q, s) = got
    assert s["tile_drain"] == 16 and s["tile_n"] == 128 and s["tile_store"] == store
    assert torch.equal(p, q)
    assert all(r[k] == s[k] for k in SAME)


def test_batch_with_graph(solver):
    hs = [hamiltonian(n) for n in (640, 383, 256, 130, 64, 5)]
    ne = [h.shape[0] / 2 for h in hs]
    kw = dict(precision="bf16x3", tile_n=128, tile_ctas=1, tile_store=1)
    ps, _ = solver.density_matrix_batched(hs, ne, solver.params(60, 0.1, tile_drain=8, **kw))
    for _ in range(2):
        qs, _ = solver.density_matrix_batched(hs, ne, solver.params(60, 0.1, tile_drain=16, flags=fo.FO_FLAG_GRAPH, **kw))
        assert all(torch.equal(p, q) for p, q in zip(ps, qs))


@pytest.mark.parametrize("n", [64, 300, 1000])
def test_the_reported_tile_can_be_asked_for(n):
    h = hamiltonian(n)
    s = fo.Solver(0)
    try:
        p, r = s.density_matrix(h, n / 2, s.params(100, 0.1, precision="bf16x3"))
        kw = {k: r[k] for k in ("tile_n", "tile_ctas", "tile_drain", "tile_store")}
        q, t = s.density_matrix(h, n / 2, s.params(100, 0.1, precision="bf16x3", **kw))
    finally:
        s.close()
    assert {k: t[k] for k in kw} == kw and torch.equal(p, q)


@pytest.mark.parametrize("kw", [dict(tile_n=0), dict(tile_n=128, tile_ctas=2), dict(tile_n=128, tile_persist=2),
                                dict(tile_n=128, chain=2)])
def test_other_requests_for_sixteen_are_refused(solver, kw):
    h = hamiltonian(64)
    with pytest.raises(fo.FermiError) as e:
        solver.density_matrix(h, 32.0, solver.params(60, 0.1, precision="bf16x3", tile_drain=16, **kw))
    assert e.value.status == fo.FO_ERR_ARG
