"""The allocation-free bounds on both sides of the line below which the context entry point runs one
launch, and at sizes of several reduction passes: that entry point's bits, in a row on one stream without a
synchronisation between the calls (each overwrites the shared partial results)."""
import pytest
import torch

import paper_2306_12616_gb300 as fo

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_sizes_in_a_row(solver):
    g = torch.Generator(device=DEV).manual_seed(5)
    hs, outs = [], []
    for n in (1, 7, 255, 256, 257, 300, 2500, 129, 4100):
        h = torch.randn(n, n + 3, generator=g, device=DEV, dtype=torch.float64)[:, :n]
        h *= torch.exp(4.0 * torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64))
        if n == 300:
            h[17, 250] = float("inf")
        hs.append(h)
    stream = torch.cuda.current_stream().cuda_stream
    for h in hs:
        out = torch.full((3,), float("nan"), dtype=torch.float64, device=DEV)
        assert fo.fo_spectral_bounds_noalloc(h.data_ptr(), h.shape[0], h.stride(0), out.data_ptr(), stream) == fo.FO_OK
        outs.append(out)
    for h, out in zip(hs, outs):
        assert torch.equal(out, solver.spectral_bounds(h)), h.shape[0]
        assert float(out[2]) == (1.0 if h.shape[0] == 300 else 0.0)
