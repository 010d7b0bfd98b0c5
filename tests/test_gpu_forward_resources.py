"""What a forward-model plan holds and asks for: nothing the size of its box, and nothing of cuFFT."""
import numpy as np
import pytest

import oracle
import phantoms as ph
from gpu_common import TOL, gdict, pai, rel, to_gpu, to_np  # noqa: F401

pytestmark = pytest.mark.gpu

G = [ph.Geometry(dim=2, nx=60, nt=130, nz=40), ph.Geometry(dim=3, nx=14, ny=10, nt=40, nz=12)]


@pytest.mark.parametrize("g", G, ids=["2d", "3d"])
def test_no_cufft_plan_is_made(pai, g, monkeypatch):
    monkeypatch.setenv("PAI_FAULT_CUFFT_PLAN", "0")  # the first cuFFT plan creation would fail
    model = pai.ForwardModel(gdict(g, K=3))
    f = ph.random_image(51, g).astype(np.float32)
    assert rel(to_np(model(to_gpu(f))), oracle.forward_model(g, f.astype(np.float64))) < TOL


@pytest.mark.parametrize("kw", [dict(dim=2, nx=512, nt=1024, nz=512), dict(dim=3, nx=32, ny=32, nt=128, nz=32)],
                         ids=["2d", "3d"])
def test_memory(pai, kw):
    """The spectra and little else; profiling takes an image and data, no boxes."""
    import torch
    g = ph.Geometry(**kw)
    model = pai.ForwardModel(gdict(g, K=3))
    bx, by, bz = model.box
    rows = bx * (by // 2 + 1) if g.dim == 3 else bx // 2 + 1
    layers = g.nx * (by // 2 + 1) * g.nz if g.dim == 3 else 0
    spectra = 8 * (rows * max(g.nt, g.nz) + max(rows * (bz // 2 + 2), layers))
    tables = 8 * rows + 16 * bz + 32 * g.nt + (1 << 20)  # and twiddles and work items
    assert spectra < model.info["workspace_bytes"] < spectra + tables
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    model.profile_stages(reps=1)
    assert torch.cuda.max_memory_allocated() - before <= 4 * g.nx * (g.ny if g.dim == 3 else 1) * (g.nt + g.nz) + 1024
