"""The band-grid spread of the adjoint and of the forward model at the sizes where its parts meet: rows of part of
a warp to 32 warps, fewer nodes than warps, chunks with idle lanes, nodes crowding on one cell and coarse time steps
whose bands are longer than the grid."""
import numpy as np
import pytest

import oracle
import phantoms as ph
from gpu_common import TOL, gdict, pai, rel, to_gpu, to_np  # noqa: F401

pytestmark = pytest.mark.gpu

ADJOINT = [
    (dict(dim=2, nx=4, nt=8, nz=6), 32), (dict(dim=2, nx=4, nt=60, nz=34), 128),
    (dict(dim=2, nx=6, nt=120, nz=66, dt=0.8), 256), (dict(dim=2, nx=8, nt=200, nz=64, dt=3.9), 512),
    (dict(dim=2, nx=4, nt=500, nz=6), 1024), (dict(dim=2, nx=64, nt=512, nz=256, dx=0.2), 1024),
    (dict(dim=2, nx=4, nt=1000, nz=2), 2048), (dict(dim=2, nx=40, nt=1024, nz=1030, dx=0.3), 2048),
    (dict(dim=2, nx=12, nt=2000, nz=70, dt=2.2), 4096), (dict(dim=2, nx=4, nt=4000, nz=90), 8192),
    (dict(dim=3, nx=6, ny=4, nt=300, nz=130, dx=0.3, dy=0.4), 1024)]


@pytest.mark.parametrize("kw,M", ADJOINT, ids=lambda v: str(v) if isinstance(v, int) else f"{v['nx']}x{v['nt']}-{v['nz']}")
def test_adjoint_edges(pai, kw, M, monkeypatch):
    import torch
    monkeypatch.setenv("PAI_SPREAD", "pairs")
    g = ph.Geometry(**kw)
    plan = pai.Plan(gdict(g, K=3, oversampling=2))
    assert plan.info["M"] == M
    h = ph.random_image(21, g).astype(np.float32)
    a = plan.adjoint(to_gpu(h))
    assert rel(to_np(a), oracle.adjoint(g, h.astype(np.float64))) < TOL
    assert torch.equal(a, plan.adjoint(to_gpu(h)))


MODEL = [dict(dim=2, nx=8, nt=10, nz=4), dict(dim=2, nx=40, nt=250, nz=30, dt=0.3), dict(dim=2, nx=6, nt=2000, nz=8, dt=0.01),
         dict(dim=2, nx=20, nt=100, nz=16, dt=2.5), dict(dim=2, nx=30, nt=1000, nz=20, dx=0.5, dt=0.2),
         dict(dim=3, nx=4, ny=6, nt=12, nz=6), dict(dim=3, nx=10, ny=4, nt=500, nz=10, dt=0.03),
         dict(dim=3, nx=12, ny=8, nt=40, nz=12, dt=1.6, c=1.2)]


@pytest.mark.parametrize("kw", MODEL, ids=lambda v: f"{v['dim']}d-{v['nx']}x{v['nt']}-{v['nz']}")
def test_forward_model_edges(pai, kw):
    g = ph.Geometry(**kw)
    model = pai.ForwardModel(gdict(g, K=3))
    f = ph.random_image(22, g).astype(np.float32)
    assert rel(to_np(model(to_gpu(f))), oracle.forward_model(g, f.astype(np.float64))) < TOL


def test_window_left_open_on_a_tiny_problem(pai):
    """Few taps can ask for rows far longer than the nodes (M = 1024 for 3 nodes): warps without nodes."""
    g = ph.Geometry(dim=2, nx=4, nt=8, nz=6)
    h = ph.random_image(23, g).astype(np.float32)
    assert rel(to_np(pai.Plan(gdict(g)).adjoint(to_gpu(h))), oracle.adjoint(g, h.astype(np.float64))) < TOL


@pytest.mark.parametrize("kw", [dict(dim=2, nx=54, nt=66, nz=30), dict(dim=2, nx=64, nt=128, nz=64)], ids=["cufft", "own"])
def test_calls_from_fresh_threads_and_new_buffers(pai, kw):
    """A plan's first calls launch directly and repeated ones replay a graph: the same bits either way, on changing
    buffers and from a thread that has made no CUDA call before."""
    import threading

    import torch
    g = ph.Geometry(**kw)
    plan = pai.Plan(gdict(g, K=3))
    ps = [to_gpu(ph.random_data(30 + i, g)) for i in range(3)]
    outs = [torch.empty(g.image_shape, device="cuda") for _ in range(2)]
    ref = [plan.reconstruct(p).clone() for p in ps]
    for i in range(24):  # every pair of buffers four times
        assert torch.equal(plan.reconstruct(ps[i % 3], out=outs[i % 2]), ref[i % 3])
    h = to_gpu(ph.random_image(40, g))
    got = []
    t = threading.Thread(target=lambda: got.append(plan.adjoint(h).clone()))
    t.start()
    t.join()
    assert len(got) == 1 and torch.equal(got[0], plan.adjoint(h))


@pytest.mark.parametrize("kw", [dict(dim=2, nx=60, nt=2000, nz=200, dt=0.9), dict(dim=3, nx=12, ny=10, nt=500, nz=40, dt=0.2)],
                         ids=["2d", "3d"])
def test_forward_model_repeats_bit_for_bit(pai, kw):
    """Every cell belongs to one warp, also those a pass over two nodes touches beyond the last of them."""
    import torch
    g = ph.Geometry(**kw)
    model = pai.ForwardModel(gdict(g, K=3))
    f = to_gpu(ph.random_image(41, g))
    ref = model(f).clone()
    assert all(torch.equal(model(f), ref) for _ in range(20))
