"""Calls under a caller's stream capture: refused with a status whether a plan replays graphs or launches its
kernels directly, with the capture and the plan intact; plans made with PAI_USE_GRAPH=0 are captured."""
import pytest

import phantoms as ph
from gpu_common import gdict, pai  # noqa: F401

pytestmark = pytest.mark.gpu

# a small plan (graphs), one on cuFFT, and one above the size from which kernels are launched directly
SHAPES = {"graphs": ph.Geometry(dim=2, nx=64, nt=128, nz=64), "cufft": ph.Geometry(dim=2, nx=60, nt=130, nz=62),
          "direct": ph.Geometry(dim=2, nx=2048, nt=4096, nz=2048)}


def _call(pai, op, g):
    import torch
    plan = pai.ForwardModel(gdict(g, K=3)) if op == "forward" else pai.Plan(gdict(g, K=3))
    plan.set_deterministic(True)
    n_in, n_out = (g.nt, g.nz) if op == "reconstruct" else (g.nz, g.nt)
    x = torch.randn((g.nx, n_in), device="cuda")
    out = torch.zeros((g.nx, n_out), device="cuda")
    fn = plan if op == "forward" else getattr(plan, op)
    return plan, x, out, lambda: fn(x, out)


@pytest.mark.parametrize("warm", [0, 3])
@pytest.mark.parametrize("op,shape", [("reconstruct", "graphs"), ("adjoint", "cufft"), ("reconstruct", "direct"),
                                      ("adjoint", "direct"), ("forward", "graphs")])
def test_refused(pai, op, shape, warm):
    import torch
    plan, x, out, call = _call(pai, op, SHAPES[shape])
    for _ in range(warm):
        call()
    torch.cuda.synchronize()
    out.zero_()
    mark = torch.zeros(4, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mark += 1
        with pytest.raises(pai.PAIError):
            call()
    graph.replay()
    torch.cuda.synchronize()
    assert mark.eq(1).all() and out.eq(0).all()
    ref = call().clone()
    assert ref.norm() > 0 and torch.equal(call(), ref)


def test_captured_without_graphs(pai, monkeypatch):
    import torch
    monkeypatch.setenv("PAI_USE_GRAPH", "0")
    plan, x, out, call = _call(pai, "reconstruct", SHAPES["graphs"])
    ref = call().clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
