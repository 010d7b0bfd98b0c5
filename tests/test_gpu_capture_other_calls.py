"""Calls under a caller's stream capture beside reconstruct, adjoint and forward model: host-memory calls and stage
profiling wait for the device and are refused with the capture intact; spectrum and cutoff are captured."""
import pytest

import phantoms as ph
from gpu_common import gdict, pai  # noqa: F401

pytestmark = pytest.mark.gpu

G = ph.Geometry(dim=2, nx=64, nt=128, nz=64)


def _calls(plan):
    import torch
    p, f = torch.randn((G.nx, G.nt)).pin_memory(), torch.empty((G.nx, G.nz)).pin_memory()
    d_p, d_f = p.cuda(), torch.empty((G.nx, G.nz), device="cuda")
    return {"host": lambda: plan.reconstruct_host(p, f), "host_async": lambda: plan.reconstruct_host_async(p, f),
            "profile": lambda: plan.profile_stages(d_p, d_f, reps=1), "reconstruct": lambda: plan.reconstruct(d_p, d_f)}


@pytest.mark.parametrize("use_graph", ["0", "1"])
@pytest.mark.parametrize("warm", [0, 3])
@pytest.mark.parametrize("op", ["host", "host_async", "profile"])
def test_refused_with_the_capture_intact(pai, op, warm, use_graph, monkeypatch):
    import torch
    monkeypatch.setenv("PAI_USE_GRAPH", use_graph)
    plan = pai.Plan(gdict(G, K=3))
    calls = _calls(plan)
    for _ in range(warm):
        calls[op]()
    plan.host_wait()
    torch.cuda.synchronize()
    mark = torch.zeros(4, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mark += 1
        with pytest.raises(pai.PAIError) as e:
            calls[op]()
        assert e.value.status == 4
    graph.replay()
    torch.cuda.synchronize()
    assert mark.eq(1).all()
    calls[op]()
    plan.host_wait()
    calls["reconstruct"]()
    torch.cuda.synchronize()


def test_spectrum_and_cutoff_are_captured(pai):
    import torch
    plan = pai.Plan(gdict(G, K=3))
    plan.set_cutoff(9.0)
    p = torch.randn((G.nx, G.nt), device="cuda")
    ref, cut = plan.spectrum(p).clone(), plan.cutoff(p).clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out, c = plan.spectrum(p), plan.cutoff(p)
    torch.view_as_real(out).zero_()
    c.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref)) and torch.equal(c, cut)
