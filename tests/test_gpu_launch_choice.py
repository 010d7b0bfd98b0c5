"""Which plans replay a graph and which launch their kernels directly, and that the results do not depend on it."""
import threading

import pytest

from gpu_common import pai  # noqa: F401

pytestmark = pytest.mark.gpu


def _volume(nx, ny, nt, nz):
    return dict(dim=3, nx=nx, ny=ny, nt=nt, nz=nz, dx=1.0, dy=1.0, dt=0.6, c=1.0, dz=1.0, oversampling=2.0, K=3.0)


# the line lies where a reconstruction and its adjoint take 0.22 ms together; they take 0.18, 0.15 and 0.7 ms here (the
# first has more samples and voxels than a 2-D slice of 0.23 ms)
@pytest.mark.parametrize("size,direct", [((128, 256, 256, 64), False), ((256, 256, 64, 64), False),
                                         ((256, 256, 512, 256), True)], ids=lambda v: str(v))
def test_direct_only_where_the_kernels_outlast_the_launches(pai, size, direct):
    g = _volume(*size)
    assert [pai.Plan(g).info["uses_graph"] for _ in range(2)] == [0 if direct else 1] * 2  # timed, then reused


def test_plans_that_are_not_timed_may_replay_graphs(pai, monkeypatch):
    monkeypatch.setenv("PAI_AUTOTUNE", "0")
    g = dict(dim=2, nx=2048, nt=4096, nz=2048, dx=1.0, dt=1.0, c=1.0, dz=1.0, oversampling=2.0, K=3.0)
    assert pai.Plan(g).info["uses_graph"] == 1


def test_same_bits_on_one_thread_and_on_changing_threads(pai):
    """Direct launches while calls stay on one thread, graph replays when they change threads (a gradient step)."""
    import torch
    plan = pai.Plan(_volume(128, 256, 256, 64))
    plan.set_deterministic(True)
    p = torch.randn((128, 256, 256), device="cuda")
    h = torch.randn((128, 256, 64), device="cuda")
    f, a = plan.reconstruct(p).clone(), plan.adjoint(h).clone()
    out, grad = torch.empty_like(f), torch.empty_like(a)
    for _ in range(5):
        out.zero_(), grad.zero_()
        torch.cuda.synchronize()
        plan.reconstruct(p, out=out)
        t = threading.Thread(target=plan.adjoint, args=(h, grad))
        t.start()
        t.join()
        assert torch.equal(out, f) and torch.equal(grad, a)
    x = p.clone().requires_grad_(True)
    for _ in range(5):
        (g,) = torch.autograd.grad(pai.PAIRecon.apply(x, plan), x, h)
        assert torch.equal(g, a)


def test_forward_models_never_replay_graphs(pai):
    model = pai.ForwardModel(dict(dim=2, nx=64, nt=128, nz=64, dx=1.0, dt=1.0, c=1.0, dz=1.0))
    assert model.info["uses_graph"] == 0
