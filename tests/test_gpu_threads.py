"""Plans of different sizes called from several threads at once, each on a stream of its own: their kernels are the same
functions with different amounts of shared memory."""
import threading

import pytest

from gpu_common import pai  # noqa: F401

pytestmark = pytest.mark.gpu


def _forward(pai, nt):
    return pai.ForwardModel(dict(dim=2, nx=16, nt=nt, nz=8, dx=1.0, dt=0.01, c=1.0, dz=1.0, oversampling=2.0, K=3.0)), (16, 8)


def _plan(pai, nt):
    return pai.Plan(dict(dim=2, nx=32, nt=nt, nz=64, dx=1.0, dt=1.0, c=1.0, dz=1.0, oversampling=2.0, K=3.0)), (32, nt)


@pytest.mark.parametrize("make", [_forward, _plan], ids=["forward", "eager"])
def test_threads_with_plans_of_their_own(pai, make, monkeypatch):
    import torch
    monkeypatch.setenv("PAI_USE_GRAPH", "0")  # (forward models launch directly whatever it says)
    work = []
    for nt in (8000, 4000, 2000):  # 136, 68 and 34 KB a row
        plan, shape = make(pai, nt)
        x = torch.randn(shape, device="cuda")
        ref = (plan if make is _forward else plan.reconstruct)(x).clone()
        work.append((plan, x, ref, torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []

    def run(plan, x, ref, stream):
        try:
            call = plan if make is _forward else plan.reconstruct
            with torch.cuda.stream(stream):
                out = torch.empty_like(ref)
                for _ in range(2000):
                    call(x, out)
                stream.synchronize()
                assert torch.equal(out, ref)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
