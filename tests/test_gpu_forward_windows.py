"""The forward model with every window: tap counts 4 to 24 and truncated sinc, by its own row kernel or by node pairs,
rows of up to 32 warps and rows that the own kernel does not fit.  Against the oracle the bound is the FP32 one plus
the window's predicted error; against the node pairs' list spread it is the FP32 one, whatever the window's error."""
import numpy as np
import pytest

import oracle
import phantoms as ph
from gpu_common import TOL, gdict, pai, rel, to_gpu, to_np  # noqa: F401

pytestmark = pytest.mark.gpu

GEOMS = {"2d": ph.Geometry(dim=2, nx=50, nt=128, nz=36, dt=0.7),
         "3d": ph.Geometry(dim=3, nx=12, ny=10, nt=40, nz=12, dt=0.6)}
_ref = {}


def _case(key):
    if key not in _ref:
        f = ph.random_image(33, GEOMS[key]).astype(np.float32)
        _ref[key] = f, oracle.forward_model(GEOMS[key], f.astype(np.float64))
    return (GEOMS[key], *_ref[key])


@pytest.mark.parametrize("H", range(2, 13))
@pytest.mark.parametrize("method", ["kb", "tsinc"])
@pytest.mark.parametrize("key", sorted(GEOMS))
def test_every_window(pai, key, method, H, monkeypatch):
    g, f, ref = _case(key)
    kw = gdict(g, method=method, K=H / 2.0, oversampling=2.0)
    model = pai.ForwardModel(kw)
    assert model.info["taps"] == 2 * H
    got = to_np(model(to_gpu(f)))
    assert rel(got, ref) < TOL + model.info["predicted_error"]
    monkeypatch.setenv("PAI_SPREAD", "tap")
    assert rel(got, to_np(pai.ForwardModel(kw)(to_gpu(f)))) < TOL


@pytest.mark.parametrize("K", [1.0, 3.0])
@pytest.mark.parametrize("kw,M", [(dict(dim=2, nx=4, nt=8000, nz=6, dt=0.01), 16384),
                                  (dict(dim=2, nx=6, nt=3000, nz=40, dt=0.02), 8192),
                                  (dict(dim=3, nx=4, ny=2, nt=8000, nz=4, dt=0.002, dx=4.0, dy=4.0), 16384)],
                         ids=["2d-32warps", "2d-16warps", "3d-too-long-for-row-pairs"])
def test_long_rows(pai, kw, M, K):
    g = ph.Geometry(**kw)
    f = ph.random_image(34, g).astype(np.float32)
    model = pai.ForwardModel(gdict(g, K=K))
    assert model.info["M"] == M
    ref = oracle.forward_model(g, f.astype(np.float64))
    assert rel(to_np(model(to_gpu(f))), ref) < TOL + model.info["predicted_error"]


def test_node_pairs_repeat_bit_for_bit(pai):
    import torch
    g = GEOMS["3d"]
    model = pai.ForwardModel(gdict(g, method="tsinc", K=3))
    model.set_deterministic(True)
    f = to_gpu(ph.random_image(35, g))
    ref = model(f).clone()
    assert all(torch.equal(model(f), ref) for _ in range(20))
