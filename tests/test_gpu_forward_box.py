"""The forward model's transforms of a box that is never stored: image and detector extents that leave
remainders in the column tiles, buffers on a 4-byte boundary, and the cutoff applied in place."""
import ctypes

import numpy as np
import pytest

import oracle
import oracle.cutoff as oc
import phantoms as ph
from gpu_common import TOL, gdict, pai, rel, to_gpu, to_np  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [
    ph.Geometry(dim=2, nx=2, nt=8, nz=2), ph.Geometry(dim=2, nx=62, nt=34, nz=6),
    ph.Geometry(dim=2, nx=250, nt=258, nz=130, dt=0.5), ph.Geometry(dim=3, nx=2, ny=4, nt=10, nz=2),
    ph.Geometry(dim=3, nx=30, ny=14, nt=18, nz=34), ph.Geometry(dim=3, nx=10, ny=34, nt=60, nz=4, dt=0.6)],
    ids=lambda g: f"{g.dim}d-{g.nx}x{g.ny}x{g.nt}-{g.nz}")
def test_extents_and_alignment(pai, g):
    import torch
    model = pai.ForwardModel(gdict(g, K=3))
    img = ph.random_image(11, g).astype(np.float32)
    got = model(to_gpu(img))
    assert rel(to_np(got), oracle.forward_model(g, img.astype(np.float64))) < TOL
    # the same from and into buffers that start on a 4-byte boundary, bit for bit, nothing beside them written
    x = torch.zeros(img.size + 1, device="cuda")
    y = torch.full((got.numel() + 2,), 7.0, device="cuda")
    x[1:] = to_gpu(img).ravel()
    model.set_deterministic(True)
    ref = model(to_gpu(img))
    st = model._lib.pai_forward_model(model._h, ctypes.c_void_p(x.data_ptr() + 4), ctypes.c_void_p(y.data_ptr() + 4))
    assert st == 0
    assert torch.equal(y[1:-1], ref.ravel()) and y[0] == 7.0 and y[-1] == 7.0


@pytest.mark.parametrize("g", [ph.Geometry(dim=2, nx=40, nt=66, nz=24), ph.Geometry(dim=3, nx=16, ny=12, nt=20, nz=10)],
                         ids=["2d", "3d"])
def test_data_model_in_place(pai, g):
    img = ph.random_image(12, g).astype(np.float32)
    got = to_np(pai.ForwardModel(gdict(g, K=3), cutoff=9.0)(to_gpu(img)))
    ref = oc.apply(oracle.forward_model(g, img.astype(np.float64)), 9.0)
    assert rel(got, ref) < TOL
