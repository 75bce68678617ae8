"""Kernels whose tiles run over consecutive nodes of the flattened lattice,
at the sizes where that can go wrong: one node more or less than a tile, tiles
that span rows, planes and lattices of a batch, and narrow lattices.

Tolerances are those of the same kernels' parity tests (one FP32 step: 1e-5 of
each weight).
"""
import numpy as np
import pytest

import oracle.d3q19 as o3
from paper_2403_18466_gb300 import inputs
from test_gpu_d3q19 import W, _dev, _np, _weights, field3d, lbm, wpe  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("nx,ny,nz,B", [(31, 1, 1, 1), (11, 3, 1, 1), (8, 4, 2, 1), (5, 3, 3, 3),
                                        (2, 1, 33, 2), (97, 3, 2, 1)])
def test_d3q19_f32_tiles(lbm, nx, ny, nz, B):  # noqa: F811
    """FP32 learned D3Q19 step (tiles of 32 nodes) against the oracle."""
    tau, F = 0.6, 2e-4
    theta = _weights(22)
    lat = lbm.Lattice3D(nx, ny, nz, B, tau=tau, force_amp=F, force_mode=1, device=DEV)
    lat.set_state(_dev(field3d(B, nz, ny, nx, seed=41, neq=0.02)))
    g = o3.stream_push(_np(lat.get_state()))
    th = torch.tensor(theta, dtype=torch.float32, device=DEV)
    lat.step(1, "mlp_f32", lbm.weights3d_struct(th))
    prm = o3.params(tau, force_amp=F, force_mode=1)
    ref = o3.stream_pull(o3.step(o3.MLP, g, prm, np.float32(theta).astype(float)))
    bgk = o3.stream_pull(o3.step(o3.BGK, g, prm))
    got = _np(lat.get_state())
    assert wpe(got, ref) <= 1e-5 and wpe(ref, bgk) > 100 * wpe(got, ref)
    assert lat.status() == lbm.LBM_OK
