"""Infinite and NaN voxels reach the bins that weigh them and no other: the
projection of a volume that holds some is finite, and bit for bit that of the
volume without them, wherever the projection of their indicator is zero.  Views
along the axes put voxels on bins exactly (a weight of zero beside one of one)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("nz", [1, 3, 20, 36, 130])
@pytest.mark.parametrize("vial,mu", [(0.0, 0.0), (9.0, 0.05)])
def test_non_finite_voxels_reach_only_their_bins(storage, nz, vial, mu):
    import paper_2604_08997_gb300 as sipo
    nx = ny = 21
    nd, na = 23, 16
    ang = np.concatenate([np.arange(8) * (math.pi / 4), np.random.default_rng(nz).uniform(0, 2 * math.pi, na - 8)])
    real = torch.float32 if storage == "f32" else torch.float64
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[9:12, 8:13, nz // 3: nz // 3 + 1] = 1.0
    ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                           dict(kase=2, band_width=2),
                           dict(storage=sipo.SIPO_F32 if storage == "f32" else sipo.SIPO_F64, max_iter=0))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(nz)
    vol = torch.randn((ny, nx, nz), generator=gen, device="cuda", dtype=real)
    spots = [(4, 10, 0, math.inf), (10, 4, nz - 1, math.nan), (13, 12, nz // 2, -math.inf), (0, 0, 0, math.inf)]
    flag = torch.zeros_like(vol)
    for y, x, z, _ in spots:
        flag[y, x, z] = 1.0
    run = lambda v: sipo.sipo_project(ctx, v, torch.empty((na, nd, nz), device="cuda", dtype=real))
    reach = run(flag) != 0
    plain = run(torch.where(flag != 0, torch.zeros_like(vol), vol))
    for y, x, z, value in spots:
        vol[y, x, z] = value
    out = run(vol)
    assert bool(reach.any())
    assert not bool(torch.isfinite(out[reach]).any())
    assert torch.equal(out[~reach], plain[~reach])
    sipo.sipo_destroy(ctx)
