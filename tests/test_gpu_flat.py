"""The flat (few z values) operator kernels at the edges of their tiles: 31 bins
and 32 voxels a warp, chunks of 16 (FP32) or 8 (FP64) lines, z up to 8, against
the oracle.  Tolerances as for the z-lane kernels: FP32 weights carry at most
1.5e-5 absolute error in u, averaged over the taps of an output; FP64 1e-12."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

CASES = [
    # nx, ny, nz, views, bins, vial, mu
    (32, 31, 1, 9, 31, 0.0, 0.0),       # one tile of bins, one of voxels
    (33, 16, 1, 8, 32, 0.0, 0.0),       # one bin, one voxel over
    (95, 70, 1, 17, 125, 33.0, 0.02),   # tiles of bins with a remainder, vial and attenuation
    (64, 64, 2, 5, 63, 31.0, 0.0),      # z stride 2, vial without attenuation
    (17, 40, 7, 6, 62, 0.0, 0.0),       # odd z, detector wider than the grid
    (40, 17, 3, 4, 12, 8.0, 0.1),       # detector narrower than the grid
    (3, 200, 1, 7, 201, 0.0, 0.0),      # long lines one way
    (200, 3, 1, 7, 201, 0.0, 0.0),      # and the other
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("uniform", [True, False])
def test_flat_pair_matches_the_oracle(case, storage, uniform):
    import paper_2604_08997_gb300 as sipo
    nx, ny, nz, na, nd, vial, mu = case
    rng = np.random.default_rng(nx + 7 * ny)
    # uniform views include the axes, where voxels fall on bins exactly
    ang = np.arange(na) * (2 * math.pi / na) if uniform else np.sort(rng.uniform(0, 2 * math.pi, na))
    dt = torch.float32 if storage == "f32" else torch.float64
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[ny // 3: ny // 3 + 2, nx // 3: nx // 3 + 2] = 1.0
    ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                           dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32 if storage == "f32" else
                                                            sipo.SIPO_F64, max_iter=0))
    geo = Geometry(nx, ny, nz, ang, nd, vial_radius=vial, mu=mu)
    ops = Operators(geo)
    vol, sino = rng.uniform(-1, 1, geo.vol_shape), rng.uniform(-1, 1, geo.sino_shape)
    out_s = torch.empty(geo.sino_shape, dtype=dt, device="cuda")
    out_v = torch.empty(geo.vol_shape, dtype=dt, device="cuda")
    sipo.sipo_project(ctx, torch.tensor(vol, dtype=dt, device="cuda"), out_s)
    sipo.sipo_backproject(ctx, torch.tensor(sino, dtype=dt, device="cuda"), out_v)
    for out, ref in ((out_s, ops.A(vol)), (out_v, ops.AT(sino))):
        err = np.linalg.norm(out.cpu().numpy().astype(np.float64) - ref) / np.linalg.norm(ref)
        assert err <= (1e-5 if storage == "f32" else 1e-12)
    sipo.sipo_destroy(ctx)
