"""The plain FP32 backprojection whose rows are read in place (nz not a multiple of 4),
over the view counts at which a tile's views are shared by more warps, against the
oracle (1e-5, the bound of the other operator tests); it does not depend on the
entry that a context's solver step was timed for."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("na", [1, 6, 7, 8, 13, 14, 27, 28, 55, 56, 60])
@pytest.mark.parametrize("nz", [13, 66])
def test_shared_views_match_the_oracle(na, nz):
    import paper_2604_08997_gb300 as sipo
    nx, ny, nd = 22, 19, 27
    rng = np.random.default_rng(na + nz)
    ang = np.sort(rng.uniform(0, 2 * math.pi, na))
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[8:12, 9:13, 3:9] = 1.0
    sino = rng.uniform(-1, 1, (na, nd, nz))
    x = torch.tensor(sino, dtype=torch.float32, device="cuda")
    outs = []
    for tile in (-1, 3, 4):
        ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=9.0, mu=0.02), tgt,
                               dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32, max_iter=0, tile_cfg=tile))
        outs.append(sipo.sipo_backproject(ctx, x, torch.full((ny, nx, nz), 5.0, device="cuda")).clone())
        sipo.sipo_destroy(ctx)
    ref = Operators(Geometry(nx, ny, nz, ang, nd, vial_radius=9.0, mu=0.02)).AT(sino)
    assert np.linalg.norm(outs[0].cpu().numpy().astype(np.float64) - ref) <= 1e-5 * np.linalg.norm(ref)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
