"""The two-bin projector at the edges of its pairs (and the staged backprojector
on the same geometries, whose boxes are then larger than the detector): odd and even numbers of bins,
bins 0 and 1 (the literal weight rule), rays off the vial, views that leave a
tile of four partly filled, against the oracle.  FP32 bound as for the other operator tests."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("nd", [1, 2, 3, 15, 16, 17, 31])
@pytest.mark.parametrize("na", [1, 3, 5])
@pytest.mark.parametrize("vial,mu", [(0.0, 0.0), (6.5, 0.05)])
def test_pairs_match_the_oracle(nd, na, vial, mu):
    import paper_2604_08997_gb300 as sipo
    nx, ny, nz = 14, 17, 36
    rng = np.random.default_rng(nd + 100 * na)
    for ang in (np.arange(na) * (2 * math.pi / na), np.sort(rng.uniform(0, 2 * math.pi, na))):
        tgt = np.zeros((ny, nx, nz), np.float32)
        tgt[7:10, 5:9, 10:20] = 1.0
        ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                               dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32, max_iter=0))
        geo = Geometry(nx, ny, nz, ang, nd, vial_radius=vial, mu=mu)
        vol = rng.uniform(-1, 1, geo.vol_shape)
        out = torch.full(geo.sino_shape, 5.0, dtype=torch.float32, device="cuda")
        sipo.sipo_project(ctx, torch.tensor(vol, dtype=torch.float32, device="cuda"), out)
        ref = Operators(geo).A(vol)
        err = np.linalg.norm(out.cpu().numpy().astype(np.float64) - ref) / max(np.linalg.norm(ref), 1e-300)
        assert err <= 1e-5
        sino = rng.uniform(-1, 1, geo.sino_shape)
        dose = torch.full(geo.vol_shape, 5.0, dtype=torch.float32, device="cuda")
        sipo.sipo_backproject(ctx, torch.tensor(sino, dtype=torch.float32, device="cuda"), dose)
        ref = Operators(geo).AT(sino)
        err = np.linalg.norm(dose.cpu().numpy().astype(np.float64) - ref) / max(np.linalg.norm(ref), 1e-300)
        assert err <= 1e-5
        sipo.sipo_destroy(ctx)
