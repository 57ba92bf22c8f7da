"""Long thin slices in double precision: the flat projector forms its candidate
window in single precision and keeps it to sides of 16384; longer ones take the
kernels with lanes over z.  Against the sum over voxels in 64 bits.  Tolerance:
u carries a few roundings of a coordinate below the side M, so a weight is off by
at most 4 x 2^-52 M."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("side", [16384, 16385, 524288, 1000003])
@pytest.mark.parametrize("along_x", [True, False])
def test_long_slices_lose_no_tap(side, along_x):
    import paper_2604_08997_gb300 as sipo
    nx, ny = (side, 24) if along_x else (24, side)
    ang = np.array([0.0, 0.2, 0.78, -0.7])
    if not along_x:
        ang = math.pi / 2 - ang
    nd = side
    tgt = np.zeros((ny, nx, 1), np.float32)
    tgt[1, 1, 0] = 1.0
    ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=1, angles=ang, n_det=nd), tgt, dict(kase=2, band_width=1),
                           dict(storage=sipo.SIPO_F64, max_iter=0))
    vol = np.random.default_rng(side).uniform(-1, 1, (ny, nx, 1))
    out = torch.empty((len(ang), nd, 1), dtype=torch.float64, device="cuda")
    sipo.sipo_project(ctx, torch.from_numpy(vol).cuda(), out)
    x = (np.arange(nx) - (nx - 1) / 2)[None, :]
    y = (np.arange(ny) - (ny - 1) / 2)[:, None]
    ref = np.zeros((len(ang), nd))
    for k, th in enumerate(ang):
        u = x * np.cos(th) + y * np.sin(th) + (nd - 1) / 2
        i = np.floor(u).astype(np.int64)
        w = u - i
        for bins, val in ((i, (1 - w) * vol[..., 0]), (i + 1, w * vol[..., 0])):
            ok = (bins >= 0) & (bins < nd)
            ref[k] += np.bincount(bins[ok], val[ok], nd)
    err = np.linalg.norm(out.cpu().numpy()[..., 0] - ref) / np.linalg.norm(ref)
    assert err <= 4 * 2.0 ** -52 * side
    sipo.sipo_destroy(ctx)
