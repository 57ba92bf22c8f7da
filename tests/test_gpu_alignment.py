"""Buffers of a caller that start 4, 8 or 12 bytes off a 16-byte boundary, under
a point spread function: the blur moves four z values at a time only where the
buffers allow it.  Radii for both of its forms (x and y in one pass, and one
pass an axis where the z radius is above 16), against the oracle, with the bound
of the other single-precision operator tests."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators, apply_psf

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def _rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b))


def _shifted(shape, shift):
    n = int(np.prod(shape))
    return torch.zeros(n + 8, dtype=torch.float32, device="cuda")[shift:shift + n].view(shape)


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("sigma", [(1.0, 0.8, 1.2), (0.7, 0.7, 4.5)])
def test_blur_of_buffers_off_the_16_byte_boundary(shift, sigma):
    import paper_2604_08997_gb300 as sipo
    nx, ny, nz, na, nd = 12, 10, 64, 7, 15
    rng = np.random.default_rng(shift)
    ang = np.sort(rng.uniform(0, math.pi, na))
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[4:7, 4:8, 20:40] = 1.0
    ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, psf_sigma=sigma), tgt,
                           dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32, max_iter=0))
    geo = Geometry(nx, ny, nz, ang, nd, psf_sigma=sigma)
    ops = Operators(geo)
    vol, sino = rng.uniform(0, 1, geo.vol_shape), rng.uniform(0, 1, geo.sino_shape)
    v, s, out = _shifted(geo.vol_shape, shift), _shifted(geo.sino_shape, shift), _shifted(geo.vol_shape, shift)
    v.copy_(torch.from_numpy(vol))
    sipo.sipo_project(ctx, v, s)
    assert _rel(s, ops.A(vol)) <= 1e-5
    s.copy_(torch.from_numpy(sino))
    sipo.sipo_backproject(ctx, s, out)
    assert _rel(out, ops.AT(sino)) <= 1e-5
    sipo.sipo_psf_apply(ctx, v, out)
    assert _rel(out, apply_psf(geo, vol)) <= 1e-5
    grad = sipo.sipo_psf_grad(ctx, s, v)
    ref = sipo.sipo_psf_grad(ctx, s.clone(), v.clone())
    np.testing.assert_allclose(grad, ref, rtol=1e-5)
    sipo.sipo_destroy(ctx)
