"""The double-precision operators at the z extents where their kernels change (flat
forms, single values, pairs, pairs of groups, ragged ends) and with buffers 8 bytes
off a 16-byte boundary, against the oracle, to 1e-12 as in the other FP64 tests.
Outputs are guarded: nothing is written outside them."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def _check(nx, ny, nz, na, nd, vial, mu, shift=0):
    import paper_2604_08997_gb300 as sipo
    rng = np.random.default_rng(nz + 1000 * shift + nd)
    ang = np.sort(rng.uniform(0, 2 * math.pi, na))
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[ny // 2 - 1: ny // 2 + 2, nx // 2 - 1: nx // 2 + 2, nz // 2: nz // 2 + 1] = 1.0
    ctx = sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                           dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F64, max_iter=0))
    geo = Geometry(nx, ny, nz, ang, nd, vial_radius=vial, mu=mu)
    ops = Operators(geo)
    for shape, out_shape, call, ref in ((geo.vol_shape, geo.sino_shape, sipo.sipo_project, ops.A),
                                        (geo.sino_shape, geo.vol_shape, sipo.sipo_backproject, ops.AT)):
        x = rng.uniform(-1, 1, shape)
        src = torch.zeros(x.size + 4, dtype=torch.float64, device="cuda")
        src[shift: shift + x.size] = torch.from_numpy(x.reshape(-1)).cuda()
        n = int(np.prod(out_shape))
        buf = torch.full((n + 64,), 7.0, dtype=torch.float64, device="cuda")
        out = buf[32 + shift: 32 + shift + n].view(out_shape)
        call(ctx, src[shift: shift + x.size].view(shape), out)
        want = ref(x)
        assert np.linalg.norm(out.cpu().numpy() - want) <= 1e-12 * np.linalg.norm(want)
        assert bool((buf[: 32 + shift] == 7.0).all()) and bool((buf[32 + shift + n:] == 7.0).all())
    sipo.sipo_destroy(ctx)


@pytest.mark.parametrize("nz", [1, 2, 3, 4, 5, 6, 7, 9, 10, 31, 32, 33, 34, 63, 64, 66, 127, 128, 130, 256, 258])
@pytest.mark.parametrize("nd", [17, 29])
def test_every_extent_matches_the_oracle(nz, nd):
    _check(13, 11, nz, 9, nd, 6.0, 0.03)


@pytest.mark.parametrize("nz", [2, 4, 7, 34, 128])
def test_buffers_8_bytes_off(nz):
    _check(12, 10, nz, 7, 15, 0.0, 0.0, shift=1)


@pytest.mark.parametrize("nz", [6, 7, 9, 10])
def test_large_slices(nz):
    _check(128, 126, nz, 3, 131, 61.0, 0.0)
