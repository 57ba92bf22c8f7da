"""The single-precision operator kernels at the edges of their tiles.

z forms: one case per form of z groups (16-, 8- and 4-byte groups, one to eight
a lane, ragged ends and more than one tile), against the oracle.  Backprojector:
every tile entry gives the same sums bit for bit, on tiles of eight and of two
rows (the entries add the same terms in the same order), and they match the oracle.  Tolerance: FP32 weights carry at most
1.5e-5 absolute error in u, about 1e-7 of an output after the sum over its taps;
1e-5 is the bound that the other operator tests hold."""
import math

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def _context(nx, ny, nz, ang, nd, vial, mu, storage, tile=-1):
    import paper_2604_08997_gb300 as sipo
    tgt = np.zeros((ny, nx, nz), np.float32)
    tgt[ny // 3: 2 * ny // 3, nx // 3: 2 * nx // 3, nz // 4: max(nz // 4 + 1, 3 * nz // 4)] = 1.0
    return sipo.sipo_create(dict(nx=nx, ny=ny, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                            dict(kase=2, band_width=2), dict(storage=storage, max_iter=0, tile_cfg=tile))


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


# forms: {1,1} 13, 31; {1,2} 33, 63; {1,4} 65, 127; {1,8} 129, 255; two tiles of {1,4} / {1,8} 257, 300 (odd: 301);
# {2,1} 34, 62; {2,2} 66, 126; {2,3} 130, 160, 190; {2,4} 194, 254; {4,1} 96, 128; {4,2} 196, 252 and whole 256, 512
@pytest.mark.parametrize("nz", [13, 31, 33, 63, 65, 127, 129, 255, 257, 301, 34, 62, 66, 126, 130, 160, 190, 194, 254,
                                258, 96, 128, 196, 252, 256, 260, 384, 512])
def test_every_z_form_matches_the_oracle(nz):
    import paper_2604_08997_gb300 as sipo
    rng = np.random.default_rng(nz)
    nx, ny, na, nd = 13, 11, 9, 17
    ang = np.sort(rng.uniform(0, 2 * math.pi, na))
    ctx = _context(nx, ny, nz, ang, nd, 6.0, 0.03, sipo.SIPO_F32)
    geo = Geometry(nx, ny, nz, ang, nd, vial_radius=6.0, mu=0.03)
    ops = Operators(geo)
    vol, sino = rng.uniform(-1, 1, geo.vol_shape), rng.uniform(-1, 1, geo.sino_shape)
    # guarded outputs: nothing is written outside
    out_s = torch.full((na * nd * nz + 64,), 7.0, dtype=torch.float32, device="cuda")
    out_v = torch.full((nx * ny * nz + 64,), 7.0, dtype=torch.float32, device="cuda")
    s, v = out_s[32:-32].view(geo.sino_shape), out_v[32:-32].view(geo.vol_shape)
    sipo.sipo_project(ctx, torch.tensor(vol, dtype=torch.float32, device="cuda"), s)
    sipo.sipo_backproject(ctx, torch.tensor(sino, dtype=torch.float32, device="cuda"), v)
    assert _rel(s.cpu().numpy(), ops.A(vol)) <= 1e-5
    assert _rel(v.cpu().numpy(), ops.AT(sino)) <= 1e-5
    for g in (out_s, out_v):
        assert float(g[:32].min()) == float(g[:32].max()) == float(g[-32:].min()) == float(g[-32:].max()) == 7.0
    sipo.sipo_destroy(ctx)


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_buffers_off_the_16_byte_boundary(shift):
    """Buffers that start 4, 8 or 12 bytes off a 16-byte boundary take narrower groups."""
    import paper_2604_08997_gb300 as sipo
    rng = np.random.default_rng(shift)
    nx, ny, nz, na, nd = 12, 10, 64, 7, 15
    ang = np.sort(rng.uniform(0, math.pi, na))
    ctx = _context(nx, ny, nz, ang, nd, 0.0, 0.0, sipo.SIPO_F32)
    ops = Operators(Geometry(nx, ny, nz, ang, nd))
    n = nx * ny * nz
    vol = rng.uniform(-1, 1, (ny, nx, nz)).astype(np.float32)
    buf = torch.zeros(n + 8, dtype=torch.float32, device="cuda")
    view = buf[shift:shift + n].view(ny, nx, nz)
    view.copy_(torch.from_numpy(vol))
    out = torch.empty((na, nd, nz), dtype=torch.float32, device="cuda")
    sipo.sipo_project(ctx, view, out)
    assert _rel(out.cpu().numpy(), ops.A(vol)) <= 1e-5
    sipo.sipo_backproject(ctx, out, view)
    assert _rel(view.cpu().numpy(), ops.AT(out.cpu().numpy())) <= 1e-5
    sipo.sipo_destroy(ctx)


@pytest.mark.parametrize("case", [
    # nx, ny, nz, views, bins, vial, mu
    (128, 128, 520, 5, 131, 0.0, 0.0),     # tiles of 8 rows, three z tiles of 256 with a remainder of 8
    (131, 125, 392, 4, 120, 61.0, 0.02),   # z tiles of 128, ragged x and y, rows off both detector ends
    (128, 126, 100, 7, 140, 0.0, 0.0),     # one partial z tile, ragged y
    (121, 128, 256, 3, 90, 60.0, 0.03),    # detector narrower than the grid, an odd view left
    (30, 37, 130, 9, 40, 0.0, 0.0),        # nz % 4 != 0: the views of a tile in shares
    (40, 37, 256, 9, 50, 0.0, 0.0),        # tiles of 2 rows, a half tile at the end
])
@pytest.mark.parametrize("uniform", [True, False])
def test_backprojector_entries_agree_bit_for_bit(case, uniform):
    import paper_2604_08997_gb300 as sipo
    nx, ny, nz, na, nd, vial, mu = case
    rng = np.random.default_rng(nx)
    ang = np.arange(na) * (2 * math.pi / na) if uniform else np.sort(rng.uniform(0, 2 * math.pi, na))
    sino = rng.uniform(-1, 1, (na, nd, nz)).astype(np.float32)
    ref = None
    for tile in (0, 2, 3, 4, 5, 6):
        ctx = _context(nx, ny, nz, ang, nd, vial, mu, sipo.SIPO_F32, tile)
        out = torch.full((ny, nx, nz), 3.0, dtype=torch.float32, device="cuda")
        sipo.sipo_backproject(ctx, torch.from_numpy(sino).cuda(), out)
        o = out.cpu().numpy()
        if ref is None:
            ref = o
            assert _rel(o, Operators(Geometry(nx, ny, nz, ang, nd, vial_radius=vial, mu=mu)).AT(sino)) <= 1e-5
        np.testing.assert_array_equal(o, ref, err_msg=f"tile {tile}")
        sipo.sipo_destroy(ctx)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("nz,psf", [(256, 0.0), (300, 0.0), (100, 0.8)])
def test_solves_agree_over_the_backprojector_entries(storage, nz, psf):
    """The fused solver step on staged tiles and on rows read in place: the same
    iterates whatever the entry."""
    import paper_2604_08997_gb300 as sipo
    n, na = 120, 6
    ang = np.arange(na) * (math.pi / na)
    c = np.arange(n) - (n - 1) / 2
    disc = (c[:, None] ** 2 + c[None, :] ** 2 <= 50.0 ** 2).astype(np.float32)
    tgt = np.repeat(disc[:, :, None], nz, axis=2)
    tgt[:, :, : nz // 8] = 0.0
    ys = []
    for tile in (3, 4, 5):
        ctx = sipo.sipo_create(dict(nx=n, ny=n, nz=nz, angles=ang, n_det=n, psf_sigma=(psf, psf, psf)), tgt,
                               dict(kase=2, band_width=2, inhibit_ratio=0.9),
                               dict(storage=sipo.SIPO_F32 if storage == "f32" else sipo.SIPO_BF16, kkt_tol=0.0,
                                    max_iter=12, check_every=4, tile_cfg=tile))
        y = torch.empty(ctx.sino_shape, dtype=torch.float32, device="cuda")
        sipo.sipo_solve(ctx, y)
        ys.append(y.cpu().numpy())
        sipo.sipo_destroy(ctx)
    assert float(np.abs(ys[0]).max()) > 0.0
    np.testing.assert_array_equal(ys[1], ys[0])
    np.testing.assert_array_equal(ys[2], ys[0])
