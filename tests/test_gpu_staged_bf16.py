"""BF16 storage with z extents that are 4 mod 8: rows of the solver's sinograms are
not whole 16 bytes, which a tensor map needs, so the solver reads them in place and
says so, while the plain operator of the same context (FP32 buffers) stages its rows.
The sums are the same for every entry, bit for bit."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def _context(nz, storage, tile):
    import paper_2604_08997_gb300 as sipo
    n, na = 40, 9
    c = np.arange(n) - (n - 1) / 2
    disc = (c[:, None] ** 2 + c[None, :] ** 2 <= 144.0).astype(np.float32)
    return sipo.sipo_create(dict(nx=n, ny=n, nz=nz, angles=np.arange(na) * (math.pi / na), n_det=n, vial_radius=19.0),
                            np.repeat(disc[:, :, None], nz, axis=2), dict(kase=2, band_width=2, inhibit_ratio=0.9),
                            dict(storage=storage, kkt_tol=0.0, max_iter=8, check_every=4, tile_cfg=tile))


@pytest.mark.parametrize("nz,storage,staged", [(36, "bf16", False), (100, "bf16", False), (260, "bf16", False),
                                               (40, "bf16", True), (100, "f32", True)])
def test_reported_entry_is_the_one_that_runs(nz, storage, staged):
    import paper_2604_08997_gb300 as sipo
    st = sipo.SIPO_F32 if storage == "f32" else sipo.SIPO_BF16
    ctx, ref = _context(nz, st, -1), _context(nz, st, 4)
    ya, yb = (torch.empty(ctx.sino_shape, device="cuda") for _ in range(2))
    a, b = sipo.sipo_solve(ctx, ya), sipo.sipo_solve(ref, yb)
    assert (a["tile_cfg"] >= 5) == staged and b["tile_cfg"] == 4
    assert torch.equal(ya, yb)
    sino = torch.randn(ctx.sino_shape, device="cuda")
    va, vb = (torch.empty(ctx.vol_shape, device="cuda") for _ in range(2))
    assert torch.equal(sipo.sipo_backproject(ctx, sino, va), sipo.sipo_backproject(ref, sino, vb))
    sipo.sipo_destroy(ctx)
    sipo.sipo_destroy(ref)
