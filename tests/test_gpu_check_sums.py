"""The check step's sums do not depend on which z values a lane holds: a solve whose
slices are put in another order (single ones where nz is not a multiple of 4,
groups of four otherwise) reports the same residuals and, after a restart, the same
primal weight.  Slices are independent but for scalars formed from sums over all of
them.  Tolerance: a sum passes at most some hundred FP64 additions on its way from a
thread to the total, a relative error of 100 * 1.1e-16; 1e-12 holds a hundred times
that, and is a hundredth of what a sum of several values in single precision leaves
(6e-8 each, about 1e-10 over some thousand of them)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

REL_P, REL_D, OMEGA, RESTARTS = 2, 3, 6, 7


def _trace(heights, storage):
    import paper_2604_08997_gb300 as sipo
    n, na, nz = 16, 6, len(heights)
    c = np.arange(n) - (n - 1) / 2
    disc = (c[:, None] ** 2 + (c[None, :] - 1.5) ** 2 <= 16.0).astype(np.float32)
    ctx = sipo.sipo_create(dict(nx=n, ny=n, nz=nz, angles=np.arange(na) * (math.pi / na) + 0.1, n_det=n),
                           np.ascontiguousarray(disc[:, :, None] * heights),
                           dict(kase=sipo.SIPO_GENERAL, band_width=2),
                           dict(storage=storage, kkt_tol=0.0, max_iter=80, check_every=8))
    sipo.sipo_solve(ctx)
    out = sipo.sipo_get_trace(ctx)
    sipo.sipo_destroy(ctx)
    return out


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("nz", [65, 130, 160, 200])
def test_check_sums_do_not_depend_on_the_order_of_the_slices(nz, storage):
    import paper_2604_08997_gb300 as sipo
    rng = np.random.default_rng(nz)
    heights = rng.uniform(0.3, 1.0, nz).astype(np.float32)
    width = 4 if nz % 4 == 0 else 1
    order = (rng.permutation(nz // width)[:, None] * width + np.arange(width)).reshape(-1)
    st = sipo.SIPO_F32 if storage == "f32" else sipo.SIPO_BF16
    a, b = _trace(heights, st), _trace(heights[order], st)
    assert a.shape == b.shape and a[-1, RESTARTS] >= 1
    n = int(np.argmax(a[:, RESTARTS] >= 1)) + 1  # up to the first check after a restart
    assert float(a[:n, REL_D].max()) > 0.0
    np.testing.assert_allclose(b[:n][:, [REL_P, REL_D, OMEGA, RESTARTS]],
                               a[:n][:, [REL_P, REL_D, OMEGA, RESTARTS]], rtol=1e-12, atol=0)
