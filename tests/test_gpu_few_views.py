"""The single-precision projector takes other kernels where a launch would leave most
of the chip empty (one bin a warp instead of two, narrower z groups, z lanes
instead of lanes over bins).  All of them add the same terms in the same order: the
sums of a few views are, bit for bit, those of the same views among many, for finite
volumes and for volumes that hold infinite and NaN voxels, and they match the oracle
(1e-5, the bound of the other operator tests)."""
import math
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle.operators import Geometry, Operators

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
NX, NY, FEW = 14, 17, 7


def _project(ang, nd, vial, mu, vol):
    import paper_2604_08997_gb300 as sipo
    nz = vol.shape[2]
    tgt = np.zeros((NY, NX, nz), np.float32)
    tgt[7:10, 5:9, nz // 2: nz // 2 + 1] = 1.0
    ctx = sipo.sipo_create(dict(nx=NX, ny=NY, nz=nz, angles=ang, n_det=nd, vial_radius=vial, mu=mu), tgt,
                           dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32, max_iter=0))
    out = sipo.sipo_project(ctx, vol, torch.full((len(ang), nd, nz), 5.0, device="cuda"))
    torch.cuda.synchronize()
    sipo.sipo_destroy(ctx)
    return out


@pytest.mark.parametrize("vial,mu", [(0.0, 0.0), (6.5, 0.05)])
@pytest.mark.parametrize("nz", [1, 2, 5, 8, 13, 36, 66, 100, 130, 256, 300])
@pytest.mark.parametrize("nd", [1, 2, 3, 16, 17, 31])
def test_few_views_and_many_give_the_same_sums(nd, nz, vial, mu):
    rng = np.random.default_rng(nd + 100 * nz)
    # 12000 rays or pairs fill the chip at any extent; the few are spread among the many
    many = 12000 // ((nd + 1) // 2)
    ang = np.concatenate([np.arange(8) * (math.pi / 4), rng.uniform(0, 2 * math.pi, many - 8)])
    ang = ang[rng.permutation(many)]
    at = np.sort(rng.choice(many, FEW, replace=False))
    vol = torch.from_numpy(rng.uniform(-1, 1, (NY, NX, nz)).astype(np.float32)).cuda()
    few, all_ = _project(ang[at], nd, vial, mu, vol), _project(ang, nd, vial, mu, vol)
    assert torch.equal(few, all_[at])
    ref = Operators(Geometry(NX, NY, nz, ang[at], nd, vial_radius=vial, mu=mu)).A(vol.cpu().numpy().astype(np.float64))
    err = np.linalg.norm(few.cpu().numpy().astype(np.float64) - ref) / max(np.linalg.norm(ref), 1e-300)
    assert err <= 1e-5
    vol[3, 7, 0], vol[9, 4, nz - 1], vol[12, 9, nz // 2] = math.inf, math.nan, -math.inf
    few, all_ = _project(ang[at], nd, vial, mu, vol), _project(ang, nd, vial, mu, vol)[at]
    assert torch.equal(torch.isnan(few), torch.isnan(all_))
    assert torch.equal(torch.nan_to_num(few, 0.0, 9e30, -9e30), torch.nan_to_num(all_, 0.0, 9e30, -9e30))


def test_tap_list_of_pairs_has_no_unwritten_place():
    """The check of the attenuated tests (a strong attenuation, whose products underflow)
    with views enough for two bins a warp."""
    sys.path.insert(0, ROOT)
    from paper_2604_08997_gb300.build import build
    build(checked=True)
    code = ("import sys; sys.path[:0] = [%r, %r]; import test_gpu_attenuated as t; t._project(*t._problem(600)); "
            "from paper_2604_08997_gb300 import _abi; print('CHECK_FLAGS', hex(_abi.load().sipo_check_flags()))"
            % (ROOT, HERE))
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=1200,
                       env=dict(os.environ, SIPO_LIBRARY="checked"))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    flags = int([l for l in r.stdout.splitlines() if l.startswith("CHECK_FLAGS")][-1].split()[1], 16)
    assert flags & 0x40000000, "the child did not load the checked build"
    assert flags & 1 == 0, f"checks fired: {flags:#x}"
