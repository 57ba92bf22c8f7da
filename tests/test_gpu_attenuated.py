"""The two-bin projector under an attenuation so strong that products of weight
and attenuation underflow to zero in single precision (mu R = 110; exp(-104) is
below the smallest float).  A candidate whose product is zero is no tap: the
checked build counts the places that each lane reserves in the tap list against
those it writes.  Rays whose factors all stay within the float range agree with
the sum over voxels in 64 bits, to 1.5e-5 absolute in a tap's weight (the bound
on u of the other operator tests) and 4e-6 of an output for the rounded factors and the sum (64 roundings)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
N, NZ, R, MU = 21, 16, 10.0, 11.0


def _problem(na=12):
    ang = np.arange(na) * (2 * np.pi / na) + 0.05
    vol = np.random.default_rng(5).uniform(0.5, 1.0, (N, N, NZ)).astype(np.float32)
    return ang, vol


def _project(ang, vol):
    import torch
    import paper_2604_08997_gb300 as sipo
    tgt = np.zeros((N, N, NZ), np.float32)
    tgt[8:12, 9:13, 4:12] = 1.0
    ctx = sipo.sipo_create(dict(nx=N, ny=N, nz=NZ, angles=ang, n_det=N, vial_radius=R, mu=MU), tgt,
                           dict(kase=2, band_width=2), dict(storage=sipo.SIPO_F32, max_iter=0))
    out = torch.empty((len(ang), N, NZ), dtype=torch.float32, device="cuda")
    sipo.sipo_project(ctx, torch.from_numpy(vol).cuda(), out)
    res = out.cpu().numpy().astype(np.float64)
    sipo.sipo_destroy(ctx)
    return res


def test_rays_within_the_float_range_agree_with_the_sum_in_64_bits():
    ang, vol = _problem()
    out = _project(ang, vol)
    c = np.arange(N) - (N - 1) / 2
    x, y = c[None, :], c[:, None]
    inside = x * x + y * y <= R * R
    tested = 0
    for k, th in enumerate(ang):
        u = x * np.cos(th) + y * np.sin(th) + (N - 1) / 2
        fx, fy = MU * x * np.sin(th), -MU * y * np.cos(th)
        for j in range(N):
            s = j - (N - 1) / 2
            near = inside & (np.abs(u - j) < 1 + 1e-4)
            if not near.any():
                continue
            ex = np.concatenate([(fx + 0 * fy)[near], (fy + 0 * fx)[near], (fx + fy)[near]])
            es = -MU * np.sqrt(max(R * R - s * s, 0.0))
            if np.abs(ex).max() > 80 or es < -80:
                continue
            e = np.where(near, np.exp(np.where(near, fx + fy, 0.0) + es), 0.0)
            w = np.maximum(0.0, 1.0 - np.abs(u - j))
            ref = ((w * e)[:, :, None] * vol.astype(np.float64)).sum(axis=(0, 1))
            bound = 1.5e-5 * (e[:, :, None] * vol).sum(axis=(0, 1)) + 4e-6 * ref
            assert (np.abs(out[k, j] - ref) <= bound).all(), (k, j)
            tested += 1
    assert tested >= 8


def test_tap_list_has_no_unwritten_place():
    sys.path.insert(0, ROOT)
    from paper_2604_08997_gb300.build import build
    build(checked=True)
    r = subprocess.run([sys.executable, os.path.abspath(__file__), "--exercise"], cwd=ROOT, capture_output=True,
                       text=True, timeout=1200, env=dict(os.environ, SIPO_LIBRARY="checked"))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    flags = int([l for l in r.stdout.splitlines() if l.startswith("CHECK_FLAGS")][-1].split()[1], 16)
    assert flags & 0x40000000, "the child did not load the checked build"
    assert flags & 1 == 0, f"checks fired: {flags:#x}"  # (bit 3: central rays overflow, as they do in 32 bits)


if __name__ == "__main__" and "--exercise" in sys.argv:
    sys.path.insert(0, ROOT)
    from paper_2604_08997_gb300 import _abi
    _project(*_problem())
    print("CHECK_FLAGS", hex(_abi.load().sipo_check_flags()), flush=True)
