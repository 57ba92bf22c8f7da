"""Faults of the staged backprojector belong to the context whose launch recorded
them.  The fault is made on the host (sipo_post_fault writes the words that the
kernel would write); no launch gives up and nothing faults on the device."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

NX, NY, NZ, NA, ND = 16, 14, 32, 6, 17


def test_null_context_and_bits_are_refused():
    from paper_2604_08997_gb300 import _abi
    lib = _abi.load()
    assert lib.sipo_check_fault(None) == -1
    assert lib.sipo_post_fault(None, 1) == -1


def _context(sipo, sigma=(0.0, 0.0, 0.0)):
    tgt = np.zeros((NY, NX, NZ), np.float32)
    tgt[5:9, 6:10, 8:20] = 1.0
    return sipo.sipo_create(dict(nx=NX, ny=NY, nz=NZ, angles=np.arange(NA) * (math.pi / NA), n_det=ND,
                                 psf_sigma=sigma), tgt, dict(kase=2, band_width=2, inhibit_ratio=0.9),
                            dict(storage=sipo.SIPO_F32, kkt_tol=0.0, max_iter=8, check_every=4))


@pytest.mark.gpu
def test_pending_fault_is_reported_once_by_the_next_call_of_its_context():
    import paper_2604_08997_gb300 as sipo
    from paper_2604_08997_gb300._abi import SIPO_ERR_NUMERIC, SIPO_ERR_TIMEOUT, sipo_post_fault
    a, b = _context(sipo), _context(sipo, (1.0, 1.0, 1.0))
    sino = torch.rand((NA, ND, NZ), device="cuda")
    vol = torch.rand((NY, NX, NZ), device="cuda")
    good = sipo.sipo_backproject(a, sino, torch.empty_like(vol)).clone()
    calls = [lambda c: sipo.sipo_project(c, vol, torch.empty_like(sino)),
             lambda c: sipo.sipo_backproject(c, sino, torch.empty_like(vol)),
             lambda c: sipo.sipo_psf_grad(c, sino, vol), lambda c: sipo.sipo_solve(c),
             lambda c: sipo.sipo_solve_batched([c]), lambda c: sipo.sipo_check_fault(c)]
    for call in calls:
        for bits, code in ((1, SIPO_ERR_TIMEOUT), (2, SIPO_ERR_NUMERIC), (3, SIPO_ERR_TIMEOUT)):
            sipo_post_fault(b, bits)
            for other in calls:  # another context is not charged with it
                other(a)
            with pytest.raises(sipo.SipoError) as e:
                call(b)
            assert e.value.code == code
            call(b)  # reported once; the context stays usable
    assert torch.equal(sipo.sipo_backproject(a, sino, torch.empty_like(vol)), good)
    sipo.sipo_destroy(a)
    sipo.sipo_destroy(b)
