"""The binned spectra of float32 fields in any units: P(k) and the cross spectrum scale with the
product of the amplitudes, r_c does not change, and non-finite fields give non-finite powers.

Tolerances as for fields of order one (test_gpu_dispatch.py): the powers are FP64 sums of a float32
transform, 1e-5; the amplitudes keep every mode a normal float32 number. Amplitudes next to
1e-14 and 1e15 put the products of a warp on either side of the range of float pairs.
"""
import pytest
import torch

import synth
from gpu_helpers import f32, lib, need_gpu, rel_l2
from oracle import spectra as osp

pytestmark = pytest.mark.gpu
BOX, NBINS = 10.0, 16


@pytest.fixture(scope="module")
def dh():
    need_gpu()
    return lib()


@pytest.mark.parametrize("n", [17, 32])
@pytest.mark.parametrize("amp,amp_b", [(1e-30, 1e-30), (1e-24, 1e-24), (1e18, 1e18), (1e25, 1e25),
                                       (1e-30, 1e25), (1e-15, 1e-15), (1e-14, 1e-14),
                                       (3e13, 3e13), (1e15, 1e15), (1.0, 1e-27), (1e20, 1.0)])
def test_spectra_of_any_amplitude(dh, n, amp, amp_b):
    a, a_o = f32(synth.field(n, 8) * amp)
    b, b_o = f32(synth.field(n, 9) * amp_b)
    _, po, no = osp.power_spectrum(a_o, BOX, NBINS)
    pb = osp.power_spectrum(b_o, BOX, NBINS)[1]
    pxo = osp.power_spectrum(a_o, BOX, NBINS, b_o)[1]
    _, pk, nm = (t.cpu() for t in dh.power_spectrum(a, BOX, NBINS))
    assert torch.equal(nm, torch.as_tensor(no, dtype=torch.float64))
    assert rel_l2(pk, po) < 1e-5
    _, px, _ = (t.cpu() for t in dh.power_spectrum(a, BOX, NBINS, b=b))
    scale = (po * pb).sqrt()
    assert ((px - pxo).norm() / scale.norm()).item() < 1e-5
    _, rc, _ = dh.cross_correlation(a, b, BOX, NBINS)
    want = torch.where(scale > 0, pxo / scale.clamp_min(1e-300), torch.zeros_like(scale))
    assert (rc.cpu() - want).abs().max() < 1e-5


def test_zero_and_non_finite_fields(dh):
    n = 16
    a = f32(synth.field(n, 8))[0]
    zero = torch.zeros_like(a)
    _, pk, nm = dh.power_spectrum(zero, BOX, 8)
    assert (pk == 0).all() and (nm > 0).all()
    _, px, _ = dh.power_spectrum(a, BOX, 8, b=zero)
    assert (px == 0).all()
    _, rc, _ = dh.cross_correlation(a, zero, BOX, 8)
    assert (rc == 0).all()
    for bad in (float("inf"), float("nan")):
        x = a.clone()
        x[1, 2, 3] = bad
        assert not torch.isfinite(dh.power_spectrum(x, BOX, 8)[1]).any()
        assert not torch.isfinite(dh.power_spectrum(x, BOX, 8, b=a)[1]).any()
