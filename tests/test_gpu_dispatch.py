"""The routes that a call takes by its size: sweep forms, particle blocks and spectrum bins at the
edges of their rules, against the general route or the oracle.

Tolerances. Two sweep forms differ by the rounding of a few dozen float32 operations per cell:
1e-6 relative L2 (10 ulp). The force readout sums eight float32 products: 1e-6. Spectra: FP64
sums of a float32 transform, whose modes carry about 1e-6 of the rms mode: 1e-5 for the bins,
1e-4 for their derivative; k and mode counts are sums of exact terms, 1e-12.
"""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import f32, lib, need_gpu, rel_l2
from oracle import pm as opm
from oracle import spectra as osp

pytestmark = pytest.mark.gpu
TILE = 1


@pytest.fixture(scope="module")
def dh():
    need_gpu()
    return lib()


@pytest.mark.parametrize("n", [4, 5, 33, 96, 97, 98, 100])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_default_sweeps_match_the_tile(dh, n, axis):
    u, _ = f32(synth.gas_state(n, 3))
    lam, _ = f32(synth.rng(4).normal(size=(5, n, n, n)))
    for variant in (0, 4, 5):
        got = dh.sweep(u, axis, 0.4, variant=variant)
        assert rel_l2(got, dh.sweep(u, axis, 0.4, variant=TILE)) < 1e-6, variant


@pytest.mark.parametrize("n", [4, 5, 33, 96, 97, 98, 100])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_adjoint_does_not_depend_on_the_segments(dh, n, axis):
    """A cell's adjoint is the same arithmetic wherever its line is cut: bitwise equal for
    segments of 32, 16 and the fitted length (whole lines, ragged last segments, one segment)."""
    u, _ = f32(synth.gas_state(n, 3))
    lam, _ = f32(synth.rng(4).normal(size=(5, n, n, n)))
    want, _ = dh.sweep_adjoint(u, lam, axis, 0.4)
    for variant in (2, 3, 4):
        got, _ = dh.sweep_adjoint(u, lam, axis, 0.4, variant=variant)
        assert torch.equal(got, want), variant


@pytest.mark.parametrize("n", [42, 43, 45, 48, 64, 80])  # bricks from 43 on, 16 or 32 wide
def test_readout_and_deposit(dh, n):
    box = float(n)
    s, s_o = f32(synth.displacements(n, 5, 2.5))
    g, g_o = f32(synth.field(n, 6, shape=(3, n, n, n)))
    assert rel_l2(dh.interp_cic(g, s, n, box), opm.interp(g_o, s_o, n, box, index_fp32=True)) < 1e-6
    one = torch.ones(n ** 3, dtype=torch.float64)
    assert rel_l2(dh.deposit_cic(s, n, box), opm.deposit(s_o, one, n, box, index_fp32=True)) < 1e-6


def test_deposit_values_of_any_size_and_sign(dh):
    """Values whose fixed-point weights pass 2^31 and 2^32 units, and negative ones."""
    n, box = 16, 16.0
    s, s_o = f32(synth.displacements(n, 7, 0.8))
    v, v_o = f32(np.where(np.arange(n ** 3) % 3 == 0, -1.0, 1.0) * 10.0 ** (np.arange(n ** 3) % 7 - 3))
    got = dh.deposit_cic(s, n, box, values=v)
    want = opm.deposit(s_o, v_o, n, box, index_fp32=True)
    assert rel_l2(got, want) < 1e-6


@pytest.mark.parametrize("n,nbins", [(2, 4), (3, 1), (5, 3), (16, 8), (17, 30), (45, 22), (64, 40)])
def test_spectra_bins(dh, n, nbins):
    box = 10.0
    a, a_o = f32(synth.field(n, 8))
    b, b_o = f32(synth.field(n, 9))
    k, pk, nm = (t.cpu() for t in dh.power_spectrum(a, box, nbins))
    ko, po, no = osp.power_spectrum(a_o, box, nbins)
    assert torch.equal(nm, torch.as_tensor(no, dtype=torch.float64))
    assert torch.allclose(k, torch.as_tensor(ko, dtype=torch.float64), rtol=1e-12, atol=0)
    assert rel_l2(pk, po) < 1e-5
    _, px, _ = dh.power_spectrum(a, box, nbins, b=b)
    _, pxo, _ = osp.power_spectrum(a_o, box, nbins, b_o)
    assert (px.cpu() - torch.as_tensor(pxo)).norm() < 1e-5 * torch.as_tensor(po).norm()
    w = torch.linspace(-1.0, 1.0, nbins, dtype=torch.float64)
    da = dh.power_spectrum_adjoint(a, box, nbins, w.cuda())
    x = a_o.clone().requires_grad_(True)
    (g,) = torch.autograd.grad((osp.power_spectrum(x, box, nbins)[1] * w).sum(), x)
    assert rel_l2(da, g) < 1e-4
    _, rc, _ = dh.cross_correlation(a, b, box, nbins)
    pb = osp.power_spectrum(b_o, box, nbins)[1]
    want = torch.where((po > 0) & (pb > 0), pxo / (po * pb).clamp_min(1e-300).sqrt(), torch.zeros_like(po))
    assert (rc.cpu() - want).abs().max() < 1e-5
