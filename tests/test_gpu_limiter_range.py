"""Limiter partials of tiny differences: a transverse momentum of 1e-19 on a uniform flow, whose
face differences (about 1e-20) square below float32's range while their product does not vanish.

Tolerance. The fluxes carry float32 rounding (6e-8) and neighbours differ by a tenth of them or
more, so the ratio that the partials depend on is good to about 2e-6: 1e-5 relative L2.
"""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import f32, lib, need_gpu, rel_l2
from oracle import hydro as ohy

pytestmark = pytest.mark.gpu
GAMMA, NU = 5.0 / 3.0, 0.4


@pytest.mark.parametrize("variant", [0, 1, 2, 4])
@pytest.mark.parametrize("n", [15, 16])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_adjoint_of_tiny_transverse_momenta(n, axis, variant):
    need_gpu()
    dh = lib()
    x = np.sin(2 * np.pi * np.arange(n) / n + 0.1)
    row = 1e-19 * (0.5 + 0.5 * synth.rng(2).random((n, n, n)).mean(axis=2 - axis, keepdims=True))
    U = np.zeros((5, n, n, n))
    U[0], U[4] = 1.0, 2.5
    U[1 + axis] = 0.3
    shape = [1, 1, 1]
    shape[2 - axis] = n
    U[1 + (axis + 1) % 3] = row * x.reshape(shape)
    u, u_o = f32(U)
    lam, lam_o = f32(synth.rng(4).normal(size=(5, n, n, n)))
    v = u_o.clone().requires_grad_(True)
    (want,) = torch.autograd.grad((ohy.sweep(v, "xyz"[axis], NU, GAMMA) * lam_o).sum(), v)
    got, dnu = dh.sweep_adjoint(u, lam, axis, NU, variant=variant)
    assert torch.isfinite(got).all() and np.isfinite(float(dnu))
    t = 1 + (axis + 1) % 3
    assert rel_l2(got[t], want[t]) < 1e-5
    assert rel_l2(got, want) < 1e-5
