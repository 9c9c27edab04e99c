"""Weight gradient of the closure at the edges of its line tiles and x segments.

A field tiled twice along every axis has the same training gradient as the field itself:
every voxel's network input, output and target repeat, and the loss is a mean over voxels.
The factor 1/8 of the per-voxel loss weight is a power of two, so every bfloat16 rounding
agrees and only the order of the float32 sums differs: each accumulator takes up to a few
thousand sequential additions, an error of about 6e-8 x sqrt(4000) = 4e-6 of its value, and
the bar is 1e-4. The grids cover one line tile and several (6 lines each, full and ragged),
line lengths that are multiples of 16 and not, one x segment and two (from 129 cells on).
The smallest grids are pinned to the oracle's float64 gradient in test_gpu_closure.py.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import f32, lib, need_gpu, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dh():
    need_gpu()
    return lib()


def closure(dh, seed):
    from paper_2502_02294_gb300._lib import CLOSURE_NWEIGHTS
    w = 0.05 * np.random.default_rng(seed).standard_normal(CLOSURE_NWEIGHTS).astype(np.float32)
    c = dh.Closure(w)
    c.set_norm([0.16, 0, 0, 0, 1e-3], [0.05, 0.01, 0.01, 0.01, 1e-3],
               [0.01, 0.002, 0.002, 0.002, 0.003])
    return c


@pytest.mark.parametrize("n", [2, 3, 8, 9, 18, 36, 64, 65, 72])
def test_gradient_of_a_tiled_field(dh, n):
    gas, _ = f32(synth.gas_state(n, 5))
    tgt, _ = f32(synth.gas_state(n, 6))
    c = closure(dh, 7)
    loss, g = c.gradient(gas, tgt)
    loss2, g2 = c.gradient(gas.repeat(1, 2, 2, 2).contiguous(), tgt.repeat(1, 2, 2, 2).contiguous())
    c.status()
    c.close()
    assert np.isfinite(g).all()
    assert abs(loss - loss2) <= 1e-5 * abs(loss)
    assert rel_l2(g2, g) < 1e-4
