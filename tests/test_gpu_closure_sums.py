"""Precision of the weight gradient's sums over voxels: the last layer's, with operands known exactly.

Zero weights and chosen biases make every hidden activation a constant and the gradient at the
output a scaled bfloat16 target, so dW = activation x sum of the gradient, in 64 bits.

Tolerance for gradients of one sign: the tensor core adds at most 32 MMAs in a row, each losing
at most 2^-23 of the partial sum, which grows linearly: 16.5 x 2^-23 = 2.0e-6, plus 3e-7 for the
rounded additions of the chains.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import lib, need_gpu

pytestmark = pytest.mark.gpu
LAYERS = ((5, 16), (16, 16), (16, 16), (16, 5))


@pytest.mark.parametrize("n,B", [(16, 1), (33, 3), (64, 2), (96, 1), (128, 1), (130, 1)])
def test_last_layer_weight_gradient(n, B):
    need_gpu()
    dh = lib()
    rng = np.random.default_rng(n)
    w = []
    for l, (ci, co) in enumerate(LAYERS):
        w += [np.zeros(27 * ci * co), rng.uniform(0.5, 2.0, co) if l < 3 else np.zeros(co)]
    c = dh.Closure(np.concatenate(w).astype(np.float32))
    c.set_norm([0.0] * 5, [1.0] * 5, [1.0] * 5)
    target = torch.from_numpy((rng.standard_normal((B, 5, n, n, n)) + 4.0).astype(np.float32)).cuda()
    _, g = c.gradient(torch.zeros_like(target), target)
    g = torch.as_tensor(np.asarray(g)).double()
    b = torch.from_numpy(w[5].astype(np.float32)).double()
    act = (0.5 * b * (1.0 + torch.erf(b / 2 ** 0.5))).to(torch.bfloat16).double()
    scale = float(np.float32(2.0) * np.float32(1.0 / (5.0 * float(n) ** 3 * B)))
    dz = ((-target) * scale).to(torch.bfloat16).double().sum((0, 2, 3, 4)).cpu()
    o = sum(27 * ci * co + co for ci, co in LAYERS[:3])
    want = (act[None, :, None] * dz).expand(27, 16, 5)
    assert ((g[o:o + 27 * 80].reshape(27, 16, 5) - want).abs() / want.abs()).max() < 2.3e-6
    assert ((g[o + 27 * 80:] - dz).abs() / dz.abs()).max() < 1e-6
    c.close()
