"""The staged weight-gradient kernel (wgrad.cuh) against the FP64 reference where its work is dealt
out differently: 32^3 (rows of 32 and 16 voxels, several planes per chunk; the per-tap kernel on the
coarsest level) and 64^3 (every level on it).  Tolerances are those of the
gradient test at 16^3: BF16 activations and weights, so 10% of each layer's gradient norm.
"""
import numpy as np
import pytest
import torch

from oracle import unet as U
from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 64])
def test_weight_and_bias_gradients(gpu_lib, n):
    rng = np.random.default_rng(n)
    delta = synth.lognormal_delta(n, -2.0, 1.2, 11)
    target = delta + 0.3 * rng.standard_normal((n, n, n))
    p = U.init_params(5)
    p[-1] = 0.1
    net = gpu_lib.UNet()
    net.set_params(p)
    net.loss_grad(torch.from_numpy(delta).cuda(), torch.from_numpy(target).float().cuda(), -0.8, 0.4, 0.9)
    g = net.get_params(grads=True).astype(np.float64)
    _, want = U.loss_grad(p, delta, target, -0.8, 0.4, 0.9)
    at = 0
    for ci, co in U.CONVS:
        for size in (27 * ci * co, co):  # weights, biases
            a, b = g[at:at + size], want[at:at + size]
            at += size
            assert np.linalg.norm(a - b) <= 0.1 * np.linalg.norm(b), (ci, co, size)
