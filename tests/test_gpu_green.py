"""The Poisson solve's mode factor (pm.cu, k_green), one thread to the modes (+-kz, +-ky, kx): every plane
that is its own mirror, from the smallest grid up.  Tolerance: 1e-12 of max |psi|, that of the solve's
other comparison with the oracle.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16, 128])
def test_poisson_modes(gpu_lib, n):
    d = np.random.default_rng(n).standard_normal((n, n, n))
    z, y, x = np.meshgrid(*(np.arange(n),) * 3, indexing="ij")
    for kz, ky, kx in ((n // 2, 0, 0), (0, n // 2, 0), (n // 2, n // 2, n // 2), (1, n // 2, 3), (n - 1, n - 2, 0)):
        d += np.cos(2 * np.pi * (kz * z + ky * y + kx * x) / n)
    want = O.poisson_fft(d, O.coefficients(0.0, 0.2, 0.7), 0.7)
    got = gpu_lib.poisson_solve(torch.from_numpy(d).cuda(), 0.7, 0.2).cpu().numpy()
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
