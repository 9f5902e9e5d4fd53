"""The FP64 cell arithmetic (cell64.cuh) against the CPU oracle: every mask value, both signs of nu
and kappa, floored and unfloored cells, and the sizes at which the launch shape or kernel changes.

Tolerances: a cell is some fifty FP64 operations whose largest terms are 12 |nu| u/h^2, 100 kappa
(u/h^2)^2 and f; 200 roundings of 2^-53 of their sum bound a residual, and a sweep's value u + e
agrees to the 1e-12 of the field's largest value that the other single-sweep tests use.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("nu,kappa", [(1.1, 0.7), (-0.9, 0.6), (0.8, -0.5), (1.0, 0.0)])
@pytest.mark.parametrize("masked", [False, True])
def test_fp64_sweep_and_residual_cells(gpu_lib, n, nu, kappa, masked):
    import torch

    rng = np.random.default_rng(n + masked)
    u = rng.standard_normal((n, n, n)) / n ** 2
    f = 3.0 * rng.standard_normal((n, n, n))
    km = rng.integers(0, 10, size=(n, n, n)).astype(np.uint8) if masked else None  # 8 and 9: no screening
    ut, ft = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    kt = torch.from_numpy(km).cuda() if masked else None
    r, fl = (x.cpu().numpy() for x in gpu_lib.pm_mg_residual(ut, ft, 0.25, nu, kappa, 0.35, kmask=kt))
    want, want_fl = O.residual(u, f, 0.25, nu, kappa, 0.35, kmask=km)
    same = fl == want_fl
    assert np.mean(~same) < 1e-4  # a discriminant may round across the floor
    scale = np.abs(u).max() * n * n
    term = 12.0 * abs(nu) * scale + 100.0 * abs(kappa) * scale ** 2 + np.abs(f).max()
    assert np.abs(r - want)[same].max() <= 200 * 2.0 ** -53 * term
    got = gpu_lib.pm_mg_sweep(ut, ft, 0.25, nu, kappa, 0.35, kmask=kt).cpu().numpy()
    want = O.smooth_sweep(u, f, 0.25, nu, kappa, 0.35, kmask=km)
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
