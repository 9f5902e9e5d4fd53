"""The float-float conversions on the integer pipe, through a solve that performs none or few outer
iterations: with max_cycles = 0 a mixed solve returns its guess converted to float pairs and back,
less its mean.

Tolerance: a float pair holds 48 bits and more, the mean is removed twice in FP64: 2^-47 of the field's
largest value.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16, 64])
@pytest.mark.parametrize("kind", ["zero", "ordinary", "ties"])
def test_guess_survives_the_conversion(gpu_lib, n, kind):
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, n, n))
    if kind == "zero":
        x[:] = 0.0
    if kind == "ties":  # mantissas at and beside the middle between two floats, and at a carry
        m = rng.integers(2 ** 23, 2 ** 24, x.shape).astype(np.float64)
        x = np.where(x > 0, 1.0, -1.0) * (m + 0.5 + rng.integers(-1, 2, x.shape) * 2.0 ** -29) * 2.0 ** -24
        x.flat[::7] = 1.0 - 2.0 ** -25
    guess = torch.from_numpy(x * 1e-3 / n ** 2).cuda()
    delta = torch.from_numpy(rng.standard_normal((n, n, n)) * 1e3).cuda()
    want = guess.cpu().numpy()
    want = want - want.mean()
    ctx = gpu_lib.Context(precision=1, max_cycles=0)
    phi, info = gpu_lib.scalar_mg_solve(delta, -0.5, 0.0, 1.0, 1e-8, phi=guess, ctx=ctx, raise_on_noconv=False)
    assert not info["guess_rejected"]
    assert np.abs(phi.cpu().numpy() - want).max() <= 2.0 ** -47 * np.abs(want).max()
