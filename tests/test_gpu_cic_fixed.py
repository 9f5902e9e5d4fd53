"""The fixed-point CIC weights (pm.cu): the deposit bit for bit against the oracle where a weight
product can round either way, and the force at the same particles against its plain evaluation.

Positions: cell centres and faces and their neighbours in FP64 (weights 0, 1 and within one ulp of
them), the first half cell (s < 0) and the first cell (s < 1, inexact weights), dyadic fractions whose
weight products sit on exact ties of 2^-40, coordinates outside [0, 1), and random ones.
Force tolerance: 24 products and sums of 2^-53 each of the largest corner value: 1e-14 of it.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def positions(n, np_, seed):
    rng = np.random.default_rng(seed)
    e = [0.0, 0.5 / n, 1.5 / n, 1.0 / n, 0.25 / n, 1e-9, 1e-18, 1e-300, 1.0 - 0.5 / n, 1.0 - 1.0 / n, 1.0 - 2.0 ** -53]
    e += [float(np.nextafter(v, s)) for v in e[1:8] for s in (0.0, 1.0)]
    # s = i + k/2^14 per axis: products of three are odd multiples of 2^-42 .. 2^-40, ties included
    dyadic = (rng.integers(0, n, 4000) + 0.5 + rng.integers(0, 2 ** 14, 4000) * 2.0 ** -14) / n
    vals = np.concatenate([np.array(e), dyadic % 1.0, rng.random(4000), rng.random(500) * 2.0 / n])
    return np.ascontiguousarray(rng.choice(vals, size=(3, np_)))


@pytest.mark.parametrize("n,count", [(8, 5000), (32, 33333), (128, 100001), (512, 20000)])
def test_deposit_bits(gpu_lib, n, count):
    pos = positions(n, count, n)
    got = gpu_lib.pm_deposit_cic_fixed(torch.from_numpy(pos).cuda(), n).cpu().numpy()
    assert np.array_equal(got, O.deposit_cic(pos, n))
    got = gpu_lib.pm_deposit_cic(torch.from_numpy(pos).cuda(), n).cpu().numpy()
    assert np.array_equal(got, O.density(O.deposit_cic(pos, n), count))


def test_density_with_a_power_of_two_mean(gpu_lib):
    for n, count in ((16, 16 ** 3), (16, 2 * 16 ** 3), (32, 32 ** 3 // 8), (16, 1)):
        pos = positions(n, count, count)
        got = gpu_lib.pm_deposit_cic(torch.from_numpy(pos).cuda(), n).cpu().numpy()
        assert np.array_equal(got, O.density(O.deposit_cic(pos, n), count))


@pytest.mark.parametrize("n,count", [(8, 1), (16, 777), (64, 50001)])
@pytest.mark.parametrize("order", [4, 2])
def test_force(gpu_lib, n, count, order):
    rng = np.random.default_rng(n + order)
    psi, chi = rng.standard_normal((2, n, n, n))
    pos = positions(n, count, 5 * n)
    ctx = gpu_lib.Context(grad_order=order)
    got = gpu_lib.force_interp(torch.from_numpy(psi).cuda(), torch.from_numpy(chi).cuda(), -1.0, 0.2, 1.0,
                               torch.from_numpy(pos).cuda(), ctx=ctx).cpu().numpy()
    g = O.accel_grid(psi, chi, gpu_lib.coefficients(-1.0, 0.2, 1.0)["xi"], n, order=order)
    want = O.interp_cic(g, pos)
    assert np.abs(got - want).max() <= 1e-14 * np.abs(g).max()
