"""One outer iteration through the cluster launch of the coarse inner levels (coarse_cluster.cuh) against
the same iteration through the level-by-level launches: the corrections themselves, not what they
converge to.  The launch counts say which form ran (only the level launches have a coarsest-level kernel).

Tolerance: both evaluate the same FP32 formulas, a rounding of 2^-24 of a 32^3 level's largest terms (12 nu
u/h^2) moves its smoothest correction by up to 12 (32/2 pi)^2 2^-24 = 2e-5 of itself; 1e-4 of the
correction's norm for the few sweeps and four levels.
"""
import numpy as np
import pytest
import torch

from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu


def fields(gpu_lib, n, aB, aM):
    """A density with voids on the floor and the field two iterations into its solve."""
    delta = torch.from_numpy(synth.lognormal_delta(n, -2.0, 1.5, 90 + n)).cuda()
    guess, info = gpu_lib.scalar_mg_solve(delta, aB, aM, 1.0, 1e-8, raise_on_noconv=False,
                                          ctx=gpu_lib.Context(precision=1, max_cycles=2, autotune=0))
    return delta, guess, info["floored_cells"]


def iterate(gpu_lib, delta, guess, aB, aM, single, **params):
    ctx = gpu_lib.Context(precision=1, max_cycles=1, autotune=0, **params)
    ctx.trace_reset()
    phi = guess.clone()
    if single:
        info = gpu_lib.scalar_mg_solve(delta, aB, aM, 1.0, 1e-14, phi=phi, ctx=ctx, raise_on_noconv=False)[1]
    else:
        info = gpu_lib.scalar_mg_solve_batched([delta], [aB], [aM], [1.0], 1e-14, phis=[phi], ctx=ctx,
                                               raise_on_noconv=False)[1][0]
    assert info["cycles"] == 1 and not info["guess_rejected"]
    return (phi - guess).cpu().numpy(), ctx.trace_get()["coarsest"]["launches"]


@pytest.mark.parametrize("n", [64, 128])
@pytest.mark.parametrize("aB,aM", [(-0.5, 0.0), (-2.0, 0.5), (-1.0, 0.2)])
@pytest.mark.parametrize("params", [{}, {"npre": 1, "npost": 3}, {"npre": 0}, {"npre": 3, "npost": 0},
                                    {"inner_cycles": 2}, {"coarse_sweeps": 3}])
def test_one_iteration(gpu_lib, n, aB, aM, params):
    delta, guess, floored = fields(gpu_lib, n, aB, aM)
    assert floored > 0
    want, launches = iterate(gpu_lib, delta, guess, aB, aM, False, batch_persistent=0, **params)
    assert launches > 0
    for single in (True, False):
        got, launches = iterate(gpu_lib, delta, guess, aB, aM, single, batch_persistent=1, **params)
        if launches:
            pytest.skip("the device does not hold the cluster")
        assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
