"""The cluster launch of the coarse inner levels (coarse_cluster.cuh) against the level-by-level
launches, over the sweep counts it loops on, and the cooperative launch that stands in for it.

The two differ in the order of FP32 sums only, inside a preconditioner: the same outer iterations to
1e-8 and fields that agree to 1e-6, the tolerance of the batched solve's other comparisons.
"""
import numpy as np
import pytest
import torch

from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu


def boxes():
    out = [(64, -0.5, 0.0), (64, -2.0, 0.5), (128, -1.0, 0.2)]
    return [torch.from_numpy(synth.lognormal_delta(n, -2.0, 1.2, 60 + k)).cuda() for k, (n, _, _) in enumerate(out)], \
        [b for _, b, _ in out], [m for _, _, m in out], [1.0] * len(out)


def solve(gpu_lib, hook=None, **params):
    ctx = gpu_lib.Context(precision=1, max_cycles=200, **params)
    if hook:
        ctx.batch_barrier_test(*hook)
    phis, infos = gpu_lib.scalar_mg_solve_batched(*boxes(), 1e-8, ctx=ctx)
    return [p.cpu().numpy() for p in phis], [i["cycles"] for i in infos]


def assert_alike(a, b):
    for p, q, i, j in zip(a[0], b[0], a[1], b[1]):
        assert abs(i - j) <= 1
        assert np.linalg.norm(p - q) <= 1e-6 * np.linalg.norm(q)


@pytest.mark.parametrize("npre,npost", [(2, 2), (1, 3), (0, 2), (3, 0)])
def test_cluster_matches_level_launches(gpu_lib, npre, npost):
    assert_alike(solve(gpu_lib, npre=npre, npost=npost, batch_persistent=1),
                 solve(gpu_lib, npre=npre, npost=npost, batch_persistent=0))


def test_cooperative_launch_matches_cluster(gpu_lib):
    # the test hook selects the cooperative launch; its barrier number is never reached
    assert_alike(solve(gpu_lib, hook=(0, 10 ** 6), batch_persistent=1), solve(gpu_lib, batch_persistent=1))
