"""The batched solve's device flags and tables are in place before the boxes' streams read them: a
context whose flags were left down by an earlier call (every box converged) gives the bits and the
iteration counts of a fresh one, call after call, for the cluster and for the cooperative launch.

No tolerance: the reductions have a fixed order and the kernel variants are fixed (autotune = 0).
"""
import pytest
import torch

from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu

EFT = [(64, -0.5, 0.0), (64, -2.0, 0.5), (64, -1.0, 0.2), (128, -0.5, 0.0)]


def solve(gpu_lib, ctx, deltas):
    phis, infos = gpu_lib.scalar_mg_solve_batched(deltas, [b for _, b, _ in EFT], [m for _, _, m in EFT],
                                                  [1.0] * len(EFT), 1e-8, ctx=ctx)
    return phis, [i["cycles"] for i in infos]


def context(gpu_lib, cooperative):
    ctx = gpu_lib.Context(precision=1, max_cycles=200, autotune=0)
    if cooperative:  # the test hook selects that launch; its barrier number is never reached
        ctx.batch_barrier_test(0, 10 ** 6)
    return ctx


@pytest.mark.parametrize("cooperative", [False, True])
def test_later_calls_match_a_fresh_context(gpu_lib, cooperative):
    deltas = [torch.from_numpy(synth.lognormal_delta(n, -2.0, 1.2, 80 + k)).cuda() for k, (n, _, _) in enumerate(EFT)]
    want, cycles = solve(gpu_lib, context(gpu_lib, cooperative), deltas)
    assert min(cycles) > 1  # the graph launches, which lower the flags, ran
    ctx = context(gpu_lib, cooperative)
    for _ in range(6):
        got, c = solve(gpu_lib, ctx, deltas)
        assert c == cycles
        assert all(torch.equal(a, b) for a, b in zip(got, want))
