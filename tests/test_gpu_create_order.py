"""A context or a network that is made on a stream of its own is cleared before its handle is out, also
while the legacy stream, on which the clears run, is busy (here for about 0.1 s): the first calls give
the bits of an ordinary context's."""
import numpy as np
import pytest
import torch

from oracle import unet as U
from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu


def first_calls(gpu_lib):
    n = 16
    delta = torch.from_numpy(synth.lognormal_delta(n, -2.0, 1.2, 3)).cuda()
    pos = torch.from_numpy(np.random.default_rng(3).random((3, 5000))).cuda()
    torch.cuda.synchronize()
    return n, delta, pos


def calls(gpu_lib, ctx, n, delta, pos):
    with torch.cuda.stream(ctx.stream):
        rho = gpu_lib.pm_deposit_cic(pos, n, ctx=ctx)
        chi, info = gpu_lib.scalar_mg_solve(delta, -0.5, 0.0, 1.0, 1e-8, ctx=ctx)
        net = gpu_lib.UNet(ctx)
        net.set_params(U.init_params(2))
        loss = net.loss_grad(delta, delta.float(), -0.5, 0.0, 1.0)
        grads = net.get_params(grads=True)
    ctx.stream.synchronize()
    return rho.cpu(), chi.cpu(), info["cycles"], loss, torch.from_numpy(np.asarray(grads).copy())


def test_first_calls_on_a_side_stream(gpu_lib):
    n, delta, pos = first_calls(gpu_lib)
    want = calls(gpu_lib, gpu_lib.Context(precision=1, autotune=0), n, delta, pos)
    for _ in range(3):
        side = torch.cuda.Stream()
        torch.cuda._sleep(200_000_000)  # on the default stream
        got = calls(gpu_lib, gpu_lib.Context(precision=1, autotune=0, stream=side), n, delta, pos)
        for a, b in zip(got, want):
            assert torch.equal(a, b) if isinstance(a, torch.Tensor) else a == b
