"""What the force evaluation holds on the device: four fields for the grid force, one for the total
potential where there is a chi, and that one shared with the whole step."""
import pytest
import torch

pytestmark = pytest.mark.gpu

N = 256
FIELD = 8 * N ** 3
SLACK = 32 << 20  # context buffers and the allocator's granularity


def held(fn):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    fn()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def test_force_workspace(gpu_lib):
    g = torch.Generator(device="cuda").manual_seed(1)
    psi, chi = (torch.randn((N,) * 3, generator=g, dtype=torch.float64, device="cuda") for _ in range(2))
    pos = torch.rand((3, 1000), generator=g, dtype=torch.float64, device="cuda")
    acc, kept = torch.empty_like(pos), psi.clone()
    ctx = gpu_lib.Context()
    run = lambda c: gpu_lib.force_interp(psi, c, -1.0, 0.2, 1.0, pos, acc=acc, ctx=ctx)  # noqa: E731
    run_small = gpu_lib.force_interp(psi[:8, :8, :8].contiguous(), None, -1.0, 0.2, 1.0, pos, ctx=ctx)  # noqa: F841
    assert held(lambda: run(None)) <= 4 * FIELD + SLACK
    assert held(lambda: run(chi)) <= FIELD + SLACK
    assert held(lambda: run(chi)) <= SLACK
    assert torch.equal(psi, kept)


def test_step_shares_the_potential(gpu_lib):
    pos = torch.rand((3, 64 ** 3), dtype=torch.float64, device="cuda")
    vel = torch.zeros_like(pos)
    chi = torch.zeros((N,) * 3, dtype=torch.float64, device="cuda")
    psi, acc = torch.zeros_like(chi), torch.empty_like(pos)
    ctx = gpu_lib.Context(precision=1, max_cycles=200)
    gpu_lib.pm_step(pos, vel, N, -0.5, 0.0, 1.0, 1e-4, 1e-6, chi, ctx=ctx)
    assert held(lambda: gpu_lib.force_interp(psi, chi, -0.5, 0.0, 1.0, pos, acc=acc, ctx=ctx)) <= SLACK
