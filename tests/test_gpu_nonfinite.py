"""NaN, infinities and signed zeros where values are compared or converted by their bits: the FP64 cells
(cell64.cuh) against the CPU oracle, whose comparisons are C's, and the float-float conversions
(outer_ff.cuh, internal.cuh) through solves.

Cells: non-finite exactly where the oracle's are; finite values by the bounds of
test_gpu_fp64_cells.py (200 roundings of the largest terms; 1e-12 for a sweep).
Conversions of values outside 2^+-70: 2^-47 of the largest, as in test_gpu_ff_bits.py.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

BAD = {"nan": np.nan, "-nan": np.copysign(np.nan, -1.0), "inf": np.inf, "-inf": -np.inf}


@pytest.mark.parametrize("n", [8, 64])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("where", ["source", "field"])
@pytest.mark.parametrize("bad", sorted(BAD))
@pytest.mark.parametrize("nu,kappa", [(1.1, 0.7), (-0.9, 0.6), (1.0, 0.0)])
def test_fp64_cells(gpu_lib, n, masked, where, bad, nu, kappa):
    rng = np.random.default_rng(n + masked)
    u = rng.standard_normal((n, n, n)) / n ** 2
    f = 3.0 * rng.standard_normal((n, n, n))
    scale = np.abs(u).max() * n * n
    term = 12.0 * abs(nu) * scale + 100.0 * abs(kappa) * scale ** 2 + np.abs(f).max()
    (f if where == "source" else u)[3, 5, n - 1] = BAD[bad]
    km = rng.integers(0, 10, size=(n, n, n)).astype(np.uint8) if masked else None
    ut, ft = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    kt = torch.from_numpy(km).cuda() if masked else None
    r, fl = (x.cpu().numpy() for x in gpu_lib.pm_mg_residual(ut, ft, 0.25, nu, kappa, 0.35, kmask=kt))
    want, want_fl = O.residual(u, f, 0.25, nu, kappa, 0.35, kmask=km)
    ok = np.isfinite(want)
    assert not ok.all() or bad in ("inf", "-inf")  # an infinite source may floor its cell, a NaN may not
    assert np.array_equal(np.isfinite(r), ok)
    assert np.array_equal(fl[~ok], want_fl[~ok])
    same = ok & (fl == want_fl)
    assert np.mean(fl != want_fl) < 1e-4
    assert np.abs(r - want)[same].max() <= 200 * 2.0 ** -53 * term
    got = gpu_lib.pm_mg_sweep(ut, ft, 0.25, nu, kappa, 0.35, kmask=kt).cpu().numpy()
    want = O.smooth_sweep(u, f, 0.25, nu, kappa, 0.35, kmask=km)
    ok = np.isfinite(want)
    assert np.array_equal(np.isfinite(got), ok)
    assert np.abs(got - want)[ok].max() <= 1e-12 * np.abs(want[ok]).max()


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_fp64_double_root_at_zero(gpu_lib, sign):
    """eta = 0 and a cell whose dN/dc and residual are both zero: the update is zero (of the two forms of
    the root, the one that divides by dN/dc would be 0/0).  Exact in binary: one cell of -1/512 on 8^3."""
    n = 8
    u = np.zeros((n, n, n))
    u[2, 2, 2] = -1.0 / 512.0
    nu = kappa = sign
    f = np.full((n, n, n), sign * 0.375)  # nu L - kappa q2 at that cell
    got = gpu_lib.pm_mg_sweep(torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda(), 0.0, nu, kappa, 0.0).cpu().numpy()
    want = O.smooth_sweep(u, f, 0.0, nu, kappa, 0.0)
    assert want[2, 2, 2] == u[2, 2, 2] == got[2, 2, 2]
    assert np.isfinite(got).all()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", [16, 64])
@pytest.mark.parametrize("bad", ["nan", "-nan", "inf"])  # a source of -infinity is a floored cell
def test_solve_reports_a_bad_source(gpu_lib, precision, n, bad):
    d = np.random.default_rng(n).standard_normal((n, n, n))
    d[1, 2, 3] = BAD[bad]
    with pytest.raises(gpu_lib.PMError) as e:
        gpu_lib.scalar_mg_solve(torch.from_numpy(d).cuda(), -0.5, 0.0, 1.0, 1e-8,
                                ctx=gpu_lib.Context(precision=precision, autotune=0))
    assert e.value.status == gpu_lib.PM_ERR_NONFINITE


@pytest.mark.parametrize("bad", sorted(BAD))
def test_bad_guess_is_dropped(gpu_lib, bad):
    n = 32
    d = torch.from_numpy(np.random.default_rng(1).standard_normal((n, n, n))).cuda()
    guess = torch.zeros_like(d)
    guess[4, 5, 6] = BAD[bad]
    ctx = gpu_lib.Context(precision=1, autotune=0)
    phi, info = gpu_lib.scalar_mg_solve(d, -0.5, 0.0, 1.0, 1e-8, phi=guess, ctx=ctx)
    want, _ = gpu_lib.scalar_mg_solve(d, -0.5, 0.0, 1.0, 1e-8, ctx=ctx)
    assert info["guess_rejected"] and torch.equal(phi, want)


@pytest.mark.parametrize("n", [8, 64])
def test_small_guess_survives_the_conversion(gpu_lib, n):
    # 2^-71 and below: outside the range of the integer conversion, well inside a float pair's
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, n, n)) * 2.0 ** -74
    guess = torch.from_numpy(x).cuda()
    delta = torch.from_numpy(rng.standard_normal((n, n, n))).cuda()
    phi, info = gpu_lib.scalar_mg_solve(delta, -0.5, 0.0, 1.0, 1e-8, phi=guess, raise_on_noconv=False,
                                        ctx=gpu_lib.Context(precision=1, max_cycles=0))
    want = x - x.mean()
    assert not info["guess_rejected"]
    assert np.abs(phi.cpu().numpy() - want).max() <= 2.0 ** -47 * np.abs(want).max()
