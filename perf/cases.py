"""Workloads of the particle-mesh library, as a user's program runs them through its public API.

Each case is one call (or one training step) of the path: the CIC deposit, the Poisson solve,
the force at the particles, the scalar-field solve in FP64 and in mixed precision, a batched
solve, a whole PM step, the learned start and its training step.  ``listed()`` names them,
``draw(rng)`` gives others of the same ranges, ``prepare`` makes seeded inputs on the GPU and
``run`` makes one pass.  ``exact`` evaluates the same quantities in 64 bits with plain torch.
"""
import math
import time

import numpy as np
import torch

from paper_2604_15434_gb300 import api, learned

TOL = 1e-8  # the benchmark's relative residual
PI2 = 2.0 * math.pi
# U-Net convolutions (inputs, outputs, level); the first one's 16 inputs hold 4 real channels
CONVS = [(16, 16, 0), (16, 16, 0), (16, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2), (96, 32, 1), (32, 32, 1),
         (48, 16, 0), (16, 16, 0)]


def listed():
    return [
        # the smallest call: a test-sized box (32^3 particles on 32^3 cells), launch latency
        {"name": "deposit_32", "kind": "deposit", "n": 32, "np": 32 ** 3, "sigma": 1.0, "shuffled": False},
        # the deposit of the 256^3 particle-mesh configuration, particles in lattice order
        {"name": "deposit_256", "kind": "deposit", "n": 256, "np": 256 ** 3, "sigma": 2.0, "shuffled": False},
        # its force evaluation: gradient of the total potential, interpolated to 256^3 particles
        {"name": "force_256", "kind": "force", "n": 256, "np": 256 ** 3, "sigma": 2.0, "shuffled": False},
        # its standard Poisson solve
        {"name": "poisson_256", "kind": "poisson", "n": 256},
        # the scalar field of the 32^3 configuration in FP64, the library's default precision
        {"name": "solve_fp64_32", "kind": "solve", "n": 32, "precision": 0, "aB": -0.5, "aM": 0.0, "a": 1.0,
         "sigma": 1.0},
        # an FP64 solve at an ordinary size, half the box on the void floor
        {"name": "solve_fp64_128", "kind": "solve", "n": 128, "precision": 0, "aB": -2.0, "aM": 0.5, "a": 1.0,
         "sigma": 1.5},
        # the mixed-precision solve at an ordinary size
        {"name": "solve_mixed_128", "kind": "solve", "n": 128, "precision": 1, "aB": -2.0, "aM": 0.5, "a": 1.0,
         "sigma": 1.5},
        # the benchmark's mesh: one mixed-precision solve of the 512^3 lognormal box, cold start
        {"name": "solve_mixed_512", "kind": "solve", "n": 512, "precision": 1, "aB": -0.5, "aM": 0.0, "a": 1.0,
         "sigma": 1.5},
        # a parameter study: 24 boxes of 64^3, 128^3 and 256^3 with their own parameters in one call
        {"name": "batch_24", "kind": "batch", "boxes": 24, "largest": 256, "pick": 1007},
        # one whole PM step of the 256^3 configuration
        {"name": "pm_step_256", "kind": "step", "n": 256, "np": 256 ** 3, "aB": -1.0, "aM": 0.2, "a": 1.0,
         "sigma": 2.0},
        # the learned initial guess of a 256^3 box (network and FFT)
        {"name": "warm_start_256", "kind": "warm", "n": 256, "aB": -0.5, "aM": 0.0, "a": 1.0, "sigma": 1.5},
        # one training step of the network at the resolution it is trained at
        {"name": "train_128", "kind": "train", "n": 128, "aB": -1.0, "aM": 0.2, "a": 1.0, "sigma": 1.5},
    ]


def _coef(aB0, aM0, a, om=0.3):
    """nu, xi, kappa, the chi source factor and the Poisson factor at scale factor a."""
    oma = om / (om + (1.0 - om) * a ** 3)
    aB, aM = aB0 * (1.0 - oma) / (1.0 - om), aM0 * (1.0 - oma) / (1.0 - om)
    geff = oma ** (aM0 / (3.0 * (1.0 - om)))
    c2 = -aM + aB * (1.0 + aM) - 1.5 * oma * (1.0 + aB) + 3.0 * aB * oma + 1.5 * oma * geff
    e2 = om / a ** 3 + 1.0 - om
    xi, pois = aB - aM, 1.5 * geff * a * om
    return {"nu": -c2 + aB * (2.0 * aM - aB), "xi": xi, "kappa": (-4.0 * aB + 2.0 * aM) / (4.0 * e2 * a ** 4),
            "src": xi * pois, "pois": pois}


def _params(rng):
    """EFT parameters of the sampled boxes: near-singular draws are drawn again."""
    while True:
        aB, aM, a = rng.uniform(-2.0, 0.0), rng.uniform(0.0, 1.0), rng.uniform(0.3, 1.0)
        c = _coef(aB, aM, a)
        if abs(c["nu"]) >= 0.1 and abs(c["xi"] / c["nu"]) <= 4.0:
            return {"aB": aB, "aM": aM, "a": a}


def _particles(rng, n):
    """A particle count for a mesh of n cells a side: from an eighth to twice the cells, any number."""
    return max(1, min(256 ** 3, int(n ** 3 * 2.0 ** rng.uniform(-3.0, 1.0))))


def draw(rng):
    kind = rng.choice(["deposit", "force", "poisson", "solve", "solve", "batch", "step", "warm", "train"])
    if kind in ("deposit", "force"):
        n = rng.choice([16, 32, 64, 128, 256])
        return {"kind": kind, "n": n, "np": _particles(rng, n), "sigma": rng.uniform(0.5, 2.0),
                "shuffled": rng.random() < 0.3}
    if kind == "poisson":  # the time-independent factor varies with the parameters
        return {"kind": kind, "n": rng.choice([16, 32, 64, 128, 256]), **_params(rng)}
    if kind == "solve":
        precision = rng.choice([0, 1])
        return {"kind": kind, "n": rng.choice([16, 32, 64, 128] if precision == 0 else [16, 32, 64, 128, 256]),
                "precision": precision, "sigma": rng.uniform(1.0, 1.5), **_params(rng)}
    if kind == "batch":
        return {"kind": kind, "boxes": rng.randint(2, 24), "largest": rng.choice([64, 128]),
                "pick": rng.randrange(1 << 20)}
    if kind == "step":
        n = rng.choice([32, 64, 128, 256])
        return {"kind": kind, "n": n, "np": _particles(rng, n), "sigma": rng.uniform(0.5, 2.0), **_params(rng)}
    n = rng.choice([32, 64, 128, 256]) if kind == "warm" else rng.choice([32, 64, 128])
    return {"kind": kind, "n": n, "sigma": rng.uniform(1.0, 1.5), **_params(rng)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _k(n):
    m = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n
    r = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64) * n
    return r[None, None, :], m[None, :, None], m[:, None, None]


def _gaussian(n, slope, sigma, gen):
    """Zero-mean Gaussian field, P(k) ~ k^slope, standard deviation sigma."""
    w = torch.randn((n, n, n), generator=gen, device="cuda", dtype=torch.float64)
    kx, ky, kz = _k(n)
    k2 = kx ** 2 + ky ** 2 + kz ** 2
    k2[0, 0, 0] = 1.0
    wk = torch.fft.rfftn(w) * k2 ** (slope / 4.0)
    wk[0, 0, 0] = 0.0
    g = torch.fft.irfftn(wk, s=(n, n, n))
    return g * (sigma / g.std())


def _lognormal(n, sigma, gen):
    rho = torch.exp(_gaussian(n, -2.0, sigma, gen))
    return rho / rho.mean() - 1.0


def _zeldovich(count, sigma, gen, shuffled=False):
    """`count` particles (3, count): a displaced lattice, in lattice order or shuffled; where the
    lattice has more sites than that, a random subset of them."""
    m = max(2, math.ceil(round(count ** (1.0 / 3.0), 9)))
    while m ** 3 < count:
        m += 1
    dk = torch.fft.rfftn(_gaussian(m, -1.5, sigma, gen))
    ks = _k(m)
    k2 = PI2 ** 2 * (ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2)
    k2[0, 0, 0] = 1.0
    q = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m
    pos = torch.empty((3, m ** 3), device="cuda", dtype=torch.float64)
    for row, shape in enumerate(((1, 1, m), (1, m, 1), (m, 1, 1))):
        x = (torch.fft.irfftn(1j * PI2 * ks[row] * dk / k2, s=(m, m, m)) + q.reshape(shape)).reshape(-1)
        x = x - torch.floor(x)
        pos[row] = torch.where(x >= 1.0, torch.zeros_like(x), x)
    if count < m ** 3 or shuffled:
        keep = torch.randperm(m ** 3, generator=gen, device="cuda")[:count]
        pos = pos[:, keep if shuffled else keep.sort().values].contiguous()
    return pos


def _weights(seed):
    """He-normal convolution weights, small biases, a head near the channel average."""
    rng = np.random.default_rng(seed)
    parts = []
    for i, (ci, co, _) in enumerate(CONVS):
        parts += [rng.standard_normal(27 * ci * co) * math.sqrt(2.0 / (27 * (4 if i == 0 else ci))),
                  0.01 * rng.standard_normal(co)]
    parts += [0.25 * rng.standard_normal(16), [0.0]]
    return np.concatenate(parts).astype(np.float32)


def _trained():
    return learned.load_params(learned.WEIGHTS_DIR + "/unet_128")


def _boxes(case):
    """Sizes and parameters of a batch, from the case's own numbers."""
    sizes = [s for s in (64, 128, 256) if s <= case["largest"]]
    pick = np.random.default_rng(case["pick"]).integers(0, len(sizes), size=case["boxes"])
    rng = np.random.default_rng(case["pick"])
    return [(sizes[i], _params(rng)) for i in pick]


_ctx = {}


def _context(**params):
    """A program keeps one context (scratch, plans, tuned variants) for all its inputs."""
    key = tuple(sorted(params.items()))
    if key not in _ctx:
        _ctx[key] = api.Context(**params)
    return _ctx[key]


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = {"case": case}
    if kind == "deposit":
        s["ctx"] = _context()
        s["pos"] = _zeldovich(case["np"], case["sigma"], g, case["shuffled"])
    elif kind == "force":
        s["ctx"] = _context()
        s["pos"] = _zeldovich(case["np"], case["sigma"], g, case["shuffled"])
        # potentials: smooth fields of a lognormal source's spectrum (P ~ k^-2 over k^4)
        s["psi"] = _gaussian(case["n"], -6.0, 0.05, g)
        s["chi"] = _gaussian(case["n"], -6.0, 0.05, g)
    elif kind == "poisson":
        s["ctx"] = _context()
        s["delta"] = _lognormal(case["n"], 1.5, g)
    elif kind == "solve":
        s["ctx"] = _context(precision=case["precision"], max_cycles=200)
        s["delta"] = _lognormal(case["n"], case["sigma"], g)
    elif kind == "batch":
        s["ctx"] = _context(precision=1, max_cycles=200)
        s["params"] = [p for _, p in _boxes(case)]
        s["deltas"] = []
        for b, (n, _) in enumerate(_boxes(case)):  # alternately lognormal and linear (clipped) sources
            d = _lognormal(n, 1.0, g) if b % 2 == 0 else _gaussian(n, -1.5, 1.0, g).clamp(min=-1.0)
            s["deltas"].append((d - d.mean()).contiguous())
    elif kind == "step":
        s["ctx"] = _context(precision=1, max_cycles=200)
        s["pos"] = _zeldovich(case["np"], case["sigma"], g)
        s["vel"] = 0.01 * torch.randn(s["pos"].shape, generator=g, device="cuda", dtype=torch.float64)
    elif kind == "warm":
        s["net"] = api.UNet(_context())
        s["net"].set_params(_trained())
        s["delta"] = _lognormal(case["n"], case["sigma"], g)
    else:
        s["net"] = api.UNet(_context())
        s["net"].set_params(_weights(seed))
        s["delta"], s["target"] = _training_pair(case, g)
    return s


def _training_pair(case, g):
    d = _lognormal(case["n"], case["sigma"], g)
    return d, (d / (1.0 + 0.1 * d.abs())).float()  # screened where the source is strong


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "deposit":
        return api.pm_deposit_cic(s["pos"], c["n"], ctx=s["ctx"])
    if kind == "force":
        return api.force_interp(s["psi"], s["chi"], -1.0, 0.2, 1.0, s["pos"], ctx=s["ctx"])
    if kind == "poisson":
        return api.poisson_solve(s["delta"], c.get("a", 1.0), c.get("aM", 0.2), ctx=s["ctx"])
    if kind == "solve":
        return api.scalar_mg_solve(s["delta"], c["aB"], c["aM"], c["a"], TOL, ctx=s["ctx"])[0]
    if kind == "batch":
        p = s["params"]
        return api.scalar_mg_solve_batched(s["deltas"], [q["aB"] for q in p], [q["aM"] for q in p],
                                           [q["a"] for q in p], TOL, ctx=s["ctx"])[0]
    if kind == "step":
        # a cold first step from a snapshot that the program keeps
        pos, vel = s["pos"].clone(), s["vel"].clone()
        chi = torch.zeros((c["n"],) * 3, dtype=torch.float64, device="cuda")
        api.pm_step(pos, vel, c["n"], c["aB"], c["aM"], c["a"], 1e-3, TOL, chi, ctx=s["ctx"])
        return {"pos": pos, "vel": vel, "chi": chi}
    if kind == "warm":
        return s["net"].warm_start(s["delta"], c["aB"], c["aM"], c["a"])
    loss = s["net"].loss_grad(s["delta"], s["target"], c["aB"], c["aM"], c["a"])
    grads = s["net"].get_params(grads=True)
    s["net"].adam_step(1e-4)
    return {"loss": loss, "grads": grads, "weights": s["net"].get_params()}


def work(case):
    """Bytes and operations of one pass that any implementation needs."""
    kind = case["kind"]
    if kind == "batch":
        cells = sum(n ** 3 for n, _ in _boxes(case))
        return {"bytes": 16 * cells, "flops": 60 * cells}
    cells = case["n"] ** 3
    if kind == "deposit":  # positions in, density out
        return {"bytes": 24 * case["np"] + 8 * cells, "flops": 40 * case["np"]}
    if kind == "force":  # two potentials and the positions in, the force out
        return {"bytes": 16 * cells + 48 * case["np"], "flops": 24 * cells + 70 * case["np"]}
    fft = 5.0 * cells * math.log2(cells)  # a real transform there and back
    if kind == "poisson":
        return {"bytes": 16 * cells, "flops": fft}
    if kind == "solve":  # source in, field out; at least one evaluation of the operator
        return {"bytes": 16 * cells, "flops": 60 * cells}
    if kind == "step":
        return {"bytes": 96 * case["np"] + 16 * cells, "flops": fft + 84 * cells + 120 * case["np"]}
    conv = sum(54.0 * (4 if i == 0 else ci) * co * cells / 8 ** lv for i, (ci, co, lv) in enumerate(CONVS))
    if kind == "warm":
        return {"bytes": 16 * cells, "flops": conv + fft}
    return {"bytes": 12 * cells, "flops": 3.0 * conv}


# ------------------------------------------------------------------ 64-bit references

def _cic(pos, n):
    """Cell index and weight of the 8 cloud-in-cell corners of every particle."""
    s = pos * n - 0.5
    i = torch.floor(s)
    d = s - i
    i = i.long()
    for c in range(8):
        b = [c & 1, (c >> 1) & 1, (c >> 2) & 1]
        w = torch.ones_like(d[0])
        for ax in range(3):
            w = w * (d[ax] if b[ax] else 1.0 - d[ax])
        x, y, z = [(i[ax] + b[ax]) % n for ax in range(3)]
        yield (z * n + y) * n + x, w


def _exact_density(pos, n):
    acc = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    for cell, w in _cic(pos, n):
        acc.index_add_(0, cell, w)
    return acc.reshape(n, n, n) * (n ** 3 / pos.shape[1]) - 1.0


def _inverse_laplacian(f):
    """Zero-mean u with the 7-point Laplacian of u equal to f - <f> (box of side 1)."""
    n = f.shape[0]
    kx, ky, kz = _k(n)
    lam = -4.0 * n * n * (torch.sin(math.pi * kx / n) ** 2 + torch.sin(math.pi * ky / n) ** 2 +
                          torch.sin(math.pi * kz / n) ** 2)
    lam[0, 0, 0] = 1.0
    fk = torch.fft.rfftn(f) / lam
    fk[0, 0, 0] = 0.0
    return torch.fft.irfftn(fk, s=(n, n, n))


def _exact_force(psi, pos):
    n = psi.shape[0]
    out = []
    for ax in (2, 1, 0):
        r = lambda k: torch.roll(psi, -k, ax)  # noqa: E731
        g = -(8.0 * (r(1) - r(-1)) - (r(2) - r(-2))) * (n / 12.0)
        a = torch.zeros_like(pos[0])
        for cell, w in _cic(pos, n):
            a += w * g.reshape(-1)[cell]
        out.append(a)
    return torch.stack(out)


def _exact_chi(delta, c, eta=0.35, limit_s=12.0):
    """The discrete field by red-black sweeps alone; None where that takes too long."""
    n, nu, kap = delta.shape[0], c["nu"], c["kappa"]
    f = c["src"] * delta
    fnorm = (f - f.mean()).norm()
    i2, sp, q = float(n * n), -1.0 if nu >= 0.0 else 1.0, torch.arange(n, device="cuda")
    red = ((q[:, None, None] + q[None, :, None] + q[None, None, :]) & 1) == 0
    df, lsat, p = (eta * 6.0 * abs(nu) * i2) ** 2, 0.75 * nu * (1.0 - eta) / kap, -24.0 * kap * i2 * i2
    chi, lam, began = torch.zeros_like(f), 0.0, time.monotonic()

    def local():
        d = [torch.roll(chi, -1, ax) + torch.roll(chi, 1, ax) - 2.0 * chi for ax in range(3)]
        e = []
        for a, b in ((0, 1), (0, 2), (1, 2)):
            r = torch.roll(chi, -1, a) - torch.roll(chi, 1, a)
            e.append(torch.roll(r, -1, b) - torch.roll(r, 1, b))
        lap = (d[0] + d[1] + d[2]) * i2
        q2 = (2.0 * (d[0] * d[1] + d[1] * d[2] + d[2] * d[0]) - 0.125 * (e[0] ** 2 + e[1] ** 2 + e[2] ** 2)) * i2 * i2
        g = nu * lap - kap * q2 - f - lam
        ep = (-6.0 * nu + 8.0 * kap * lap) * i2
        return lap, g, ep, ep * ep - 4.0 * p * g

    for sweep in range(40000):
        for colour in (red, ~red):
            lap, g, ep, disc = local()
            sq = sp * disc.clamp(min=0.0).sqrt()
            root = torch.where(ep * sp > 0.0, -2.0 * g / (ep + sq), (sq - ep) / (2.0 * p))
            e = torch.where(disc < df, (lap - lsat) / (6.0 * i2), root)
            chi = torch.where(colour, chi + e, chi)
        if sweep % 20 == 19:
            chi = chi - chi.mean()
            lap, g, ep, disc = local()
            low = disc < df
            r = torch.where(low, nu * (lsat - lap), -g)
            gm = float(r.sum() / (~low).sum())
            lam -= gm
            if float(torch.where(low, r, r - gm).norm() / fnorm) < 1e-12:
                return chi
            if time.monotonic() - began > limit_s:
                return None
    return None


def _exact_net(flat, delta, c):
    """The network's output in 64 bits for flat parameters (a 64-bit tensor)."""
    n = delta.shape[0]
    at = 0

    def take(k):
        nonlocal at
        at += k
        return flat[at - k:at]

    def conv(x, i):  # x: (channels, n, n, n), periodic
        ci, co, _ = CONVS[i]
        w = take(27 * ci * co).reshape(27, ci, co)
        b = take(co)
        w = w.permute(2, 1, 0).reshape(co, ci, 3, 3, 3)[:, :x.shape[0]]
        y = b.reshape(co, 1, 1, 1)
        for t in range(27):
            s = torch.roll(x, (1 - t // 9, 1 - (t // 3) % 3, 1 - t % 3), (1, 2, 3))
            y = y + torch.einsum("oi,izyx->ozyx", w[:, :, t // 9, (t // 3) % 3, t % 3], s)
        return torch.relu(y)

    def pool(x):
        m = x.shape[1] // 2
        return x.reshape(x.shape[0], m, 2, m, 2, m, 2).mean((2, 4, 6))

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    one = torch.ones_like(delta)
    x = conv(torch.stack([torch.asinh(delta), c["aB"] * one, c["aM"] * one, c["a"] * one]), 0)
    s1 = conv(x, 1)
    s2 = conv(conv(pool(s1), 2), 3)
    x = conv(conv(pool(s2), 4), 5)
    x = conv(conv(torch.cat([up(x), s2]), 6), 7)
    x = conv(conv(torch.cat([up(x), s1]), 8), 9)
    w = take(17)
    return torch.einsum("c,czyx->zyx", w[:16], x) + w[16]


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "batch" or (kind in ("solve", "step") and n > 32):
        return None  # a nonlinear solve by plain sweeps takes minutes there
    s = prepare(case, seed)
    c = _coef(case.get("aB", -1.0), case.get("aM", 0.2), case.get("a", 1.0))
    if kind == "deposit":
        return _exact_density(s["pos"], n)
    if kind == "force":
        return _exact_force(s["psi"] + c["xi"] * s["chi"], s["pos"])
    if kind == "poisson":
        return _inverse_laplacian(c["pois"] * s["delta"])
    if kind == "solve":
        return _exact_chi(s["delta"], c)
    if kind == "step":
        d = _exact_density(s["pos"], n)
        chi = _exact_chi(d, c)
        if chi is None:
            return None
        v = s["vel"] + 1e-3 * _exact_force(_inverse_laplacian(c["pois"] * d) + c["xi"] * chi, s["pos"])
        x = s["pos"] + 1e-3 * v
        return {"pos": x - torch.floor(x), "vel": v, "chi": chi}
    if kind == "warm":
        flat = torch.from_numpy(_trained().astype(np.float64)).cuda()
        return _inverse_laplacian((c["src"] / c["nu"]) * _exact_net(flat, s["delta"], case))
    flat = torch.from_numpy(_weights(seed).astype(np.float64)).cuda().requires_grad_(True)
    loss = ((_exact_net(flat, s["delta"], case) - s["target"].double()) ** 2).mean()
    loss.backward()
    g = flat.grad
    # Adam's first step: both moments are bias-corrected to the gradient itself
    w = flat.detach() - 1e-4 * g / (g.abs() + 1e-8)
    return {"loss": float(loss), "grads": g.cpu().numpy(), "weights": w.cpu().numpy()}
