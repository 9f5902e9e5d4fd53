"""The weight and bias gradients against an FP64 contraction of the very operands they are formed from,
where the work is dealt out differently: all taps or one z tap per block, 16 or 32 outputs, rows of 16 to
128 voxels, chunks that begin in the middle of a plane (128^3), several x segments (256^3).

Layers 7 to 9 pass values through (one-hot centre taps), so that every activation can be read through the
head and every gradient down to layer 6's output follows from the loss with the roundings that the kernels
make.  Gradients in all voxels, or only at the ends of the chunks' rows and segments, where a row that is
left out, taken twice or misplaced is half of the sum and more.

Tolerance: a chunk is 512 products one after the other in the tensor core, whose FP32 additions truncate:
512 x 2^-24 = 3e-5 of a chunk's sum at most; 1e-4 of a layer's norm.  Biases are FP32 sums of the same
length.
"""
import numpy as np
import pytest
import torch

from oracle import unet as U
from paper_2604_15434_gb300 import synth

pytestmark = pytest.mark.gpu

EFT = (-0.8, 0.4, 0.9)
OFF = np.cumsum([0] + [27 * ci * co + co for ci, co in U.CONVS])


def one_hot(p, layer, pairs):
    """Layer `layer` passes input ci to output co for each (ci, co), without bias."""
    ci, co = U.CONVS[layer]
    p[OFF[layer]:OFF[layer + 1]] = 0.0
    w = p[OFF[layer]:OFF[layer] + 27 * ci * co].reshape(27, ci, co)
    for i, o in pairs:
        w[13, i, o] = 1.0


def head(p, w):
    p[OFF[10]:OFF[10] + 16] = w
    p[OFF[10] + 16] = 0.0


class Reader:
    """The network's activations, channel by channel through the head."""

    def __init__(self, net, base, delta):
        self.net, self.base, self.delta = net, base, delta

    def run(self, p):
        self.net.set_params(p)
        return self.net.forward(self.delta, *EFT)

    def channels(self, p, count=16):
        out = []
        for c in range(count):
            q = p.copy()
            head(q, np.eye(16, dtype=np.float32)[c])
            out.append(self.run(q).float())
        return torch.stack(out)

    def layer8_inputs(self, p, first):
        q = p.copy()
        one_hot(q, 8, [(first + c, c) for c in range(16)])
        return self.channels(q)

    def coarse(self, p):  # 32 channels of the half-size level under layer 8
        return torch.cat([self.layer8_inputs(p, f)[:, ::2, ::2, ::2] for f in (0, 16)])

    def cat2(self):
        out = []
        for f in (0, 32, 64):
            q = self.base.copy()
            one_hot(q, 6, [(f + c, c) for c in range(32)])
            out.append(self.coarse(q))
        return torch.cat(out)


def bf16(x):
    return x.bfloat16().float()


def contraction(x, dy):
    """dW[tap][ci][co] and db[co] in FP64."""
    ci, co = x.shape[0], dy.shape[0]
    d = dy.double().reshape(co, -1).T.contiguous()
    dw = torch.empty((27, ci, co), dtype=torch.float64, device="cuda")
    xd = x.double()
    for t in range(27):
        s = torch.roll(xd, (1 - t // 9, 1 - (t // 3) % 3, 1 - t % 3), (1, 2, 3))
        dw[t] = s.reshape(ci, -1) @ d
    return dw.cpu().numpy().ravel(), d.sum(0).cpu().numpy()


@pytest.mark.parametrize("n", [32, 64, 128, 256])
def test_gradients_from_their_operands(gpu_lib, n):
    rng = np.random.default_rng(n)
    delta = torch.from_numpy(synth.lognormal_delta(n, -2.0, 1.2, 21)).cuda()
    base = np.asarray(U.init_params(7), dtype=np.float32).copy()
    one_hot(base, 7, [(c, c) for c in range(32)])
    one_hot(base, 8, [(f + c, c) for f in (0, 16, 32) for c in range(16)])
    one_hot(base, 9, [(c, c) for c in range(16)])
    hw = rng.uniform(0.2, 1.0, 16).astype(np.float32) * rng.choice([-1.0, 1.0], 16).astype(np.float32)
    head(base, hw)
    net = gpu_lib.UNet()
    read = Reader(net, base, delta)
    y8, y6 = read.channels(base), read.coarse(base)
    cat1 = torch.cat([read.layer8_inputs(base, f) for f in (0, 16, 32)])
    cat2 = read.cat2()
    assert min(float((a > 0).float().mean()) for a in (y8, y6, cat1, cat2)) > 0.05
    that = read.run(base)
    edge = min(n // 2, 64)
    i = torch.arange(n, device="cuda")
    ends = (i % edge == 0) | (i % edge == edge - 1)
    where = {"all": torch.ones((n, n, n), dtype=torch.bool, device="cuda"),
             "ends": (ends[None, :, None] | ends[None, None, :]).expand(n, n, n)}
    for kind, sel in where.items():
        noise = torch.from_numpy(rng.standard_normal((n, n, n))).cuda()
        target = torch.where(sel, that + noise, that).float()
        net.set_params(base)
        net.zero_grad()
        net.loss_grad(delta, target, *EFT)
        got = net.get_params(grads=True).astype(np.float64)
        g = (2.0 * (that - target.double()) / n ** 3).float()
        d9 = torch.stack([torch.where(y8[c] > 0, bf16(g * float(hw[c])), torch.zeros_like(g)) for c in range(16)])
        dcat1 = torch.where(cat1 > 0, torch.cat([d9, d9, d9]), torch.zeros_like(cat1))
        s = torch.zeros((32,) + (n // 2,) * 3, device="cuda")
        for k in range(8):  # the children in the kernel's order
            s = s + dcat1[:32, k >> 2::2, (k >> 1) & 1::2, k & 1::2]
        d7 = bf16(s)
        d6 = torch.where(y6 > 0, d7, torch.zeros_like(d7))
        for layer, x, dy in ((9, y8, d9), (8, cat1, d9), (7, y6, d7), (6, cat2, d6)):
            dw, db = contraction(x, dy)
            a = got[OFF[layer]:OFF[layer + 1]]
            for want, have in ((dw, a[:dw.size]), (db, a[dw.size:])):
                assert np.linalg.norm(have - want) <= 1e-4 * np.linalg.norm(want), (kind, layer, want.size)
