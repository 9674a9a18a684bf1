"""Gradient and inference of the learned normal at the edges of the 16-sample
tiles, the 128-sample chunks, the 32 chunks added per round and the 128 chunks
held at once, against FP64 with BF16 operands at the same places.

Tolerance per entry: FP32 rounding can move an operand over a BF16 rounding
boundary (about 1 in 1e4 of them), which changes its terms by 2^-8: 1e-3 of the
sum of the terms' magnitudes, and 2^-7 of the largest term where few are
summed."""
import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LAM, MU = 0.4, 0.1


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _bf(x):
    import torch
    return x.float().to(torch.bfloat16).double()


def _case(n):
    import torch
    theta = torch.from_numpy(W.mlp_initial_weights(n)).float()
    theta[27 * 64:27 * 64 + 64] = 0.05
    gen = torch.Generator().manual_seed(n)
    fill = torch.rand(n, 27, generator=gen)
    nv = torch.randn(n, 3, generator=gen)
    target = torch.cat([nv / nv.norm(dim=1, keepdim=True), torch.rand(n, 1, generator=gen) - 0.5], 1)
    p, at = [], 0
    for o, i in ((64, 27), (64, 64), (4, 64)):
        p += [_bf(theta[at:at + o * i].reshape(o, i)).cuda(), theta[at + o * i:at + o * i + o].double().cuda()]
        at += o * i + o
    return theta.cuda(), fill.cuda(), target.float().cuda(), p


def _forward(p, fill):
    import torch
    w1, b1, w2, b2, w3, b3 = p
    x = _bf(fill)
    h1 = _bf(torch.relu(x @ w1.t() + b1))
    h2 = _bf(torch.relu(h1 @ w2.t() + b2))
    return x, h1, h2, h2 @ w3.t() + b3


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 129, 4096, 4097, 16384, 16385, 2 * 16384 + 77])
def test_gradient_at_the_edges_of_the_batch_split(n):
    import torch
    theta, fill, target, p = _case(n)
    grad = torch.zeros(F.MLP_NPARAM, device="cuda")
    loss = torch.zeros(1, device="cuda")
    assert F.fslbm_mlp_gradient(theta, fill, target, n, LAM, MU, grad, loss) == 0
    x, h1, h2, y = _forward(p, fill)
    tg = target.double()
    r = y[:, :3].norm(dim=1, keepdim=True)
    dot = (y[:, :3] * tg[:, :3]).sum(1, keepdim=True)
    dk = y[:, 3:] - tg[:, 3:]
    L = (1 - dot / r + LAM * dk ** 2 + MU * (r - 1) ** 2) / n
    dy = torch.cat([-tg[:, :3] / r + dot / r ** 3 * y[:, :3] + 2 * MU * (r - 1) / r * y[:, :3], 2 * LAM * dk], 1) / n
    d2 = (_bf(dy) @ p[4]) * (h2 > 0)
    d1 = (_bf(d2) @ p[2]) * (h1 > 0)
    got = grad.double()
    at = 0
    for d, h in ((d1, x), (d2, h1), (dy, h2)):
        for ref, mag, top in ((_bf(d).t() @ h, _bf(d).abs().t() @ h.abs(),
                               (_bf(d).abs().max(0).values[:, None] * h.abs().max(0).values)),
                              (d.sum(0), d.abs().sum(0), d.abs().max(0).values)):
            a = got[at:at + ref.numel()].reshape(ref.shape)
            err = (a - ref).abs() - 1e-3 * mag - 2.0 ** -7 * top
            assert err.max() <= 0, (tuple(ref.shape), float(err.max()))
            at += ref.numel()
    assert abs(float(loss) - float(L.sum())) <= 1e-3 * float(L.abs().sum())


@pytest.mark.parametrize("n", [1, 16, 17, 129, 152 * 3 * 8 * 16 + 3])
def test_inference_at_the_edges_of_the_tiles(n):
    import torch
    theta, fill, _, p = _case(n)
    out = torch.full((n + 1, 4), 7.0, device="cuda")
    assert F.fslbm_mlp_infer(theta, fill, n, out) == 0
    _, _, h2, y = _forward(p, fill)
    assert ((out[:n].double() - y).abs() <= 2.0 ** -7 * (h2.abs() @ p[4].abs().t()) + 1e-6).all()
    assert (out[n] == 7.0).all()
