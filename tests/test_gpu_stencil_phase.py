"""Fill levels of sine surfaces at phases far from zero, where the FP32 argument
of the sine is rounded coarsely: the counts are those of every sample with the
kernel's own arguments (formed here in FP32 like the kernel's, the sine itself in
FP64), so a cell, row or run is only taken as a whole where that rounding cannot
change a sample. A sample within about 1e-6 of the surface may fall either way:
about one in 40 000 of the rows' crossings a unit of error, and a run whose
argument lies on a rounding tie moves by up to 16 samples; 40 of a cell's 262 144
samples bounds both."""
import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F

pytestmark = pytest.mark.gpu
SUBS = 64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _surfaces(n, size):
    rng = np.random.default_rng(11)
    v = rng.standard_normal((n, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    u = rng.standard_normal((n, 3))
    u -= (u * v).sum(1)[:, None] * v
    u /= np.linalg.norm(u, axis=1)[:, None]
    P = np.zeros((n, 12))
    P[:, 0] = 3
    P[:, 1:4], P[:, 9:12] = v, u
    P[:, 4] = rng.uniform(-0.7, 0.7, n)
    P[:, 5] = 5.0
    P[:, 6] = rng.uniform(0.1, 1.0, n)
    P[:, 7] = rng.uniform(0.1, 1.2, n)
    P[:, 8] = rng.uniform(0.5, 1.0, n) * size
    return P


def _counts(row):
    f32 = np.float32
    n0, e1, s, A, k, ph = row[1:4], row[9:12], row[4], row[6], row[7], row[8]
    fe, fn = e1.astype(f32), n0.astype(f32)
    kf, pf, Af, As = f32(k), f32(ph), f32(A), f32(A * np.sin(ph))
    o = ((np.arange(SUBS, dtype=f32) + f32(0.5)) / f32(SUBS)).astype(f32)
    out = []
    for q in range(27):
        c = np.array([q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1], float)
        b = c - 0.5 - s * n0
        bu, bw = f32(b @ e1), f32(b @ n0)
        yz_u = (o[0] * fe[0] + o[:, None] * fe[1] + o[None, :] * fe[2]).astype(f32)
        yz_w = (o[0] * fn[0] + o[:, None] * fn[1] + o[None, :] * fn[2]).astype(f32)
        u0, w0 = (bu + yz_u).astype(f32), (bw + yz_w).astype(f32)
        cnt = 0
        for seg in range(0, SUBS, 16):
            ur = (u0 + f32(seg) * (fe[0] / f32(SUBS))).astype(f32)
            arg = (float(kf) * ur.astype(float) + float(pf)).astype(f32).astype(float)
            j = np.arange(16)
            x = arg[..., None] + j * float(f32(k * e1[0] / SUBS))
            w = w0.astype(float)[..., None] + (seg + j) * float(fn[0] / f32(SUBS))
            cnt += int(np.sum(w <= float(Af) * np.sin(x) - float(As)))
        out.append(cnt)
    return np.array(out)


@pytest.mark.parametrize("size", [6.0, 1e4, 6e4, 6e5, 6e6])
def test_counts_are_those_of_every_sample(size):
    import torch
    P = _surfaces(6, size)
    fill = torch.empty(len(P), 27, device="cuda")
    target = torch.empty(len(P), 4, device="cuda")
    assert F.fslbm_mlp_stencils(torch.from_numpy(P).cuda(), len(P), fill, target) == 0
    got = np.rint(fill.cpu().numpy().astype(float) * SUBS ** 3).astype(int)
    ref = np.array([_counts(r) for r in P])
    assert np.abs(got - ref).max() <= 40
