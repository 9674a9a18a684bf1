"""Training surfaces where whole cells, rows and runs are counted without
their samples: surfaces just inside and outside a cell's corners, the
smallest and largest radii, steep and flat sines, normals along the axes.
Fill levels against FP64 samples and chords at the same points: a sample can
fall on the other side only where the FP32 evaluation (2e-5 for amplitudes up
to 8) places it within rounding of the surface, which is a surface share of a
cell, so 5e-4 of its volume bounds it; chords are FP32 sums, 3e-5."""
import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

pytestmark = pytest.mark.gpu
C = np.array([[q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1] for q in range(27)], float)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _rows():
    rows = []
    s2, s3 = 1 / np.sqrt(2), 1 / np.sqrt(3)
    for n0, e1 in (((0, 0, 1), (1, 0, 0)), ((1, 0, 0), (0, 1, 0)), ((0, -1, 0), (0, 0, 1)), ((s2, s2, 0), (s2, -s2, 0)),
                   ((s3, s3, s3), (s2, -s2, 0)), ((-s3, s3, -s3), (s2, s2, 0))):
        for s in (-0.5, 0.0, 0.5, 0.366):
            for r in (2.0, 2.5, 30.0):
                rows += [(1, *n0, s, r, 0, 0, 0, *e1), (2, *n0, s, r, 0, 0, 0, *e1)]
            for A, lam, ph in ((8.0, 16.0, 1.5707963), (8.0, 16.0, 0.0), (1.0, 256.0, 3.0), (4.0, 40.0, 5.5)):
                rows.append((3, *n0, s, 0, A, 2 * np.pi / lam, ph, *e1))
    return np.array(rows, float)


def test_fill_levels_are_those_of_all_samples():
    import torch
    rows = _rows()
    n = len(rows)
    fill = torch.empty(n, 27, dtype=torch.float32, device="cuda")
    tgt = torch.empty(n, 4, dtype=torch.float32, device="cuda")
    assert F.fslbm_mlp_stencils(torch.from_numpy(rows).cuda(), n, fill, tgt) == 0
    got = fill.cpu().numpy().astype(float)
    P = torch.from_numpy(rows).cuda()
    sub = (torch.arange(64, dtype=torch.float64, device="cuda") + 0.5) / 64 - 0.5
    z, y, x = torch.meshgrid(sub, sub, sub, indexing="ij")
    for i in range(n):
        kind, n0, s, r, A, k, ph, e1 = rows[i, 0], P[i, 1:4], rows[i, 4], rows[i, 5], rows[i, 6], rows[i, 7], rows[i, 8], P[i, 9:12]
        for q in range(27):
            d = [g + C[q, a] - s * float(n0[a]) for a, g in enumerate((x, y, z))]
            if kind == 3:
                u = sum(d[a] * e1[a] for a in range(3))
                w = sum(d[a] * n0[a] for a in range(3))
                ref, tol = float((w <= A * (torch.sin(k * u + ph) - np.sin(ph))).double().mean()), 5e-4
            else:
                o = [(s + (-r if kind == 1 else r)) * float(n0[a]) - C[q, a] for a in range(3)]
                h2 = r * r - (y[:, :, 0] - o[1]) ** 2 - (z[:, :, 0] - o[2]) ** 2
                h = h2.clamp(min=0).sqrt()
                ch = ((o[0] + h).clamp(max=0.5) - (o[0] - h).clamp(min=-0.5)).clamp(min=0) * (h2 > 0)
                ref, tol = float(ch.mean()), 3e-5
                ref = ref if kind == 1 else 1 - ref
            assert abs(got[i, q] - ref) < tol, (i, q, rows[i])
