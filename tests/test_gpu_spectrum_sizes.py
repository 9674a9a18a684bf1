"""Bed spectrum over the sizes where the factored transforms can go wrong:
the smallest series, odd and prime extents, every radix, the largest extents
of shared memory, and one column and row beyond them, where the direct sums
run. PSD against numpy's FP64 transform: its error is a few roundings of the
largest value (N log N sums of relative 1e-16), so 1e-12 of the largest PSD
value bounds both; the peak follows from the PSD."""
import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


@pytest.mark.parametrize("nt,nx", [(2, 2), (2, 3), (3, 2), (3, 5), (5, 7), (16, 81), (25, 121), (29, 349), (30, 210),
                                   (97, 97), (100, 1024), (1793, 13), (3585, 6), (7168, 4), (3, 7168), (2, 7165),
                                   (2, 7169), (7169, 3)])
def test_psd_matches_numpy(nt, nx):
    import torch
    rng = np.random.default_rng(nt * 10007 + nx)
    t, x = np.arange(nt)[:, None], np.arange(nx)[None, :]
    j, l = max(1, nx // 5), -(nt // 3)
    h = 100.0 + 2.0 * np.sin(2 * np.pi * (j * x / nx + l * t / nt) + 0.3) + 0.2 * rng.standard_normal((nt, nx))
    psd = torch.full((nt, nx), np.nan, dtype=torch.float64, device="cuda")
    rc, peak = F.fslbm_bed_spectrum(torch.from_numpy(h).cuda(), nt, nx, 1.0, 10.0, psd)
    assert rc == 0
    got = psd.cpu().numpy()
    ref = np.abs(np.fft.fft2(h - h.mean())) ** 2 / (nt * nx)
    assert np.abs(got - ref).max() < 1e-12 * max(ref.max(), 1.0)
    top = got[:, 1:nx // 2 + 1]
    at = np.unravel_index(int(top.argmax()), top.shape)
    assert peak[0] == nx / (at[1] + 1)
    assert abs(peak[3] - 2 * np.sqrt(top.max() / (nt * nx))) < 1e-12
    ls = at[0] if at[0] <= nt // 2 else at[0] - nt
    assert peak[1] == (np.inf if ls == 0 else nt * 10.0 / abs(ls))


def test_series_with_nan_gives_a_result():
    import torch
    h = torch.full((6, 40), float("nan"), dtype=torch.float64, device="cuda")
    psd = torch.empty_like(h)
    rc, _ = F.fslbm_bed_spectrum(h, 6, 40, 1.0, 1.0, psd)
    assert rc == 0 and bool(torch.isnan(psd).all())
