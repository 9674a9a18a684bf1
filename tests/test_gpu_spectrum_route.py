"""The bed spectrum of extents with a large prime factor takes no longer than
that of slightly longer ones beyond the factored transforms' range, where the
direct sums run (whose time grows with the extents): twice the time would be
the factored way's one block per two rows or four columns, which the direct
sums spread over the GPU."""
import time

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


def _time(nt, nx):
    import torch
    h = torch.randn(nt, nx, dtype=torch.float64, device="cuda")
    psd = torch.empty_like(h)
    best = float("inf")
    for _ in range(6):
        torch.cuda.synchronize()
        t = time.perf_counter()
        rc, _ = F.fslbm_bed_spectrum(h, nt, nx, 1.0, 10.0, psd)
        best = min(best, time.perf_counter() - t)
        assert rc == 0
    return best


@pytest.mark.parametrize("size,direct", [((20, 7159), (20, 7187)), ((40, 7162), (40, 7187)), ((20, 3499), (20, 7187)),
                                         ((7159, 20), (7187, 20))])
def test_large_prime_factors(size, direct):
    assert _time(*size) < 1.5 * _time(*direct)
