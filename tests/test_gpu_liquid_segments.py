"""Liquid kernels of the 16-bit formats on segments of 256 cells: row lengths
just beyond a segment, of one and a half, of two segments less a pair, and
short ones; walls and periodic axes; spheres across segment borders. PDFs
against the FP64 oracle within the storage's rounding after an even and after
an odd last step (16 roundings of 2^-11 and 2^-8 of deviations below 0.02 w), cell
types exact."""
import numpy as np
import pytest

import oracle as O
from helpers import oracle_from_workload, weights
from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


@pytest.mark.parametrize("storage,tol", [(F.STORE_FP16, 2e-4), (F.STORE_BF16, 2e-3)])
@pytest.mark.parametrize("nx,ny,nz,periodic", [(258, 8, 12, (1, 0, 0)), (320, 6, 14, (1, 1, 0)), (384, 7, 12, (0, 0, 0)),
                                               (510, 6, 12, (1, 0, 0)), (62, 9, 13, (1, 0, 0)), (4, 6, 14, (1, 0, 0))])
@pytest.mark.parametrize("steps", [3, 4])
def test_segments_match_the_oracle(storage, tol, nx, ny, nz, periodic, steps):
    import torch
    w = W.Workload(name="seg", nx=nx, ny=ny, nz=nz, periodic=periodic, tau=0.55, g=(5e-6, 0.0, -5e-5), liquid_height=9.0,
                   diameter=4.0, bed="none").generate()
    if nx > 60:
        w.xyz = np.array([[20.3, 3.1, 4.2], [nx - 1.6 if periodic[0] else nx - 4.0, 3.0, 3.2], [min(255.8, nx / 2), 3.2, 4.1]])
        w.radius = np.array([1.9, 1.7, 1.8])
        w.fixed = np.array([0, 1, 0], np.uint8)
    sim = F.Simulation.from_workload(w, storage=storage, stream=torch.cuda.Stream())
    o = oracle_from_workload(w)
    sim.step(steps)
    o.step(steps)
    to = o.get(O.F_TYPE)
    assert (sim.get(F.FIELD_TYPE) == to).all()
    fl = (to == 1) | (to == 2)
    dev = np.abs(sim.get(F.FIELD_PDF)[:, fl] - o.get(O.F_PDF)[:, fl]) / weights()[:, None]
    assert dev.max() < tol
