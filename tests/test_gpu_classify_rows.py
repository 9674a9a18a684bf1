"""Interface and solid-surface lists for rows of every kind of last 32-cell
word, x periodic and walled: a cell left out of either list shows at once (an
interface cell stays uncollided, a surface cell's links keep stale values),
against the oracle after four steps. FP32: 6e-8 per operation, some 30 of them
a step, 1e-5 of a PDF in all; a stale or missing link is wrong by 1e-3 and
more of it."""
import numpy as np
import pytest

import oracle as O
from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

from helpers import oracle_from_workload, pdf_rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


@pytest.mark.parametrize("nx", [13, 31, 32, 33, 63, 65, 97])
@pytest.mark.parametrize("periodic", [(1, 0, 0), (0, 1, 0)])
def test_lists_of_every_row_length(nx, periodic):
    w = W.Workload(name="rows", nx=nx, ny=11, nz=21, periodic=periodic, liquid_height=14.3, diameter=5.0, bed="hex",
                   bed_height=9.0, seed=2).generate()
    sim = F.Simulation.from_workload(w)
    o = oracle_from_workload(w)
    sim.step(4)
    o.step(4)
    types = o.get(O.F_TYPE)
    assert (types == F.SOLID).any() and (types == F.INTERFACE).any()
    assert np.array_equal(sim.get(F.FIELD_TYPE), types)
    assert pdf_rel_err(sim.get(F.FIELD_PDF), o.get(O.F_PDF), types) < 1e-5
    sim.close()
