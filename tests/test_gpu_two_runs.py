"""Two runs of different particle counts in one process, stepped in turn past
the capture of their graphs and from two host threads at once (with graphs and
with direct launches): each gives the state it gives alone. The box holds no
liquid, so nothing is summed in a changing order and the states are bitwise
the same."""
import threading

import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F

pytestmark = pytest.mark.gpu

FIELDS = (F.FIELD_P_X, F.FIELD_P_U, F.FIELD_P_OMEGA, F.FIELD_TYPE)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _sim(n, direct):
    import torch
    p = F.fslbm_default_params()
    p.nx, p.ny, p.nz = 256, 64, 64
    p.bc_flags = F.PERIODIC_X
    p.g[:] = [1e-4, 0.0, -2e-4]
    p.liquid_height = 0.0
    sim = F.Simulation(p, torch.cuda.Stream())
    k = np.arange(n)
    xyz = np.stack([2.1 + 4.2 * (k % 60), 3.0 + 4.1 * (k // 60 % 14), 2.0 + 4.0 * (k // 840)], 1)
    xyz += np.random.default_rng(n).uniform(-0.1, 0.1, xyz.shape)
    sim.add_spheres(xyz, np.full(n, 2.0))
    if direct:
        sim.set_flow_control(0.0, 0.0, 1 << 30)      # no graphs with the flow control on
    return sim


def _state(sim):
    return [sim.get(f) for f in FIELDS]


def _alone(n, steps, direct):
    sim = _sim(n, direct)
    sim.step(steps)
    return _state(sim)


# particle counts that run in the same kernel with different block sizes
@pytest.mark.parametrize("sizes", [(3, 64), (1030, 2000), (34, 2000)])
@pytest.mark.parametrize("direct", [False, True])
def test_runs_do_not_disturb_one_another(sizes, direct):
    alone = [_alone(n, 600, direct) for n in sizes]
    a, b = (_sim(n, direct) for n in sizes)
    for _ in range(50):
        a.step(2)
        b.step(2)
    threads = [threading.Thread(target=lambda s=s: [s.step(5) for _ in range(100)]) for s in (a, b)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for sim, ref in zip((a, b), alone):
        for x, y in zip(_state(sim), ref):
            assert np.array_equal(x, y)
