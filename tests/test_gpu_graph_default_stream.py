"""Graph replay on the legacy default stream: the steps of a simulation there
(captured on a stream of the library's own, replayed on the default stream)
give bitwise the state of direct launches (a flow-rate control whose gain is
zero keeps the graphs off), stay ordered with other work of the default
stream, and follow a change of the body force; the timing hooks see every
step, also when they are switched off and on again between replays."""
import numpy as np
import pytest

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


def _sim(storage, stream):
    return F.Simulation.from_workload(W.tiny().generate(), storage=storage, stream=stream, spheres=False)


@pytest.mark.parametrize("storage", [F.STORE_FP32, F.STORE_FP16])
def test_default_stream_replay_is_bitwise_direct_launches(storage):
    import torch
    legacy = torch.cuda.default_stream()
    assert legacy.cuda_stream == 0
    a, b, c = _sim(storage, legacy), _sim(storage, legacy), _sim(storage, torch.cuda.Stream())
    b.set_flow_control(0.0, 0.0, 1000000)
    n = a.n
    for steps in (1, 2, 7, 4):
        # a device write queued before the steps on the default stream and a
        # read queued after them, without a synchronisation between
        x = torch.zeros(1 << 20, device="cuda")
        x += 1.0
        for s in (a, b, c):
            s.step(steps)
        out = [torch.empty(27 * n, dtype=torch.float64, device="cuda") for _ in range(3)]
        for s, o in zip((a, b, c), out):
            F._check(F.fslbm_get_fields(s.h, F.FIELD_PDF, [o], on_device=True), "get")
        assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
        assert float(x.sum()) == 1 << 20
        for s in (a, b, c):
            s.set_body_force([3e-6 * steps, 0.0, -1e-5])
    assert np.array_equal(a.get(F.FIELD_TYPE), b.get(F.FIELD_TYPE))


def test_timing_switched_between_replays():
    import torch
    s = _sim(F.STORE_FP32, torch.cuda.default_stream())
    s.step(4)
    for _ in range(2):
        s.timing(True)
        s.step(6)
        ms, sweeps, launches = s.timing_read()
        assert sweeps == 6 and ms > 0 and launches > 6
        s.timing(False)
        s.step(3)
        assert s.timing_read()[1] == 6
    s.sync()
