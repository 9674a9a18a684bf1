"""Field export and import: the one-pass kernel that writes device buffers
directly gives bitwise what the staged copies to host memory give, at every
storage format, after even and odd steps, for lattices no vector width
divides; a device buffer the kernel cannot address directly (here one off its
alignment) takes the staged copy with the same result; FP64 moments agree with
sums over the exported PDFs; and a state set from device buffers equals the
state set from host arrays."""
import numpy as np
import pytest

from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CELL = (F.FIELD_PDF, F.FIELD_TYPE, F.FIELD_MASS, F.FIELD_PHI, F.FIELD_RHO, F.FIELD_U, F.FIELD_NORMAL, F.FIELD_OWNER)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _sim(storage, nx, ny, nz, periodic=(1, 0, 0)):
    import torch
    w = W.Workload(name="t", nx=nx, ny=ny, nz=nz, periodic=periodic, liquid_height=0.7 * nz, diameter=5.0,
                   bed="hex", bed_height=0.5 * nz, seed=2).generate()
    return F.Simulation.from_workload(w, storage=storage, stream=torch.cuda.Stream())


def _device(sim, mask, fields, offset=0):
    """All fields of `mask` by one call into device buffers `offset` bytes off
    their natural alignment."""
    import torch
    host = [sim._alloc(f) for f in fields]
    raw = [torch.zeros(h.nbytes + 16, dtype=torch.uint8, device="cuda") for h in host]
    torch.cuda.synchronize()             # the buffers' zeroing, on another stream than the run's
    F._check(F.fslbm_get_fields(sim.h, mask, [int(r.data_ptr()) + offset for r in raw], on_device=True), "get")
    return [r.cpu().numpy()[offset:offset + h.nbytes].view(h.dtype).reshape(h.shape) for r, h in zip(raw, host)]


@pytest.mark.parametrize("storage", [F.STORE_FP32, F.STORE_FP16, F.STORE_BF16])
@pytest.mark.parametrize("size,steps", [((64, 16, 24), 3), ((37, 11, 23), 4), ((37, 11, 23), 1), ((8, 9, 16), 2)])
def test_export_routes_agree(storage, size, steps):
    sim = _sim(storage, *size)
    sim.step(steps)
    mask = sum(CELL)
    host = [sim.get(f) for f in CELL]
    for offset in (0, 4):
        for f, a, b in zip(CELL, _device(sim, mask, CELL, offset), host):
            assert a.tobytes() == b.tobytes(), (hex(f), offset)
    pdf, types, rho, u = host[0], host[1], host[4], host[5]
    fluid = (types == F.LIQUID) | (types == F.INTERFACE)
    # FP64 sums over the exported PDFs (their own rounding: 27 values at 1e-16)
    assert np.abs(pdf.sum(0) - rho)[fluid].max() < 1e-14
    C = np.array([[q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1] for q in range(27)], float)
    for a in range(3):
        j = np.tensordot(C[:, a], pdf, 1)
        ref = (j - 0.5 * rho * sim.params.g[a])[fluid] / rho[fluid]
        assert np.abs(u[a][fluid] - ref).max() < 1e-14
    assert not pdf[:, ~fluid].any() and not rho[~fluid].any()


@pytest.mark.parametrize("storage", [F.STORE_FP32, F.STORE_FP16])
@pytest.mark.parametrize("steps", [1, 2])
def test_import_routes_agree(storage, steps):
    import torch
    src = _sim(storage, 37, 11, 23)
    src.step(steps)
    pdf = src.get(F.FIELD_PDF)
    pdf *= 1.0 + 1e-3 * np.random.default_rng(1).uniform(-1, 1, pdf.shape)
    a, b = _sim(storage, 37, 11, 23), _sim(storage, 37, 11, 23)
    for s in (a, b):
        s.step(steps)
    a.set(F.FIELD_PDF, pdf)
    dev = torch.from_numpy(pdf).cuda()
    F._check(F.fslbm_set_fields(b.h, F.FIELD_PDF, [dev], on_device=True), "set")
    for f in CELL:
        assert a.get(f).tobytes() == b.get(f).tobytes(), hex(f)


@pytest.mark.parametrize("on_device", [False, True])
def test_export_refuses_null(on_device):
    import ctypes
    sim = _sim(F.STORE_FP32, 8, 9, 16)
    arr = (ctypes.c_void_p * 1)(None)
    assert F.load().fslbm_get_fields(sim.h, F.FIELD_PDF, arr, int(on_device)) == -1
    assert F.load().fslbm_set_fields(sim.h, F.FIELD_PDF, arr, int(on_device)) == -1
