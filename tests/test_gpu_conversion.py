"""Conversion, re-mapping and classification kernels at the sizes where their
lane and list handling can go wrong: extents below a warp's width, extents of
three cells with periodic wrap (where a cell's neighbours repeat), extents no
multiple of 32, walls on every axis, both excess variants. Cell types are
those of the FP64 oracle, and in the 16-bit formats the mass and the
liquid-gas separation hold."""
import numpy as np
import pytest

import oracle as O
from helpers import oracle_from_workload
from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [((32, 8, 24), (1, 0, 0), 0), ((17, 9, 21), (0, 0, 0), 0), ((16, 6, 20), (1, 1, 0), 1), ((3, 4, 20), (1, 1, 0), 0),
         ((70, 5, 19), (1, 0, 0), 1)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


def _workload(size, periodic, spheres):
    nx, ny, nz = size
    w = W.Workload(name="t", nx=nx, ny=ny, nz=nz, periodic=periodic, tau=0.6, g=(2e-4, 0.0, -8e-4), liquid_height=11.0,
                   diameter=5.0, bed="none").generate()
    if spheres and nx >= 16:
        # two overlapping mobile spheres near the surface and a fixed one
        w.xyz = np.array([[6.2, 3.1, 8.3], [9.9, 3.3, 8.1], [6.0, 2.6, 2.5]])
        w.radius = np.array([2.0, 2.0, 2.0])
        w.fixed = np.array([0, 0, 1], np.uint8)
    return w


def _surface(w):
    x, y = np.arange(w.nx) + 0.5, np.arange(w.ny) + 0.5
    return 11.0 + 2.5 * np.sin(2 * np.pi * x / w.nx)[None, :] * (1 + 0.2 * np.cos(2 * np.pi * y / w.ny))[:, None]


def _gpu(w, storage, even):
    import torch
    p = F.params_from_workload(w, storage)
    p.excess_even = even
    sim = F.Simulation(p, torch.cuda.Stream())
    if w.nspheres:
        sim.add_spheres(w.xyz, w.radius, w.fixed)
    sim.init_surface(_surface(w))
    return sim


@pytest.mark.parametrize("size,periodic,even", CASES)
@pytest.mark.parametrize("spheres", [False, True])
def test_types_match_the_oracle(size, periodic, even, spheres):
    w = _workload(size, periodic, spheres)
    sim = _gpu(w, F.STORE_FP32, even)
    o = oracle_from_workload(w, excess_even=even)
    o.init_surface(_surface(w))
    t0 = sim.get(F.FIELD_TYPE)
    for _ in range(8):
        sim.step(5)
        o.step(5)
        assert (sim.get(F.FIELD_TYPE) == o.get(O.F_TYPE)).all()
    assert (sim.get(F.FIELD_TYPE) != t0).any()                       # cells converted
    m, mo = sim.get(F.FIELD_MASS), o.get(O.F_MASS)
    assert np.abs(m - mo).max() < 1e-4
    assert sim.violations == 0


@pytest.mark.parametrize("size,periodic,even", CASES)
@pytest.mark.parametrize("storage,tol", [(F.STORE_FP16, 1e-5), (F.STORE_BF16, 1e-4)])
def test_16bit_keeps_mass_and_separation(storage, tol, size, periodic, even):
    w = _workload(size, periodic, True)
    sim = _gpu(w, storage, even)
    m0 = sim.reduce()[0]
    sim.step(41)
    assert sim.violations == 0
    assert abs(sim.reduce()[0] - m0) < tol * m0
