"""Particle map on periodic axes that a sphere nearly spans: after every step
the solid cells are those whose centre lies within the radius of the nearest
image of the centre, from the positions of the state itself (FP64; a cell
centre within 1e-9 of a surface would be left out)."""
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


def _sim(shape, periodic, g, xyz, radius, fixed=None):
    import torch
    p = F.fslbm_default_params()
    p.nx, p.ny, p.nz = shape
    p.bc_flags = sum(bit for bit, on in zip((F.PERIODIC_X, F.PERIODIC_Y, F.PERIODIC_Z), periodic) if on)
    p.g[:] = g
    p.liquid_height = 0.0                       # no liquid: the spheres fall freely
    sim = F.Simulation(p, torch.cuda.Stream())
    sim.add_spheres(xyz, radius, fixed)
    return sim


def _wrong(sim, shape, periodic, radius):
    """cells whose type is not the sphere rule's"""
    X = sim.get(F.FIELD_P_X)
    inside = np.full(shape[::-1], -np.inf)
    for c, r in zip(X, radius):
        d2 = 0.0
        for a in range(3):
            d = np.arange(shape[a]) + 0.5 - c[a]
            if periodic[a]:
                d = d - shape[a] * np.rint(d / shape[a])
            d2 = d2 + (d ** 2).reshape([-1 if 2 - a == k else 1 for k in range(3)])
        inside = np.maximum(inside, r - np.sqrt(d2))
    solid = sim.get(F.FIELD_TYPE).reshape(shape[::-1]) == 3
    return int(np.sum((solid != (inside > 0)) & (np.abs(inside) > 1e-9)))


@pytest.mark.parametrize("shape,periodic,radius", [((24, 8, 24), (1, 1, 0), 2.5), ((24, 8, 24), (1, 1, 0), 3.9),
                                                   ((7, 24, 24), (1, 0, 0), 3.2), ((24, 24, 9), (0, 1, 1), 4.3),
                                                   ((32, 24, 24), (1, 1, 1), 3.0)])
def test_sphere_crossing_a_seam(shape, periodic, radius):
    axis = int(np.argmin(shape))
    g = [0.0, 0.0, 0.0]
    g[axis] = 4e-3
    x0 = [12.3, 12.4, 12.2]
    x0[axis] = 0.55 * shape[axis]
    sim = _sim(shape, periodic, g, np.array([x0]), np.array([radius]))
    # past the axis' end, with a cell's width a few steps
    for k in range(20):
        assert _wrong(sim, shape, periodic, [radius]) == 0, k
        sim.step(3)
    assert np.sum(sim.get(F.FIELD_TYPE) == 3) > 20


@pytest.mark.parametrize("L", [10, 11, 16])
def test_sphere_that_nearly_spans_an_axis(L):
    """radii up to half the axis, where a cell's nearest image is not that of
    the integer parts' difference"""
    rng = np.random.default_rng(L)
    n = 14
    shape, periodic = (n * (L + 2), L, 2 * L + 8), (1, 1, 0)
    xyz = np.stack([(np.arange(n) + 0.5) * (L + 2), rng.uniform(0, L, n), L + 4 + rng.uniform(-1, 1, n)], 1)
    radius = 0.5 * L - rng.uniform(0.01, 0.45, n)
    sim = _sim(shape, periodic, (0.0, 3e-4, 0.0), xyz, radius)
    for k in range(20):
        assert _wrong(sim, shape, periodic, radius) == 0, k
        sim.step(2)


@pytest.mark.parametrize("fixed", [0, 1])
@pytest.mark.parametrize("z", [0.7, 23.6])
def test_sphere_across_the_z_seam_at_set_up(z, fixed):
    """no other sphere reaches the cells on the far side"""
    shape, periodic = (16, 16, 24), (1, 1, 1)
    sim = _sim(shape, periodic, (0.0, 0.0, 1e-3), np.array([[8.2, 8.1, z]]), np.array([3.0]), np.array([fixed], np.uint8))
    for k in range(10):
        assert _wrong(sim, shape, periodic, [3.0]) == 0, k
        sim.step(2)
