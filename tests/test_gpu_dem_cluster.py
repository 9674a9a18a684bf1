"""DEM sub-steps and particle grid in one thread-block cluster against the
separate launches: the same mobile particles settle in a gas-filled box while
far-away fixed spheres bring the particle count to each side of the cluster
kernel's sizes (one CTA up to 64 particles, several with up to 512 and up to
1024 threads, and beyond its range, where the separate launches run), with ten
sub-steps and with one."""
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


def _run(mobile, total, substeps=10):
    import torch
    p = F.fslbm_default_params()
    p.nx, p.ny, p.nz = 256, 64, 64
    p.bc_flags = F.PERIODIC_X
    p.g[:] = [1e-4, 0.0, -2e-4]
    p.liquid_height = 0.0
    p.dem_substeps = substeps
    p.capacity_particles = 9000
    sim = F.Simulation(p, torch.cuda.Stream())
    rng = np.random.default_rng(3)
    # mobile spheres touching the floor and one another, some across the seam
    k = np.arange(mobile)
    xyz = np.stack([(k % 60) * 4.25, 3.0 + 4.1 * (k // 60 % 5), 2.0 + 4.0 * (k // 300)], 1)
    xyz += rng.uniform(-0.1, 0.1, xyz.shape)
    rad = rng.uniform(1.9, 2.1, mobile)
    e = np.arange(total - mobile)
    far = np.stack([1.0 + 2.9 * (e % 88), 1.5 + 2.9 * (e // 88 % 21), 45.0 + 2.9 * (e // 1848)], 1)
    sim.add_spheres(np.concatenate([xyz, far]), np.concatenate([rad, np.full(len(far), 0.4)]),
                    np.concatenate([np.zeros(mobile), np.ones(len(far))]))
    sim.step(60)
    z = F.FIELD_P_X, F.FIELD_P_U, F.FIELD_P_OMEGA
    return [sim.get(f)[:mobile] for f in z], sim.get(F.FIELD_OWNER)[:30], xyz


@pytest.mark.parametrize("mobile,total,substeps", [(1, 1, 10), (5, 33, 10), (40, 64, 10), (40, 65, 10), (300, 513, 10),
                                                   (300, 1024, 10), (600, 1025, 10), (900, 2048, 10), (300, 1000, 1)])
def test_cluster_matches_separate_launches(mobile, total, substeps):
    (xa, ua, wa), oa, start = _run(mobile, 2049 if total > 512 else 8193, substeps)
    (xb, ub, wb), ob, _ = _run(mobile, total, substeps)
    assert np.abs(xa - start).max() > 0.1
    if mobile > 5:
        assert np.abs(wa).max() > 1e-4           # they touched and turned
    # the same FP32 operations in the same order; a contraction chosen
    # differently changes the last bit of a force, a relative 1e-7 a step
    assert np.abs(xa - xb).max() < 1e-5 and np.abs(ua - ub).max() < 1e-6 and np.abs(wa - wb).max() < 1e-6
    assert np.mean(oa != ob) < 1e-4
