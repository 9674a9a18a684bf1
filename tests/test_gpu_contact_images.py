"""Contacts of two spheres half a periodic axis apart, where the nearest image is
not always that of the integer parts' difference, against the FP64 oracle: free
of liquid, over the steps of one collision (24 steps). The library sums a step's
sub-steps in FP32, about 1e-7 of a force each, so 1e-5 of the largest velocity
change holds where a contact left out or taken through the wrong image changes
the velocity by all of it."""
import numpy as np
import pytest

import oracle as O
from paper_2301_10674_gb300 import fslbm as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_10674_gb300 import build as B
    B.build()
    F.load()


# integer parts L/2 apart: the real distance above half the axis (the nearest
# image is the other one), below it, and the same across the seam
@pytest.mark.parametrize("L,y0,y1,radius", [(10, 1.3, 6.9, 2.25), (10, 1.9, 6.3, 2.25), (10, 6.9, 1.3, 2.25),
                                            (8, 2.2, 6.7, 1.8), (9, 1.2, 5.9, 2.2)])
def test_contact_across_half_an_axis(L, y0, y1, radius):
    import torch
    shape = (24, L, 24)
    xyz = np.array([[12.2, y0, 12.3], [12.4, y1, 12.1]])
    r = np.array([radius, radius])
    p = F.fslbm_default_params()
    p.nx, p.ny, p.nz = shape
    p.bc_flags = F.PERIODIC_X | F.PERIODIC_Y
    p.g[:] = [0.0, 0.0, 0.0]
    p.liquid_height = 0.0
    sim = F.Simulation(p, torch.cuda.Stream())
    sim.add_spheres(xyz, r)
    o = O.Oracle(O.OracleParams(*shape, periodic=(1, 1, 0), omega=p.omega, g=(0.0, 0.0, 0.0), rho_gas=p.rho_gas,
                                liquid_height=0.0, rho_p=p.rho_p, restitution=p.restitution, friction=p.friction,
                                poisson=p.poisson, collision_time=p.collision_time, dem_substeps=p.dem_substeps,
                                lubrication=p.lubrication))
    o.add_spheres(xyz, r, np.zeros(2, np.uint8))
    sim.step(24)
    o.step(24)
    u, uo = sim.get(F.FIELD_P_U), o.get(O.P_U)
    assert np.abs(uo).max() > 1e-4                      # they touch
    assert np.abs(u - uo).max() < 1e-5 * np.abs(uo).max()
