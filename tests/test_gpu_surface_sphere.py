"""Surface statistics of droplets that are nearly spheres, where Eq. 17's D is the root of a small difference.

phi of a float32 state is a pair of float32 good to 2^-44 of its largest value 1: every |grad phi| is good to sqrt(3)
2^-44, the volume's summand to 2 x 2^-44.  So N nodes leave at most N sqrt(3) 2^-44 of the gradients' sum, 2 N 2^-44 of
the volume's, and of D^2 = 1 - (36 pi V^2)^(1/3) / area the relative errors' sum.  Against float64 sums of the
populations read back.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import inputs, workloads
from paper_2112_09972_gb300.lbm import DropletLBM

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -44


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


@pytest.mark.parametrize("box,radius", [((64, 64, 64), 12.0), ((256, 32, 64), 6.8), ((48, 45, 38), 7.0),
                                        ((128, 128, 128), 16.0), ((23, 256, 200), 4.8)])
def test_surface_of_a_near_sphere(built, box, radius):
    g = DropletLBM(box, radius, (1 / 6, 1 / 6), workloads.G_COUPLING, precision="fp32", rho_hi=workloads.RHO_HI,
                   rho_lo=workloads.RHO_LO, xi=1.0)
    hist = inputs.rescale_to_lattice(inputs.ou_gradient_history(400, 10.0, 1.0, 31), 0.1, max(box))
    g.set_gradient_table(200 * np.arange(400), hist)
    g.step(24)
    rho = g.populations().sum(axis=1)
    phi = (rho[0] - rho[1]) / (rho[0] + rho[1])
    gx, gy, gz = (0.5 * (np.roll(phi, -1, a) - np.roll(phi, 1, a))[1:-1, 1:-1, 1:-1] for a in (2, 1, 0))
    span = phi.max() - phi.min()
    area, volume = np.sum(np.sqrt(gx * gx + gy * gy + gz * gz)) / span, np.sum(phi - phi.min()) / span
    D, a, v = g.surface_deformation()
    g.close()
    rel_a, rel_v = np.sqrt(3) * EPS * phi.size / (span * area) + EPS, 2 * EPS * phi.size / (span * volume) + EPS
    assert abs(a - area) <= rel_a * area
    assert abs(v - volume) <= rel_v * volume
    ratio = np.cbrt(36.0 * np.pi * volume * volume) / area
    assert abs(D * D - max(0.0, 1.0 - ratio)) <= ratio * (rel_a + 2 / 3 * rel_v)
