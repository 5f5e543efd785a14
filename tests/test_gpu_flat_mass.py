"""Each node's mass in the float64 two-pass kernels: the populations it stores sum to the density it collided with.

The rest population is that density less the sum of the others, a difference that float64 holds exactly (the others are
between a half and all of it), so their sum in the kernel's order is the density bit for bit, and no rounding of the
equilibrium's weights can move a component's mass from step to step.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import workloads
from paper_2112_09972_gb300.lbm import DropletLBM

pytestmark = pytest.mark.gpu

C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


def _pairs(f):
    """Sum over opposite pairs, in the kernel's order."""
    s = np.zeros_like(f[0])
    for i in range(1, 19, 2):
        s = s + (f[i] + f[i + 1])
    return s


@pytest.mark.parametrize("mrt", [None, True])
def test_a_step_keeps_each_nodes_mass(built, mrt):
    g = DropletLBM((21, 18, 16), 4.0, (0.45 / 3, 0.6 / 3), workloads.G_COUPLING, precision="fp64", periodic=True,
                   rho_hi=1.0, rho_lo=workloads.RHO_LO, mrt=mrt)
    g.step(5)
    assert g.launch_variant() == 4
    f = g.populations()
    g.step(1)
    out = g.populations()
    g.close()
    for s in range(2):
        pulled = [np.roll(f[s, i], C[i][::-1], axis=(0, 1, 2)) for i in range(19)]
        rho = pulled[0]
        for i in range(1, 19, 2):
            rho = rho + (pulled[i] + pulled[i + 1])
        assert np.array_equal(out[s, 0] + _pairs(out[s]), rho)
