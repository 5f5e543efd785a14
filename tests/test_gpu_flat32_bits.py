"""The two-pass kernels of float32 boxes of any extents against the tile kernel, bit for bit.

Both form every density, collision and centre-of-mass sum with the same operations in the same order, so states and
moments are equal and not only close: a call's D is as far from the 64-bit result as the tile kernel leaves it.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import inputs, workloads
from paper_2112_09972_gb300.lbm import DropletLBM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


def _tile_rows(box):
    """Rows of the tile that is taken when no launch shape is asked for: 512 threads."""
    width = box[0] if box[0] <= 512 else 128
    return max(1, min(512 // width, box[1]))


def _run(box, radius, mrt, tile_y, steps):
    g = DropletLBM(box, radius, (0.45 / 3, 0.55 / 3), 3.5, precision="fp32", rho_hi=1.0, rho_lo=workloads.RHO_LO,
                   tile_y=tile_y, mrt=mrt)
    hist = inputs.ou_gradient_history(steps, 20.0, 1500.0, seed=13)
    g.set_gradient_table(np.arange(steps), hist)
    g.step(steps)
    out = g.populations(), g.moments(), g.deformation()[0], g.launch_variant(), g.launch_shape()
    g.close()
    return out


# the smallest box; tiles with ragged warps, ragged last rows and several tiles to a row; one z chunk and several;
# small droplets in uneven boxes, whose D shows a rounding most
@pytest.mark.parametrize("mrt", [None, True])
@pytest.mark.parametrize("box", [(4, 4, 4), (37, 29, 23), (128, 5, 9), (129, 7, 6), (260, 33, 5), (16, 12, 150),
                                 (41, 46, 18), (36, 33, 16), (60, 22, 169), (33, 118, 56), (520, 9, 6)])
def test_any_extents_are_the_tile_kernels_bits(built, box, mrt):
    radius = max(1.0, 0.2 * min(box))
    a = _run(box, radius, mrt, 0, 20)
    b = _run(box, radius, mrt, _tile_rows(box), 20)
    assert a[3] == 4 and b[3] == 0 and a[4] == b[4]
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[1], b[1])
    assert np.array_equal(a[2], b[2], equal_nan=True)
