"""The two-pass kernels of float32 and 16-bit storage against the marched kernels.

Row-tiled widths: the same node arithmetic and the same order of the centre
of mass, so the states agree bit for bit.  Other extents (float32): another
order of the same sums than the tile kernel's, so populations (largest about
1/3) differ by float32 roundings, at most some 16 x 2^-24 per step and 12
steps: 1e-5 of the largest population.
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


def _run(box, precision, steps, variant=0, tile_y=0, mrt=None, start=None):
    g = DropletLBM(box, min(box) / 5.0, (0.45 / 3, 0.55 / 3), 3.0, precision=precision, rho_hi=1.0,
                   rho_lo=workloads.RHO_LO, row_variant=variant, tile_y=tile_y, mrt=mrt)
    if start is None:
        start = inputs.perturbed_populations(g.populations(), 1e-3, seed=6)
    g.set_populations(start)
    hist = inputs.ou_gradient_history(steps, 20.0, 900.0, seed=13)
    g.set_gradient_table(np.arange(steps), hist)
    g.step(steps)
    out = (g.populations(), g.moments(), g.launch_variant())
    g.close()
    return start, out


# every width; one chunk and several, chunks of more planes than a CTA holds at
# once, ragged last chunks, the fewest rows
@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("box", [(32, 32, 32), (64, 40, 23), (64, 8, 4), (128, 16, 61), (256, 8, 37), (32, 8, 5)])
def test_rows_two_pass_bit_identical(built, box, precision):
    start, a = _run(box, precision, 15)
    _, b = _run(box, precision, 15, variant=2, start=start)
    assert a[2] == 4 and b[2] == 2
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[1], b[1])


# the collision that alone keeps float32 boxes of 2^19 to 3 * 2^18 nodes on two passes
@pytest.mark.parametrize("box", [(32, 32, 32), (64, 96, 96), (256, 8, 37)])
def test_rows_two_pass_mrt(built, box):
    start, a = _run(box, "fp32", 10, mrt=True)
    _, b = _run(box, "fp32", 10, variant=1, mrt=True, start=start)
    assert a[2] == 4 and b[2] == 1
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[1], b[1])


@pytest.mark.parametrize("mrt", [None, True])
@pytest.mark.parametrize("box", [(4, 4, 4), (37, 29, 23), (128, 5, 9), (129, 7, 6), (260, 33, 5), (16, 12, 150)])
def test_any_extents_two_pass(built, box, mrt):
    start, a = _run(box, "fp32", 12, mrt=mrt)
    _, b = _run(box, "fp32", 12, tile_y=2, mrt=mrt, start=start)
    assert a[2] == 4 and b[2] == 0
    assert np.max(np.abs(a[0] - b[0])) <= 1e-5 * np.max(np.abs(b[0]))
    assert np.allclose(a[1], b[1], rtol=1e-4, atol=1e-3 * abs(b[1][0]))
