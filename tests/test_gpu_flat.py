"""The two-pass kernels (float64, automatic launch shape) against the marched tile kernel.

Both evaluate one step from the same state; they sum in different orders, so
a population differs by a few float64 roundings of its largest term (1) per
step: 12 steps of at most 16 x 2^-53 each stay below 1e-13.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import inputs, workloads
from paper_2112_09972_gb300.lbm import DropletLBM

pytestmark = pytest.mark.gpu

TOL = 1e-13


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


# widths below, at and above the 64 threads of a CTA, ragged last CTAs, the
# smallest box, and more planes than CTAs of one plane each
BOXES = [(4, 4, 4), (37, 29, 23), (64, 5, 9), (65, 7, 6), (130, 33, 5), (16, 16, 300)]


@pytest.mark.parametrize("mrt", [None, True])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("box", BOXES)
def test_two_pass_equals_tile_kernel(built, box, periodic, mrt):
    hist = inputs.ou_gradient_history(12, 20.0, 2000.0, seed=21)
    out = []
    for tile_y in (0, 2):
        g = DropletLBM(box, min(box) / 4.0, (0.45 / 3, 0.6 / 3), 2.5, precision="fp64", periodic=periodic,
                       rho_hi=1.0, rho_lo=workloads.RHO_LO, tile_y=tile_y, mrt=mrt)
        assert (g.launch_variant() == 4) == (tile_y == 0)
        if not out:
            start = inputs.perturbed_populations(g.populations(), 1e-3, seed=5)
        g.set_populations(start)
        g.set_gradient_table(np.arange(12), hist)
        g.step(12)
        out.append((g.populations(), g.moments()))
        g.close()
    assert np.max(np.abs(out[0][0] - out[1][0])) <= TOL
    assert np.allclose(out[0][1], out[1][1], rtol=1e-12, atol=1e-9)


def test_two_pass_reads_restored_ghost_densities(built, tmp_path):
    """The ghost densities come from the loaded file, not from the context's creation."""
    mk = lambda lo: DropletLBM((20, 18, 16), 4.0, (0.5 / 3, 0.5 / 3), 3.5, precision="fp64", rho_hi=1.0, rho_lo=lo)
    a, path = mk(workloads.RHO_LO), str(tmp_path / "a.ck")
    a.step(3)
    a.save(path)
    a.step(5)
    b = mk(0.01)
    b.load(path)
    b.step(5)
    assert np.array_equal(a.populations(), b.populations())
