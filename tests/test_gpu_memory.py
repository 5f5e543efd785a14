"""A box that fits only without the memory that its faster kernels would take.

A ballast leaves what the kernels need and a little more, less than the density array of the two-pass kernels.  The box is
created all the same, on the kernel that does without.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import workloads
from paper_2112_09972_gb300.lbm import DropletLBM

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
MB = 1 << 20


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


def _ballast(leave):
    """Takes the device's memory but for about `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    if free < leave + 64 * MB:
        pytest.skip("the device is in use")
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


def _box(n, steps, tile_y=0):
    g = DropletLBM((n, n, n), n / 8, (1 / 6, 1 / 6), workloads.G_COUPLING, precision="fp64", rho_hi=workloads.RHO_HI,
                   rho_lo=workloads.RHO_LO, tile_y=tile_y)
    g.step(steps)
    g.sync()
    return g


def test_box_without_room_for_its_densities(built):
    n = 128
    for ty in (0, 2):
        _box(32, 2, ty).close()  # the kernels are loaded
    # the two buffers: 38 populations of 130 x 130 padded rows, 136 wide (x0 = 4, whole sectors); densities 35 MB
    buffers = 2 * 38 * 130 * 130 * 136 * 8
    held = _ballast(buffers + 20 * MB)
    try:
        g = _box(n, 3)
    finally:
        del held
        torch.cuda.empty_cache()
    assert g.launch_variant() == 0
    h = _box(n, 3)
    assert h.launch_variant() == 4
    assert np.max(np.abs(g.populations() - h.populations())) <= 1e-13
    g.close()
    h.close()
