"""Contexts that fit only without the memory that faster launches would take.

A ballast leaves what the kernels need and a little more, less than the density array of the two-pass kernels or the
second gradient buffer of the surrogate.  Both contexts are created all the same, on the kernels that do without.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import workloads
from paper_2112_09972_gb300.lbm import MLP, DropletLBM

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


def test_surrogate_without_room_for_grouped_launches(built):
    sizes, batch, n = (576, 256, 256, 256, 6), 1 << 20, 512
    gen = torch.Generator(device="cuda").manual_seed(2)
    x, t = torch.randn((n, 576), device="cuda", generator=gen), torch.randn((n, 6), device="cuda", generator=gen)
    torch.cuda.synchronize()

    def train(net):
        grads = net.gradients(x, t)[1]
        for _ in range(3):
            net.train_step(x, t, 1e-3)
        out = grads, net.get_params()
        net.close()
        return out

    ref = train(MLP(sizes, max_batch=batch, seed=3))
    # bfloat16: hidden gradients and output gradients, input and hidden activations, one transposed gradient and one
    # transposed activation of the widest layer; the outputs in float32; weights and partial sums below 100 MB.
    # A second transposed gradient would take 1152 MB more, the transposed activations 2688 MB.
    need = 2 * batch * (3 * 256 + 32 + 576 + 3 * 256 + 2 * 576) + 4 * batch * 32
    held = _ballast(need + 500 * MB)
    try:
        net = MLP(sizes, max_batch=batch, seed=3)
        got = train(net)
    finally:
        del held
        torch.cuda.empty_cache()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
