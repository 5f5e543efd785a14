"""A forward pass whose outputs lie at the start of its inputs: the rows of a chunk are read before any of them is
overwritten, and the next chunk's inputs lie behind its outputs."""

import pytest

from paper_2112_09972_gb300.lbm import MLP

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


@pytest.mark.parametrize("sizes,n", [((64, 64, 32), 128 * 400), ((576, 256, 256, 6), 128 * 300 + 32)])
def test_outputs_over_the_inputs(built, sizes, n):
    net = MLP(sizes, max_batch=4096, seed=3)
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((n, sizes[0]), device="cuda", generator=gen)
    y = torch.empty((n, sizes[-1]), device="cuda")
    for _ in range(3):
        z = x.clone()
        torch.cuda.synchronize()
        net.forward(x, y)
        net.forward(z, z.view(-1)[:n * sizes[-1]].view(n, sizes[-1]))
        net.sync()
        assert torch.equal(z.view(-1)[:n * sizes[-1]], y.view(-1))
    net.close()
