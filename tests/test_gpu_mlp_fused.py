"""The one-kernel forward pass (k_mlp_forward) against the layer-by-layer products, and D of special tensors.

Both forward passes take the same products in the same order with the same
rounding points, so their outputs are the same bits.  An input that is not
16-byte aligned runs layer by layer.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300.lbm import MLP

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


# the fewest and most layers it takes, every width class, one tile, several
# per SM, and rows left over for the other path
@pytest.mark.parametrize("sizes", [(64, 64, 6), (576, 256, 256, 256, 6), (128, 192, 64, 256, 128, 64, 32), (1024, 256, 1)])
@pytest.mark.parametrize("n", [128, 384, 128 * 400, 512 + 96])
def test_fused_forward_is_the_layered_one(built, sizes, n):
    net = MLP(sizes, max_batch=512, seed=3)
    rng = np.random.default_rng(4)
    net.set_normalisation(rng.normal(0, 0.1, sizes[0]), rng.uniform(0.5, 2, sizes[0]), rng.normal(0, 1, sizes[-1]),
                          rng.uniform(0.5, 2, sizes[-1]))
    net.set_params((net.get_params() + rng.normal(0, 0.01, net.param_count())).astype(np.float32))
    gen = torch.Generator(device="cuda").manual_seed(5)
    flat = torch.randn(n * sizes[0] + 1, device="cuda", generator=gen)
    x = flat[1:].reshape(n, sizes[0])  # 4 bytes off: the layered path
    y0 = torch.full((n, sizes[-1]), float("nan"), device="cuda")
    y1 = y0.clone()
    xa = x.clone()
    torch.cuda.synchronize()
    net.forward(x, y0)
    net.forward(xa, y1)
    net.sync()
    assert torch.isfinite(y0).all() and torch.equal(y0, y1)
    net.close()


def _tensors():
    rng = np.random.default_rng(9)
    out = [np.diag([2.0, 1.0, 0.5]), np.eye(3), np.zeros((3, 3)), np.diag([1.0, -1.0, 3.0]), 1e-6 * np.diag([3.0, 2, 1])]
    # the simple eigenvalue along each axis, the largest and the smallest one
    out += [np.diag(np.roll([a, 1.0, b], k)) for k in range(3) for a, b in ((1.5, 1.0), (0.7, 1.0 + 1e-6))]
    for lam in ([1.2, 1.2, 0.7], [1.5, 0.8, 0.8], [1.2, 1.2 - 1e-5, 0.7], [1 + 1e-4, 1, 1 - 2e-4], [5.0, 1.0, 1e-4],
                [1.1, 1.0, 0.9], [30.0, 20.0, 10.0], [1.0, 1e-3, 1e-5]):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        out.append((q * np.array(lam)) @ q.T)
    return out


def test_deformation_of_special_tensors(built):
    """D where the closed form is near a double root, near a sphere or near a
    vanishing eigenvalue, against numpy's eigh of the float32 tensor: 1e-12,
    the accuracy of D from M; sqrt amplifies an eigenvalue's rounding near 0."""
    net = MLP((64, 64, 6), max_batch=128, seed=0)
    x = torch.zeros((128, 64), device="cuda")
    m6 = torch.empty((128, 6), device="cuda")
    D = torch.empty(128, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for M in _tensors():
        p = np.zeros(net.param_count(), dtype=np.float32)
        p[-6:] = M[[0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]]
        net.set_params(p)
        net.deformation(x, m6, D)
        net.sync()
        m = m6.cpu().numpy().astype(np.float64)
        assert np.array_equal(m, np.tile(p[-6:].astype(np.float64), (128, 1)))
        lam = np.maximum(np.linalg.eigvalsh(m[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)), 0.0)
        s1, s3 = np.sqrt(lam[:, 2]), np.sqrt(lam[:, 0])
        ref = np.where(s1 + s3 > 0, (s1 - s3) / np.where(s1 + s3 > 0, s1 + s3, 1), 0.0)
        assert np.max(np.abs(D.cpu().numpy() - ref)) <= 1e-12
    net.close()


# both gradients of a layer and the bias sums in one launch each (512), two products but sums apart (2048), and with
# an output layer that one 32-column tile holds
@pytest.mark.parametrize("sizes,n", [((576, 256, 256, 256, 6), 512), ((576, 256, 256, 256, 6), 2048), ((64, 128, 6), 256)])
def test_grouped_training_products(built, sizes, n):
    """Against mma.sync, whose products run one launch each.  Both round to
    bfloat16 at the same points and lie within 2e-2 (relative L2) of the
    float64 model that does, so within 4e-2 of each other."""
    net = MLP(sizes, max_batch=n, seed=11)
    gen = torch.Generator(device="cuda").manual_seed(6)
    x, t = (torch.randn((n, k), device="cuda", generator=gen) for k in (sizes[0], sizes[-1]))
    torch.cuda.synchronize()
    loss, g = {}, {}
    for path in (0, 1):
        net.set_tensor_path(path)
        loss[path], g[path] = net.gradients(x, t)
    assert abs(loss[0] - loss[1]) <= 2e-3 * loss[1]
    o = 0
    for a, b in zip(sizes[:-1], sizes[1:]):
        for k in (a * b, b):
            assert np.linalg.norm(g[0][o:o + k] - g[1][o:o + k]) <= 4e-2 * np.linalg.norm(g[1][o:o + k]), (a, b, k)
            o += k
    assert o == g[0].size
    net.close()
