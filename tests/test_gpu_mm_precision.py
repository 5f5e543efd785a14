"""How far the float32 Maffettone-Minale integrator is from the float64 one over many substeps.

A stage rounds about eight terms of the size of the relaxation rate k to 2^-24, the relaxation forgets them at that same
rate, and D takes a quarter of the difference of two diagonal entries: 2 x 8 x 2^-24 / 4 = 2.4e-7.  The gradient and its
coefficient in float32 move D (below 0.3 here) by a few 2^-24 of itself, 6e-8.  What the sums over the substeps round off
is kept beside them; dropped, it alone leaves 3e-7 after a few hundred.
"""

import numpy as np
import pytest

from paper_2112_09972_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


# served by feeding and recording warps, and not
@pytest.mark.parametrize("n", [96, 32 * 4 * 160])
def test_float32_keeps_what_its_sums_round_off(built, n):
    from paper_2112_09972_gb300.lbm import mm_integrate

    T, k = 251, np.arange(n) % 96
    hist = np.stack([inputs.ou_gradient_history(T, 200.0, 300.0, 17, box_id=q) for q in range(96)], axis=1)
    A = torch.from_numpy(np.ascontiguousarray(hist.reshape(T, 96, 9)[:, k])).cuda()
    D = [mm_integrate(A, 30.0, 1.0, substeps=10, record_every=8, precision=p).cpu().numpy() for p in ("fp32", "fp64")]
    assert 0.01 < D[1].max() < 0.3
    assert np.max(np.abs(D[0] - D[1])) <= 3e-7
