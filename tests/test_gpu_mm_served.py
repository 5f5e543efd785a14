"""The float32 integrator with serving warps (few trajectories) against the one without.

Both do the same arithmetic, so a trajectory's D and M are the same bits
whether it runs among few (served) or among more than one warp to a scheduler.
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


# one row, one step, records at every and at the last step only, more rows than the prefetch depth; one lane, a warp
# and a lane, one group to a CTA, full CTAs with a last one of one group
@pytest.mark.parametrize("T,substeps,every", [(1, 3, 1), (2, 1, 1), (12, 2, 1), (27, 3, 13), (30, 1, 40)])
@pytest.mark.parametrize("n", [1, 33, 4800, 32 * 161 + 5])
def test_served_is_the_plain_integrator(built, T, substeps, every, n):
    from paper_2112_09972_gb300.lbm import mm_integrate

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    base = np.stack([inputs.rescale_to_lattice(inputs.ou_gradient_history(T + 1, 30.0, 1.0, 5, box_id=k), 0.1, 16)[:T]
                     for k in range(7)], axis=1)
    base[:, 3] = 0.0  # a drop at rest stays a sphere
    base[:, 5] *= 40.0  # and one whose droplet is drawn out without bound
    few = torch.from_numpy(np.ascontiguousarray(base[:, np.arange(n) % 7])).cuda()
    many = torch.from_numpy(np.ascontiguousarray(base[:, np.arange(32 * 4 * sms + 32) % 7])).cuda()
    D0, M0 = mm_integrate(few, 6.9, 1.0, substeps=substeps, record_every=every, precision="fp32", want_M=True)
    D1, M1 = mm_integrate(many, 6.9, 1.0, substeps=substeps, record_every=every, precision="fp32", want_M=True)
    torch.cuda.synchronize()
    assert D0.shape[0] == (T - 1) // every + 1
    for a, b in ((D0, D1[:, :n]), (M0, M1[:n])):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)
