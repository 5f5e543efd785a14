"""A checkpoint's frame origin is that of the saved run, also in a context of another launch shape.

The shapes sum the droplet's centre in different orders, so the origin of the next step is taken from the file.  The
kernels here agree bit for bit on a step from the same state and origin (float64: to rounding, 1e-13).
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


@pytest.mark.parametrize("precision,box,kw", [("fp32", (37, 29, 23), {"tile_y": 2}), ("fp32", (64, 24, 40), {"z_chunk": 5}),
                                              ("bf16dev", (64, 24, 40), {"z_chunk": 5}), ("fp64", (37, 29, 23), {"tile_y": 2})])
def test_load_into_another_launch_shape(built, tmp_path, precision, box, kw):
    def make(**k):
        return DropletLBM(box, 5.0, (0.45 / 3, 0.55 / 3), 3.5, precision=precision, rho_hi=1.0,
                          rho_lo=workloads.RHO_LO, **k)

    a, b, path = make(**kw), make(), str(tmp_path / "a.ck")
    hist = inputs.ou_gradient_history(20, 20.0, 500.0, seed=9)
    a.set_gradient_table(np.arange(20), hist)
    a.step(15)
    a.save(path)
    b.load(path)
    assert a.launch_shape() != b.launch_shape()
    a.step(1)
    b.step(1)
    if precision == "fp64":
        assert np.max(np.abs(a.populations() - b.populations())) <= 1e-13
    else:
        assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
