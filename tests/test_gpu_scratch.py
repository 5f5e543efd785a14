"""The observables' scratch, which lies in the buffer of the next step's state, is seen by nothing.

The kernels that the boxes of tests/test_gpu_observables.py do not reach: the row kernels' three variants, which copy
whole padded rows, and the tile kernel in the periodic mode; and the checkpoint file of 16-bit storage, which holds the
raw buffer.
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


def _box(box, precision, **kw):
    g = DropletLBM(box, min(box) / 5.0, (0.45 / 3, 0.55 / 3), 3.5, precision=precision, rho_hi=1.0,
                   rho_lo=workloads.RHO_LO, **kw)
    g.set_gradient_table(np.arange(12), inputs.ou_gradient_history(12, 20.0, 1500.0, seed=4))
    return g


def _look(g):
    g.fields()
    g.components(0.0, 1)
    g.surface_deformation()


@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("box,kw", [((64, 16, 20), {"row_variant": 1}), ((64, 16, 20), {"row_variant": 2}),
                                    ((128, 24, 13), {"row_variant": 2}), ((64, 16, 20), {"row_variant": 3}),
                                    ((64, 16, 20), {"row_variant": 0}), ((37, 20, 18), {"periodic": True})])
def test_steps_do_not_see_the_scratch(built, box, kw, precision):
    g, h = _box(box, precision, **kw), _box(box, precision, **kw)
    for n in (1, 2, 1, 3):
        g.step(n)
        h.step(n)
        _look(g)
    assert np.array_equal(g.populations(), h.populations())
    assert np.array_equal(g.moments(), h.moments())
    g.close()
    h.close()


@pytest.mark.parametrize("precision", ["fp16dev", "bf16dev"])
@pytest.mark.parametrize("box,kw", [((37, 20, 18), {}), ((64, 16, 20), {}), ((64, 16, 20), {"periodic": True})])
def test_equal_states_give_equal_files(built, tmp_path, box, kw, precision):
    g, h = _box(box, precision, **kw), _box(box, precision, **kw)
    paths = [tmp_path / n for n in ("g", "h", "again")]
    g.step(4)
    _look(g)
    g.step(1)
    h.step(5)
    g.save(str(paths[0]))
    h.save(str(paths[1]))
    g.load(str(paths[1]))
    g.save(str(paths[2]))
    assert paths[0].read_bytes() == paths[1].read_bytes() == paths[2].read_bytes()
    g.step(3)
    h.step(3)
    assert np.array_equal(g.populations(), h.populations())
    g.close()
    h.close()
