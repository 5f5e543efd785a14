"""lbm_components of a context with a latched condition: the components are returned beside the status."""

import ctypes

import numpy as np
import pytest

from paper_2112_09972_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session")
def built():
    from paper_2112_09972_gb300 import build

    return build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16dev"])
def test_components_after_the_mach_guard(built, precision):
    w = workloads.C1_PARITY
    g = lbm.DropletLBM((24, 20, 18), 4.0, w.visc, w.G, precision=precision, rho_lo=w.rho_lo, mach_limit=0.1)
    want = g.components(0.0, 1, max_sizes=4)
    A = np.zeros(9)
    A[1] = 0.02  # 0.2 at the walls, above 0.1 / sqrt(3)
    g.set_gradient(A, 0)
    g.step(1)
    count, sizes = ctypes.c_int32(-1), np.full(4, -1, dtype=np.int64)
    status = lbm.load_library().lbm_components(g._h, 0.0, 1, ctypes.byref(count),
                                               sizes.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)), 4)
    assert status == -5  # LBM_EMACH
    assert count.value == want[0] == 1
    assert 0 < sizes[0] and not sizes[1:].any()
    g.close()
