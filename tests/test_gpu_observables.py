"""Moments, components and surface statistics on boxes of every ragged kind, against numpy and scipy.

The fields read back are float64 sums of the stored populations, the
observables' own densities float64 (or float32 pairs good to 1e-14), so both
agree to float64 rounding of sums over the box; deviation storage sums its
stored float32 density instead, which the read-back populations reproduce to
float32 rounding (19 terms of at most 2^-24 each).
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


def _state(box, precision, periodic, seed):
    """Random blobs of both phases: densities of either component between 0.05 and 1."""
    g = DropletLBM(box, 1.0, (0.5 / 3, 0.5 / 3), 3.5, precision=precision, periodic=periodic, rho_hi=1.0,
                   rho_lo=workloads.RHO_LO)
    rng = np.random.default_rng(seed)
    Lx, Ly, Lz = box
    rho = 0.05 + 0.95 * rng.random((2, 1, Lz, Ly, Lx)) ** 2
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12).reshape(1, 19, 1, 1, 1)
    g.set_populations(inputs.perturbed_populations(rho * w, 1e-2, seed))
    return g


# the smallest box, widths around a warp and a CTA, planes of few and of many
# segments, more z planes than parts
BOXES = [(4, 4, 4), (33, 7, 5), (64, 40, 9), (130, 6, 31), (31, 5, 200)]


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-12), ("fp16dev", 4e-6)])
@pytest.mark.parametrize("box", BOXES)
def test_moments_and_surface(built, box, precision, tol):
    g = _state(box, precision, False, 3)
    ra, rb, _ = g.fields()
    phi = (ra - rb) / (ra + rb)
    w = np.maximum(phi, 0.0)
    z, y, x = np.meshgrid(*[np.arange(n) - 0.5 * (n - 1) for n in reversed(box)], indexing="ij")
    ref = np.array([np.sum(w * q) for q in (1, x, y, z, x * x, x * y, x * z, y * y, y * z, z * z)])
    scale = np.array([np.sum(w * np.abs(q)) for q in (1, x, y, z, x * x, x * y, x * z, y * y, y * z, z * z)])
    assert np.all(np.abs(g.moments() - ref) <= tol * scale)
    gx, gy, gz = (0.5 * (np.roll(phi, -1, a) - np.roll(phi, 1, a))[1:-1, 1:-1, 1:-1] for a in (2, 1, 0))
    span = phi.max() - phi.min()
    area = np.sum(np.sqrt(gx * gx + gy * gy + gz * gz)) / span
    volume = np.sum(phi - phi.min()) / span
    _, a, v = g.surface_deformation()
    assert abs(a - area) <= 10 * tol * area and abs(v - volume) <= 10 * tol * volume
    # the observables leave the state as it is, and the next step does not see their scratch
    h = _state(box, precision, False, 3)
    g.components(0.1, 1)
    g.step(2)
    h.step(2)
    assert np.array_equal(g.populations(), h.populations())


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("threshold", [-0.6, 0.0, 0.35])
@pytest.mark.parametrize("box", BOXES)
def test_components(built, box, threshold, periodic):
    ndimage = pytest.importorskip("scipy.ndimage")
    g = _state(box, "fp32", periodic, 8)
    ra, rb, _ = g.fields()
    lab, n = ndimage.label((ra - rb) / (ra + rb) > threshold)
    parent = list(range(n + 1))

    def find(a):
        while parent[a] != a:
            a = parent[a]
        return a

    if periodic:
        for axis in range(3):
            first, last = np.take(lab, 0, axis).ravel(), np.take(lab, -1, axis).ravel()
            for a, b in zip(first, last):
                if a and b:
                    parent[find(a)] = find(b)
    sizes = np.zeros(n + 1, dtype=np.int64)
    for k, c in enumerate(np.bincount(lab.ravel(), minlength=n + 1)):
        if k:
            sizes[find(k)] += c
    ref = np.sort(sizes[sizes > 0])[::-1]
    count, got = g.components(threshold, 1, max_sizes=max(len(ref), 1))
    assert count == len(ref)
    assert np.array_equal(got[:count], ref)
