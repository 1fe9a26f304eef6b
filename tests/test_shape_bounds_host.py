"""CPU: the radius beyond which the library takes the rows of a shape as outside never cuts into its
mask.  The mask is the oracle's (float32, every step rounded); the row test is that of the kernels,
fl(fl(dy dy) + fl(dz dz)) > bound."""
import ctypes as C

import numpy as np
import pytest

from oracle import density
from paper_2303_13435_gb300 import api, build, inputs


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()


def bound(shape):
    return np.float32(api.lib().ur_selftest_row_bound(C.byref(api.shape_desc(shape))))


def outside_rows(n, shape):
    c = np.asarray(shape.center, dtype=np.float32)
    ax = np.arange(n, dtype=np.float32)
    dy, dz = ax - c[1], ax - c[2]
    return (dz * dz)[:, None] * 0 + (dy * dy)[None, :] + (dz * dz)[:, None] > bound(shape)


@pytest.mark.parametrize("kind", [inputs.SHAPE_SPHERE, inputs.SHAPE_CUBE, inputs.SHAPE_OCTAHEDRON])
def test_rows_outside_have_no_mask(kind):
    rng = inputs.SplitMix64(11 + kind)
    skipped = 0
    for i in range(60):
        n = 8 + 2 * rng.randint(24)
        rot = inputs.random_rotation(rng) if i % 3 else np.eye(3, dtype=np.float32)
        if i % 5 == 4:  # a matrix that is only nearly a rotation, or a shear
            rot = (rot * (1.0 + 1e-3 * rng.uniform())).astype(np.float32)
        c = tuple(n / 2 + rng.uniform_range(-2.0, 2.0) for _ in range(3))
        sh = inputs.Shape(kind, c, float(np.float32(rng.uniform_range(0.0, 0.7) * n)), rot)
        out = outside_rows(n, sh)
        mask = density.shape_mask(n, kind, sh.center, sh.size, sh.rot)
        assert not np.any(mask[out]), (i, n, sh)
        skipped += int(out.sum())
    assert skipped > 10000


def test_shapes_without_a_bound():
    inf = np.float32(np.inf)
    assert bound(inputs.Shape(inputs.SHAPE_ALL)) == inf
    assert bound(inputs.Shape(inputs.SHAPE_WEIGHTS)) == inf
    shear = np.array([[1, 0.5, 0], [0, 1, 0], [0, 0, 1]], dtype=np.float32)
    for kind in (inputs.SHAPE_CUBE, inputs.SHAPE_OCTAHEDRON):
        assert bound(inputs.Shape(kind, (4, 4, 4), 3.0, shear)) == inf
        assert bound(inputs.Shape(kind, (4, 4, 4), 3.0, np.zeros((3, 3), dtype=np.float32))) == inf
        assert bound(inputs.Shape(kind, (4, 4, 4), 3.0, np.full((3, 3), np.nan, dtype=np.float32))) == inf
        assert bound(inputs.Shape(kind, (4, 4, 4), float("inf"), np.eye(3, dtype=np.float32))) == inf
    assert bound(inputs.Shape(inputs.SHAPE_SPHERE, (4, 4, 4), 3.3)) == np.float32(3.3) * np.float32(3.3)
