"""CPU: the rows of a plane that the column passes take as the particle's are exactly those that the row
test of the row passes, fl(fl(dy dy) + fl(dz dz)) > bound, does not take as outside; so no pass reads
or leaves out a row that another one did not write or needs.  Spheres from a few voxels to nearly flat
caps of 10^6 voxels radius, with centres inside and far outside the box."""
import ctypes as C

import numpy as np
import pytest

from paper_2303_13435_gb300 import api, build, inputs


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()


def ranges(shape, n):
    out = np.full((n, 2), -7, dtype=np.int32)
    api.lib().ur_selftest_row_ranges(C.byref(api.shape_desc(shape)), n, out.ctypes.data_as(C.POINTER(C.c_int32)))
    return out


def inside_rows(shape, n):
    c = np.asarray(shape.center, dtype=np.float32)
    ax = np.arange(n, dtype=np.float32)
    dy, dz = ax - c[1], ax - c[2]
    with np.errstate(invalid="ignore", over="ignore"):
        d2 = (dy * dy)[None, :] + (dz * dz)[:, None]
        return ~(d2 > np.float32(api.lib().ur_selftest_row_bound(C.byref(api.shape_desc(shape)))))


def check(shape, n):
    got, want = ranges(shape, n), inside_rows(shape, n)
    y = np.arange(n)
    for z in range(n):
        a, k = got[z]
        assert np.array_equal((y >= a) & (y < a + k), want[z]), (shape, n, z)
    return want


# caps of 10 and 45 rows in planes whose square root finds fewer
@pytest.mark.parametrize("c,size,plane,rows", [((125, 124.2559, -24188.54), 24235.54, 47, 11),
                                               ((125, 125.3356, -100949.3), 100966.3, 17, 45)])
def test_flat_caps(c, size, plane, rows):
    want = check(inputs.Shape(inputs.SHAPE_SPHERE, c, size), 250)
    assert want[plane].sum() == rows


@pytest.mark.parametrize("kind", [inputs.SHAPE_SPHERE, inputs.SHAPE_CUBE, inputs.SHAPE_OCTAHEDRON])
def test_particles_in_and_around_the_box(kind):
    rng = inputs.SplitMix64(5 + kind)
    for i in range(60):
        n = 8 + 2 * rng.randint(60)
        rot = inputs.random_rotation(rng) if i % 2 else np.eye(3, dtype=np.float32)
        c = tuple(n * rng.uniform_range(-0.5, 1.5) for _ in range(3))
        check(inputs.Shape(kind, c, float(np.float32(rng.uniform_range(0.0, 0.8) * n)), rot), n)


@pytest.mark.parametrize("axis", [1, 2])
def test_spheres_of_every_size(axis):
    """Radii of 10 to 10^6, the surface somewhere in the box along one axis."""
    rng = inputs.SplitMix64(90 + axis)
    n, reached = 96, 0
    for i in range(200):
        s = float(np.float32(10.0 ** rng.uniform_range(1.0, 6.0)))
        c = [n * rng.uniform_range(0.0, 1.0) for _ in range(3)]
        c[axis] = rng.uniform_range(-2.0, n + 2.0) + (s if i % 2 else -s)
        reached += int(check(inputs.Shape(inputs.SHAPE_SPHERE, tuple(c), s), n).any())
    assert reached > 150


def test_extremes():
    nan, inf = float("nan"), float("inf")
    for c in ((4, nan, 4), (4, 4, nan), (4, inf, 4), (4, -inf, 4), (4, 4, inf), (4, 1e30, 4), (4, -1e30, 1e30)):
        check(inputs.Shape(inputs.SHAPE_SPHERE, c, 3.0), 16)
    for s in (0.0, -3.0, 1e-30, 1e15):
        check(inputs.Shape(inputs.SHAPE_SPHERE, (8.0, 8.0, 8.0), s), 16)
