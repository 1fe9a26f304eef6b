"""CPU: the shape descriptor takes the first three coordinates of a centre and refuses a shorter one."""
import numpy as np
import pytest

from paper_2303_13435_gb300 import api, inputs


@pytest.mark.parametrize("center", [(1.0, 2.0, 3.0), (1.0, 2.0, 3.0, 1.0), np.array([1, 2, 3])])
def test_center(center):
    d = api.shape_desc(inputs.Shape(inputs.SHAPE_CUBE, center, 4.5, np.arange(9.0).reshape(3, 3)))
    assert (d.kind, list(d.center), d.size, list(d.rot)) == (inputs.SHAPE_CUBE, [1.0, 2.0, 3.0], 4.5, list(range(9)))


@pytest.mark.parametrize("center", [(), (1.0,), (1.0, 2.0), 1.0])
def test_short_center(center):
    with pytest.raises(IndexError):
        api.shape_desc(inputs.Shape(inputs.SHAPE_SPHERE, center, 4.5))
