"""GPU: densities in units whose zero-frequency intensity squared does not fit float32: the bin that
holds that one voxel keeps a finite sum of squares."""
import numpy as np
import pytest
import torch

from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


@pytest.mark.parametrize("n", [64, 128, 256])
def test_uniform_box(n):
    u = 1e8  # |F(0)|^2 / N^3 = 1e16 N^3 > 2e21, its square > 4e42
    dx = 0.05
    edges = inputs.linear_edges(inputs.nyquist_q(dx), n)  # the first bin: k = 0 alone
    plan = api.Plan(n, dx, edges)
    cell = torch.full((4, 4, 4), u, device="cuda")
    bins = api.fft_intensity_tiled(plan, cell, inputs.Shape(inputs.SHAPE_ALL)).cpu().numpy()
    assert bins[0, 0] == 1
    # I(0) = u^2; float32 transforms of a constant: a few eps
    assert abs(bins[1, 0] / u ** 2 - 1) < 2e-6
    assert abs(bins[2, 0] / u ** 4 - 1) < 4e-6
    assert abs(bins[4, 0] / u ** 2 - 1) < 2e-6
    # more than one voxel: SEM is defined, and finite
    many = bins[0] > 1
    assert np.isfinite(bins[1:3, bins[0] > 0]).all() and np.isfinite(bins[5, many]).all()
