"""GPU: at 1024 an adjoint for the cell alone has kernels of its own (rows across warps, 32 values per
column and thread with a range of planes); it has to equal the adjoint of the whole box."""
import numpy as np
import pytest
import torch

from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

N = 1024


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


@pytest.mark.parametrize("kind,size,shift", [(inputs.SHAPE_SPHERE, 100.0, 0.3), (inputs.SHAPE_CUBE, 60.0, -150.0),
                                             (inputs.SHAPE_OCTAHEDRON, 9.0, 511.0), (inputs.SHAPE_SPHERE, 700.0, 2.0)])
@pytest.mark.parametrize("ucell,origin", [(64, (0, 0, 0)), (37, (36, 9, 2))])
def test_cell_adjoint_alone_equals_the_whole_box(kind, size, shift, ucell, origin):
    dx = 0.05
    rot = inputs.random_rotation(inputs.SplitMix64(kind))
    sh = inputs.Shape(kind, (N / 2 + shift, N / 2 - shift, N / 2 + 0.5 * shift), size, rot)
    edges = inputs.log_edges(2 * np.pi / (N * dx), 0.9 * inputs.nyquist_q(dx), 64)
    plan = api.Plan(N, dx, edges)
    gen = torch.Generator(device="cuda").manual_seed(ucell)
    cell = torch.rand((ucell, ucell, ucell), device="cuda", generator=gen)
    ws = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
    bins = api.fft_intensity_tiled(plan, cell, sh, origin=origin, ws=ws)
    g = torch.randn(64, dtype=torch.float64, device="cuda", generator=gen) * (bins[api.BIN_COUNT] > 0)
    full, _ = api.backward(plan, g, bins, cell, sh, ws, origin=origin)
    alone, none = api.backward(plan, g, bins, cell, sh, ws, origin=origin, want_mask=False)
    assert none is None and full.norm().item() > 0
    # sums of the same float32 gradients in another order: a few thousand terms per cell voxel
    assert (alone - full).norm().item() <= 2e-6 * full.norm().item()
    del ws
    torch.cuda.empty_cache()
