"""GPU: an adjoint for the cell alone transforms only the planes and rows that the particle's mask can
reach; it has to equal the adjoint of the whole box, on both engines, and the forward that leaves the
rows outside the particle out has to equal the one that reads the stored density."""
import math

import numpy as np
import pytest
import torch

from _cases import GRAD_RTOL, normwise, oracle_grads
from oracle import density
from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

SPHERE, CUBE, OCTA, ALL = inputs.SHAPE_SPHERE, inputs.SHAPE_CUBE, inputs.SHAPE_OCTAHEDRON, inputs.SHAPE_ALL


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def particle(n, kind, frac, rot, shift):
    rng = inputs.SplitMix64(n + kind)
    r = inputs.random_rotation(rng) if rot else np.eye(3, dtype=np.float32)
    rc = 0.5 * frac * n
    size = rc / math.sqrt(3.0) if kind == CUBE else rc
    c = (n / 2 + shift, n / 2 - shift, n / 2 + 0.5 * shift)
    return inputs.Shape(kind, c, float(np.float32(size)), r)


# edges of both engines, single-stage transforms among them (8, 10)
@pytest.mark.parametrize("n", [8, 10, 48, 64, 90, 128, 150])
@pytest.mark.parametrize("kind,frac,rot,shift", [(SPHERE, 0.5, 0, 0.3), (CUBE, 0.6, 1, 0.0), (OCTA, 0.9, 1, 1.2),
                                                 (CUBE, 0.7, 0, 0.5), (SPHERE, 1.4, 0, 2.0), (SPHERE, 0.02, 0, 0.4)])
@pytest.mark.parametrize("ucell,origin", [(16, (0, 0, 0)), (7, (6, 9, 2))])
def test_cell_adjoint_alone_equals_the_whole_box(n, kind, frac, rot, shift, ucell, origin):
    dx = 0.05
    sh = particle(n, kind, frac, rot, shift)
    rng = np.random.default_rng(n + ucell)
    cell = rng.random((ucell, ucell, ucell)).astype(np.float32)
    edges = inputs.log_edges(0.7 * 2 * np.pi / (n * dx), 0.9 * inputs.nyquist_q(dx), 30)
    plan = api.Plan(n, dx, edges)
    ws = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
    # the same density through the same transforms: the spectra are equal
    F = [torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda") for _ in range(2)]
    bins = api.fft_intensity_tiled(plan, dev(cell), sh, origin=origin, ws=ws, F_out=F[0])
    api.fft_intensity(plan, api.build_density(n, dev(cell), sh, origin=origin), F_out=F[1])
    assert torch.equal(torch.view_as_real(F[0]), torch.view_as_real(F[1]))
    # (without F the forward leaves columns beyond the last bin out)
    bins = api.fft_intensity_tiled(plan, dev(cell), sh, origin=origin, ws=ws)
    g = rng.standard_normal(len(edges) - 1)
    g[bins[0].cpu().numpy() == 0] = 0.0
    full, dm = api.backward(plan, dev(g), bins, dev(cell), sh, ws, origin=origin)
    alone, none = api.backward(plan, dev(g), bins, dev(cell), sh, ws, origin=origin, want_mask=False)
    assert none is None
    a, f = alone.cpu().numpy(), full.cpu().numpy()
    if n <= 64:
        mask = density.shape_mask(n, kind, sh.center, sh.size, sh.rot)
        u = density.tiled_cell(n, cell, origin)
        gu, gm = oracle_grads((u * mask).astype(np.float64), cell, mask, dx, edges, g, bins[0].cpu().numpy().astype(np.int64),
                              origin)
        if np.linalg.norm(gu) > 0:
            assert normwise(f, gu) < GRAD_RTOL
            assert normwise(dm.cpu().numpy(), gm) < GRAD_RTOL
    # sums of the same float32 gradients in another order: a few thousand terms per cell voxel
    assert np.linalg.norm(a - f) <= 2e-6 * np.linalg.norm(f)


@pytest.mark.parametrize("n,nb", [(96, 40), (128, 64)])
@pytest.mark.parametrize("rows,cols", [(0, 0), (3, 5), (64, 1)])
def test_batch_adjoint_with_and_without_mask_gradient(n, nb, rows, cols):
    dx = 0.05
    edges = inputs.log_edges(2 * np.pi / (n * dx), inputs.nyquist_q(dx), nb)
    shapes = [particle(n, k, f, 1, 0.4) for k, f in ((SPHERE, 0.4), (CUBE, 0.5), (OCTA, 0.3))]
    shapes.append(inputs.Shape(ALL))
    cell = dev(np.random.default_rng(2).random((12, 12, 12)).astype(np.float32))
    plans = [api.Plan(n, dx, edges) for _ in shapes]
    for p in plans:
        p.set_tiles(min(rows, 4096 // (n // 2)), min(cols, 4096 // n))
    out = []
    for mask in (False, True):
        b = api.Batch(plans, cell, shapes, with_mask_grad=mask)
        b.forward()
        for i, g in enumerate(b.dl_dmean):
            g.copy_(torch.linspace(-1, 1, nb, dtype=torch.float64) * (b.bins[i][0].cpu() > 0))
        b.backward()
        out.append([t.cpu().numpy() for t in b.dl_dcell])
        if mask:
            for i, (p, sh) in enumerate(zip(plans, shapes)):
                ws = p.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
                bins = api.fft_intensity_tiled(p, cell, sh, ws=ws)
                du, dm = api.backward(p, b.dl_dmean[i], bins, cell, sh, ws)
                assert normwise(b.dl_dmask[i].cpu().numpy(), dm.cpu().numpy()) < 5e-6
                assert normwise(b.dl_dcell[i].cpu().numpy(), du.cpu().numpy()) < 5e-6
    for a, f in zip(*out):
        assert np.linalg.norm(a - f) <= 2e-6 * np.linalg.norm(f)
