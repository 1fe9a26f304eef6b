"""GPU: column passes in pairs of columns (power-of-two edges up to 512) at their edges: odd plane
counts (a last plane without a partner), slabs at either end of the box, the half spectrum, F given to
the adjoint, and the unpadded intermediate of plans that only just fit the built-in scratch."""
import numpy as np
import pytest
import torch

from _cases import GRAD_RTOL, compare_bins, normwise, oracle_forward, oracle_grads
from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n", [64, 128, 256])
@pytest.mark.parametrize("z0,nz", [(0, 1), (0, 33), (29, 35), (1, 62), (0, 64)])
def test_plane_slabs(n, z0, nz):
    rho = inputs.random_density(n, 3 + z0, (z0, nz))
    dx = 0.05
    edges = inputs.log_edges(2 * np.pi / (n * dx), inputs.nyquist_q(dx), 90)
    plan = api.Plan(n, dx, edges, z0=z0, nz=nz)
    F = torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    gb = api.fft_intensity(plan, dev(rho[z0:z0 + nz]), F_out=F).cpu().numpy()
    r64 = rho.astype(np.float64)
    ob = oracle_forward(r64, dx, edges)
    compare_bins(gb, ob, r64, f"slab {n} {z0}+{nz}")
    want = np.fft.rfftn(r64) / n ** 3
    # float32 transforms: a few eps of the root mean square per radix-8 stage
    assert normwise(F.cpu().numpy().view(np.float32), want.view(np.float64).astype(np.float64)) < 2e-6


@pytest.mark.parametrize("n,linear", [(64, True), (128, False), (256, False)])
@pytest.mark.parametrize("keep_f", [False, True])
def test_adjoint_of_a_whole_box(n, linear, keep_f):
    """Every column scaled (edges beyond the last k^2) and a cut-off inside the spectrum."""
    dx = 0.05
    for top in (3.0, 0.7):
        q = top * inputs.nyquist_q(dx)
        edges = inputs.linear_edges(q, 50) if linear else inputs.log_edges(0.5 * 2 * np.pi / (n * dx), q, 70)
        rng = np.random.default_rng(n)
        cell = rng.random((16, 16, 16)).astype(np.float32)
        shape = inputs.Shape(inputs.SHAPE_ALL)
        plan = api.Plan(n, dx, edges)
        ws = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
        F = torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda") if keep_f else None
        bins = api.fft_intensity_tiled(plan, dev(cell), shape, F_out=F, ws=ws)
        g = rng.standard_normal(len(edges) - 1)
        g[bins[0].cpu().numpy() == 0] = 0.0
        du, dm = api.backward(plan, dev(g), bins, dev(cell), shape, ws, F=F)
        i = np.arange(n) % 16
        rho = cell[np.ix_(i, i, i)].astype(np.float64)
        gu, gm = oracle_grads(rho, cell, np.ones((n, n, n)), dx, edges, g, bins[0].cpu().numpy().astype(np.int64))
        assert normwise(du.cpu().numpy(), gu) < GRAD_RTOL
        assert normwise(dm.cpu().numpy(), gm) < GRAD_RTOL


def test_plan_that_just_fits_the_builtin_scratch():
    n, nz = 256, 254  # nz N (N/2+1) 8 bytes = 64 MiB - 4 KiB
    dx = 0.05
    edges = inputs.log_edges(2 * np.pi / (n * dx), inputs.nyquist_q(dx), 64)
    plan = api.Plan(n, dx, edges, z0=1, nz=nz)
    assert plan.workspace_size(api.UR_WS_FORWARD) <= api.noalloc_scratch_bytes()
    rho = inputs.random_density(n, 5, (1, nz))
    bins = api.fft_intensity_noalloc(plan, dev(rho[1:1 + nz]), api.new_bins(plan)).cpu().numpy()
    r64 = rho.astype(np.float64)
    compare_bins(bins, oracle_forward(r64, dx, edges), r64, "unpadded rows")
