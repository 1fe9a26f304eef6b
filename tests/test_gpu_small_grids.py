"""GPU: small mixed-radix grids, on both sides of the lines between their kernels: stored rows read by
the first stage or staged, adjoint rows of one or several cell rows per block, voxel weights in the
adjoint rows, and pairs of lattice samples at the ends of odd half rows."""
import numpy as np
import pytest
import torch

from _cases import GRAD_RTOL, normwise, oracle_grads
from oracle import density
from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu

DX = 0.05


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def edges_of(n):
    return inputs.log_edges(0.7 * 2 * np.pi / (n * DX), 0.9 * inputs.nyquist_q(DX), 30)


@pytest.mark.parametrize("n", [8, 10, 30, 42, 70, 90])
@pytest.mark.parametrize("kind", [inputs.SHAPE_SPHERE, inputs.SHAPE_CUBE, inputs.SHAPE_ALL])
def test_lattice(n, kind):
    rng = np.random.default_rng(n)
    cell = rng.standard_normal((11, 11, 11)).astype(np.float32)
    sh = inputs.Shape(kind, (n / 2 + 0.3, n / 2 - 0.8, n / 2), float(np.float32(0.3 * n)),
                      inputs.random_rotation(inputs.SplitMix64(4)))
    lat = (inputs.random_rotation(inputs.SplitMix64(11)), (0.37, 5.21, 2.5))
    for dtype in ("f32", "f16"):
        want = density.tile_mask_density(n, cell, kind, sh.center, sh.size, sh.rot, lattice=lat, out_dtype=dtype)
        span = torch.tensor([2 ** 31 - 1, -1], dtype=torch.int32, device="cuda")
        ed = api.build_density(n, dev(cell), sh, out_dtype=dtype, nz_range=span, lattice=lat)
        assert ed.cpu().numpy().tobytes() == want.tobytes()
        assert tuple(span.tolist()) == tuple(density.nonzero_plane_range(want))
        part = api.build_density(n, dev(cell), sh, z_begin=n // 2, z_count=2, out_dtype=dtype, lattice=lat)
        assert torch.equal(part, ed[n // 2:n // 2 + 2])
        if dtype == "f32":  # the same transforms of the same rows, stored and generated: the spectra are equal
            plan = api.Plan(n, DX, edges_of(n))
            F = [torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda") for _ in range(2)]
            api.fft_intensity(plan, ed, F_out=F[0])
            api.fft_intensity_tiled(plan, dev(cell), sh, lattice=lat, F_out=F[1])
            assert torch.equal(torch.view_as_real(F[0]), torch.view_as_real(F[1]))


@pytest.mark.parametrize("n", [8, 10, 30, 42, 90])
@pytest.mark.parametrize("ucell,origin", [(3, (1, 2, 0)), (16, (0, 0, 0)), (90, (89, 7, 30))])
def test_weights_adjoint(n, ucell, origin):
    rng = np.random.default_rng(n + ucell)
    cell = rng.random((ucell, ucell, ucell)).astype(np.float32)
    w = (rng.random((n, n, n)) * (rng.random((n, n, n)) < 0.7)).astype(np.float32)
    edges = edges_of(n)
    plan = api.Plan(n, DX, edges)
    ws = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
    sh = inputs.Shape(inputs.SHAPE_WEIGHTS)
    bins = api.fft_intensity_tiled(plan, dev(cell), sh, origin=origin, weights=dev(w), ws=ws)
    count = bins[api.BIN_COUNT].cpu().numpy()
    g = rng.standard_normal(len(edges) - 1) * (count > 0)
    du, dm = api.backward(plan, dev(g), bins, dev(cell), sh, ws, origin=origin, weights=dev(w))
    alone, _ = api.backward(plan, dev(g), bins, dev(cell), sh, ws, origin=origin, weights=dev(w), want_mask=False)
    rho = density.tiled_cell(n, cell, origin) * w
    gu, gm = oracle_grads(rho.astype(np.float64), cell, w, DX, edges, g, count.astype(np.int64), origin)
    assert normwise(du.cpu().numpy(), gu) < GRAD_RTOL
    assert normwise(alone.cpu().numpy(), gu) < GRAD_RTOL
    assert normwise(dm.cpu().numpy(), gm) < GRAD_RTOL
