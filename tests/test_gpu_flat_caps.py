"""GPU: spheres so large that the box holds a nearly flat cap.  The rows of the cap's last planes are
decided by float32 roundings of very large squares, and every pass has to decide them alike: the fused
forward equals the one that reads the stored density, and an adjoint for the cell alone equals the
adjoint of the whole box."""
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


@pytest.mark.parametrize("n", [250, 256])
@pytest.mark.parametrize("c,size", [((125, 124.2559, -24188.54), 24235.54), ((125, 125.3356, -100949.3), 100966.3),
                                    ((125, -24188.54, 124.2559), 24235.54)])
def test_forward_and_cell_adjoint(n, c, size):
    dx = 0.05
    sh = inputs.Shape(inputs.SHAPE_SPHERE, c, size)
    rng = np.random.default_rng(n)
    cell = torch.from_numpy(rng.random((16, 16, 16)).astype(np.float32)).cuda()
    edges = inputs.log_edges(0.7 * 2 * np.pi / (n * dx), 0.9 * inputs.nyquist_q(dx), 30)
    plan = api.Plan(n, dx, edges)
    ws = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
    ws.fill_(0xFF)  # NaN wherever a pass reads what no pass wrote
    F = [torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda") for _ in range(2)]
    api.fft_intensity_tiled(plan, cell, sh, ws=ws, F_out=F[0])
    ed = api.build_density(n, cell, sh)
    assert 0 < torch.count_nonzero(ed).item() < n ** 3 // 2
    api.fft_intensity(plan, ed, F_out=F[1])
    assert torch.equal(torch.view_as_real(F[0]), torch.view_as_real(F[1]))
    ws.fill_(0xFF)
    bins = api.fft_intensity_tiled(plan, cell, sh, ws=ws)
    g = torch.from_numpy(rng.standard_normal(len(edges) - 1)).cuda() * (bins[0] > 0)
    alone, _ = api.backward(plan, g, bins, cell, sh, ws, want_mask=False)
    alone = alone.cpu().numpy()
    full, _ = api.backward(plan, g, bins, cell, sh, ws)
    full = full.cpu().numpy()
    # sums of the same float32 gradients in another order
    assert np.linalg.norm(alone - full) <= 2e-6 * np.linalg.norm(full)
