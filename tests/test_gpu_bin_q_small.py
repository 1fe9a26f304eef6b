"""GPU: Q binning of a stored intensity on small grids costs less than on larger ones."""
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


def setup(n, nbins, log=True):
    dx = 0.05
    top = inputs.nyquist_q(dx)
    edges = inputs.log_edges(2 * np.pi / (n * dx), top, nbins) if log else inputs.linear_edges(top, nbins)
    gen = torch.Generator(device="cuda").manual_seed(n)
    return api.Plan(n, dx, edges), -torch.log(torch.rand((n, n, n // 2 + 1), device="cuda", generator=gen))


def time(plan, half):
    """Of one call, in a graph of ten; the least of five."""
    with torch.cuda.stream(torch.cuda.Stream()):
        api.bin_q(plan, half)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(10):
            api.bin_q(plan, half)
    t = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        graph.replay()
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return min(t)


def test_a_smaller_grid_takes_less_time():
    # 48^3 has a sixteenth of the elements of 126^3; with serial walks of four steps it took longer
    assert time(*setup(48, 771)) < 0.9 * time(*setup(126, 771))


def test_the_unit_does_not_matter():
    """Values of 1e-30 took the histogram's float64 additions one by one, which was nine times as long; summed
    over the eight values of a step it has to be less than three times as long."""
    plan, half = setup(128, 40)
    assert time(plan, half * 1e-30) < 3 * time(plan, half)


@pytest.mark.parametrize("n", [8, 48, 140])
@pytest.mark.parametrize("power", [-140, -120, -100, -60, 60, 90, 120])
def test_scaled_sums(n, power):
    """An intensity times a power of two: sums of runs held to 48 bits, so 1e-12, on either scale."""
    plan, half = setup(n, 60)
    half = (half * 2.0 ** min(power, 0)).float().double() * 2.0 ** -min(power, 0)  # exact where it is subnormal
    half[0, 0, 0] *= 2.0 ** 6
    want = api.bin_q(plan, half.float())
    got = api.bin_q(plan, (half * 2.0 ** power).float())
    assert torch.equal(got[api.BIN_COUNT], want[api.BIN_COUNT])
    for f, p in ((api.BIN_SUM_I, power), (api.BIN_SUM_I2, 2 * power)):
        assert torch.allclose(got[f] * 2.0 ** -p, want[f], rtol=1e-12, atol=0)
