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
