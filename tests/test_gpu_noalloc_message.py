"""GPU: a plan that the built-in scratch cannot hold is refused with the bytes of the formula it names,
whatever the plan's row pitch."""
import pytest
import torch

from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 360])
def test_bytes(n):
    build.build()
    plan = api.Plan(n, 0.05, inputs.linear_edges(inputs.nyquist_q(0.05), 8))
    ed = torch.zeros((n, n, n), device="cuda")
    with pytest.raises(api.UrError, match=rf"needs {n * n * (n // 2 + 1) * 8} bytes of intermediate \(nz \* N \* \(N/2\+1\) \* 8\)"):
        api.fft_intensity_noalloc(plan, ed, api.new_bins(plan))
