"""GPU: launches whose dynamic shared memory lies just below the default limit of 48 KB, where the
kernel's static variables decide whether the limit has to be raised.  Each call runs in a process of
its own: a raised limit stays with the kernel for the rest of a process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


# the last bin count whose binned pass fits 48 KB without the static variables
@pytest.mark.parametrize("n,nbins", [(64, 735), (128, 751), (256, 759), (512, 759)])
def test_binned_pass(n, nbins):
    run(f"""
import torch
from paper_2303_13435_gb300 import api, inputs
plan = api.Plan({n}, 0.05, inputs.linear_edges(inputs.nyquist_q(0.05), {nbins}), z0={n // 2}, nz=1)
ed = torch.rand((1, {n}, {n}), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
bins = api.fft_intensity(plan, ed)
assert bins[1].sum().item() > 0
""")


# 195 rows of 42: 48.0 KB of lines, row terms and counts; 197 of 40: 47.0 KB, and 1136 bytes of static variables
@pytest.mark.parametrize("n,rows", [(42, 195), (40, 197)])
def test_batched_adjoint_rows(n, rows):
    run(f"""
import torch
from paper_2303_13435_gb300 import api, inputs
plan = api.Plan({n}, 0.05, inputs.linear_edges(inputs.nyquist_q(0.05), 20))
plan.set_tiles({rows}, 0)
cell = torch.rand((6, 6, 6), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
b = api.Batch([plan], cell, [inputs.Shape(inputs.SHAPE_SPHERE, ({n} / 2,) * 3, 12.0)])
b.forward()
b.dl_dmean[0].fill_(1.0)
b.backward()
assert torch.isfinite(b.dl_dcell[0]).all() and b.dl_dcell[0].abs().sum().item() > 0
""")


# 256 rows of 32: 48 KB of lines and row terms, and the stage tables (1120 bytes) beside them; 273 of 28: 46.9 KB
@pytest.mark.parametrize("n,rows", [(32, 256), (28, 273)])
def test_batched_rows(n, rows):
    run(f"""
import torch
from paper_2303_13435_gb300 import api, inputs
plan = api.Plan({n}, 0.05, inputs.linear_edges(inputs.nyquist_q(0.05), 20))
plan.set_tiles({rows}, 0)
cell = torch.rand((6, 6, 6), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
shape = inputs.Shape(inputs.SHAPE_SPHERE, ({n} / 2,) * 3, 12.0)
b = api.Batch([plan], cell, [shape])
bins = b.forward()[0]
one = api.fft_intensity_tiled(api.Plan({n}, 0.05, plan.edges), cell, shape)
ok = bins[api.BIN_COUNT] > 0
assert torch.allclose(bins[api.BIN_MEAN][ok], one[api.BIN_MEAN][ok], rtol=1e-5)
""")
