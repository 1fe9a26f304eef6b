"""GPU: the FP16 block sums in 16-byte groups (factors 2, 4, 8 and 16, edges that are multiples of 8)."""
import numpy as np
import pytest
import torch

from oracle import density
from paper_2303_13435_gb300 import api, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


def halves(n, top, seed):
    """Magnitudes with bits below `top`, subnormals among them, both signs."""
    rng = np.random.default_rng(seed)
    bits = rng.integers(0, top, (n, n, n), dtype=np.uint16) | (rng.integers(0, 2, (n, n, n), dtype=np.uint16) << 15)
    return bits.view(np.float16)


@pytest.mark.parametrize("f,n_src", [(2, 8), (2, 24), (2, 128), (2, 136), (4, 8), (4, 24), (4, 40), (8, 8), (8, 24), (8, 40),
                                     (16, 16), (16, 48), (16, 80)])
@pytest.mark.parametrize("out_dtype", ["f16", "f32"])
def test_block_sums_are_exact(f, n_src, out_dtype):
    # every finite half (FP16 sums overflow to infinity), and halves whose sums stay finite
    for top in (0x7C00, 0x7C00 - (3 * int(np.log2(f)) << 10)):
        ed = halves(n_src, top, f + n_src)
        for n_out in (n_src // f, n_src // f + 3, 8 * ((n_src // f + 7) // 8)):
            with np.errstate(over="ignore"):
                want = density.zoom_out(ed, f, n_out, out_dtype=out_dtype)
            got = api.zoom_density(torch.from_numpy(ed).cuda(), f, n_out, out_dtype=out_dtype).cpu().numpy()
            # a zero sum has no sign bit on the GPU (integer sum)
            assert (got + np.array(0, got.dtype)).tobytes() == (want + np.array(0, want.dtype)).tobytes(), (top, n_out)


@pytest.mark.parametrize("f", [2, 4, 8, 16])
def test_values_that_are_not_finite(f):
    """As the sums of a source that does not start on a 16-byte boundary, which takes value by value."""
    ed = halves(144, 0x5C00, f)
    ed[0, 1, 2], ed[20, 21, 47], ed[33, 0, 15], ed[33, 1, 14] = np.inf, -np.inf, np.nan, np.inf
    src = torch.from_numpy(ed).cuda()
    flat = torch.empty(144 ** 3 + 1, dtype=torch.float16, device="cuda")
    flat[1:] = src.flatten()
    for out_dtype in ("f16", "f32"):
        got = [api.zoom_density(s, f, 144 // f, out_dtype=out_dtype).cpu().numpy().tobytes()
               for s in (src, flat[1:].view(144, 144, 144))]
        assert got[0] == got[1]
