"""GPU: kernels over stored grids at the edges of their fast paths: density groups of eight voxels,
exact FP16 block sums, and Q binning of a stored intensity."""
import numpy as np
import pytest
import torch

from oracle import density, scatter
from paper_2303_13435_gb300 import api, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.lib()
    torch.cuda.init()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("kind", [inputs.SHAPE_SPHERE, inputs.SHAPE_CUBE, inputs.SHAPE_OCTAHEDRON])
@pytest.mark.parametrize("n,ucell,origin,rot", [(64, 37, (36, 1, 20), 0), (72, 48, (4, 3, 47), 5), (24, 8, (0, 0, 0), 0),
                                                (58, 16, (5, 0, 2), 9)])
def test_density_groups_are_bit_exact(kind, n, ucell, origin, rot):
    """Off-centre particles whose surface crosses groups of eight everywhere, cells of both signs."""
    rng = np.random.default_rng(n + kind)
    cell = rng.standard_normal((ucell, ucell, ucell)).astype(np.float32)
    r = inputs.random_rotation(inputs.SplitMix64(rot)) if rot else np.eye(3, dtype=np.float32)
    for size in (0.47 * n, 3.0, 0.2):
        sh = inputs.Shape(kind, (n / 2 + 0.3, n / 2 - 2.0, n / 2 + 1.75), float(np.float32(size)), r)
        for dtype in ("f32", "f16"):
            want = density.tile_mask_density(n, cell, kind, sh.center, sh.size, sh.rot, origin=origin, out_dtype=dtype)
            got = api.build_density(n, dev(cell), sh, origin=origin, out_dtype=dtype)
            assert got.cpu().numpy().tobytes() == want.tobytes(), (size, dtype)


@pytest.mark.parametrize("f", [1, 2, 3, 4, 8, 16])
@pytest.mark.parametrize("blocks,n_out", [(1, 3), (3, 16), (5, 21)])
def test_zoom_of_every_half_is_exact(f, blocks, n_out):
    """Block sums of halves of every exponent, subnormals to the largest, both signs."""
    n = f * blocks
    if n % 2:
        n_src, n_out = 2 * n, max(n_out, 2 * blocks)
    else:
        n_src = n
    rng = np.random.default_rng(f * 100 + blocks)
    bits = rng.integers(0, 0x7C00, (n_src, n_src, n_src), dtype=np.uint16)  # every finite magnitude
    ed = (bits | (rng.integers(0, 2, bits.shape, dtype=np.uint16) << 15)).view(np.float16)
    ed[0, 0, 0] = np.float16(65504)
    s = density.block_sums(ed, f)
    small = np.abs(s).max() < 65504
    for out_dtype in (["f16", "f32"] if small or f <= 2 else ["f32"]):
        with np.errstate(over="ignore"):
            want = density.zoom_out(ed, f, n_out, out_dtype=out_dtype)
        got = api.zoom_density(dev(ed), f, n_out, out_dtype=out_dtype).cpu().numpy()
        # a zero sum has no sign bit on the GPU (integer sum)
        assert (got + np.array(0, got.dtype)).tobytes() == (want + np.array(0, want.dtype)).tobytes()


def full_grid(half):
    n = half.shape[0]
    full = np.empty((n, n, n), dtype=np.float64)
    full[:, :, : n // 2 + 1] = half
    i = (-np.arange(n)) % n
    for kx in range(n // 2 + 1, n):
        full[:, :, kx] = half[i][:, i][:, :, n - kx]
    return full


@pytest.mark.parametrize("n,nbins,log", [(8, 3, False), (30, 200, True), (64, 40, True), (100, 64, False), (128, 700, True)])
@pytest.mark.parametrize("wide", [False, True])
def test_bin_q_sums(n, nbins, log, wide):
    """Sums to float64 rounding: each run is a sum of at most 128 values held to 48 bits, each
    flush one float64 addition; 1e-12 covers both for positive values."""
    dx = 0.05
    top = inputs.nyquist_q(dx) * 1.2
    edges = inputs.log_edges(2 * np.pi / (n * dx), top, nbins) if log else inputs.linear_edges(top, nbins)
    rng = np.random.default_rng(n)
    half = rng.random((n, n, n // 2 + 1))
    if wide:  # magnitudes whose squares leave the float32 range on both sides, and exact zeros
        half = 10.0 ** rng.uniform(-30, 30, half.shape) * (rng.random(half.shape) < 0.9)
    half = half.astype(np.float32)
    plan = api.Plan(n, dx, edges)
    got = api.bin_q(plan, dev(half)).cpu().numpy()
    full = full_grid(half.astype(np.float64))
    ob = scatter.bin_intensity(full, n, dx, edges)
    sq = scatter.bin_intensity(full * full, n, dx, edges)
    nz = ob["count"] > 0
    assert np.array_equal(got[0].astype(np.int64), ob["count"])
    assert np.allclose(got[1][nz], ob["sum_i"][nz], rtol=1e-12, atol=0)
    assert np.allclose(got[2][nz], sq["sum_i"][nz], rtol=1e-12, atol=0)
    assert np.all(np.isnan(got[4][~nz]))
