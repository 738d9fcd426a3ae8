"""The convolution kernels where their tiles, row strides, widths and number ranges change:
the disk bit for bit against the oracle's exact sums, the Gaussian within the FP32 bound of its
two passes."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle import lightcurve as LC  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


def _conv(c, src, profile, size, scale):
    out = torch.empty(src.ny * src.nx, dtype=torch.float32, device="cuda")
    M.mlens_convolve(torch.from_numpy(np.ascontiguousarray(c).view(np.int32).reshape(-1)).cuda(), src, profile, size,
                     out, scale=scale)
    return out.cpu().numpy().reshape(src.ny, src.nx)


def _counts(rng, ny, nx, kind):
    c = rng.poisson(25.0, (ny, nx)).astype(np.uint32)
    if kind == "spikes":
        c[rng.random((ny, nx)) < 0.02] = 60000
    if kind == "large":  # beyond 32-bit sums in some tiles only
        c[: ny // 2, : nx // 2][rng.random((ny // 2, nx // 2)) < 0.3] = 4_294_967_295
    if kind == "empty":
        c[:, nx // 3:] = 0
    return c


@pytest.mark.parametrize("kind,scale", [("spikes", 1.7), ("large", 0.3), ("empty", -2.5e-3), ("spikes", 1e30), ("spikes", 0.0)])
@pytest.mark.parametrize("px", [0.3, 5.01, 6.0, 21.3, 22.1, 37.9, 38.1, 54.0, 85.6, 86.2])
def test_disk_at_stride_and_tile_edges(px, kind, scale):
    rng = np.random.default_rng(int(10 * px))
    nx, ny = 197, 75  # ragged in both axes, 64 x 32 tiles
    src = W.Grid(0.0, nx * 0.01, 0.0, ny * 0.01, nx, ny)
    c = _counts(rng, ny, nx, kind)
    got = _conv(c, src, M.MLENS_PROFILE_DISK, px * 0.01, scale)
    js, is_ = rng.integers(0, ny, 150), rng.integers(0, nx, 150)
    js[:4], is_[:4] = (0, 0, ny - 1, ny - 1), (0, nx - 1, 0, nx - 1)
    ref = LC.convolve_at(c, src, LC.DISK, px * 0.01, scale, js, is_).astype(np.float32)
    assert np.array_equal(got[js, is_].view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("px", [3.2, 20.5, 30.0])
@pytest.mark.parametrize("over", [0, 1])
def test_disk_wide_tiles_at_the_32_bit_limit(px, over):
    """A map of enough 128 x 64 tiles; counts of exactly the largest value whose |K|-fold
    still fits 32 bits, and one above it (the 64-bit sums), and flat areas on float ties."""
    rng = np.random.default_rng(int(px) + over)
    nx, ny = 2305, 1100
    src = W.Grid(0.0, nx * 0.01, 0.0, ny * 0.01, nx, ny)
    k = len(LC.disk_offsets(px * 0.01, *LC._pix(src)))
    c = rng.poisson(25.0, (ny, nx)).astype(np.uint32)
    c[200:700, 300:1500] = (2 ** 32 - 1) // k + over
    c[800:1000, 300:1500] = 2 ** 24 // k + 1
    got = _conv(c, src, M.MLENS_PROFILE_DISK, px * 0.01, 1.0)
    js, is_ = rng.integers(0, ny, 300), rng.integers(0, nx, 300)
    ref = LC.convolve_at(c, src, LC.DISK, px * 0.01, 1.0, js, is_).astype(np.float32)
    assert np.array_equal(got[js, is_].view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("nx", [1, 255, 256, 257, 512, 513, 1025])
@pytest.mark.parametrize("px", [0.4, 1.0, 10.24, 63.9])
def test_gaussian_at_width_and_tap_edges(nx, px):
    rng = np.random.default_rng(nx)
    ny = 131
    src = W.Grid(0.0, nx * 0.01, 0.0, ny * 0.02, nx, ny)  # taller pixels: fewer taps along y
    c = _counts(rng, ny, nx, "spikes")
    got = _conv(c, src, M.MLENS_PROFILE_GAUSSIAN, px * 0.01, 0.37)
    js, is_ = rng.integers(0, ny, 60), rng.integers(0, nx, 60)
    ref = LC.convolve_at(c, src, LC.GAUSSIAN, px * 0.01, 0.37, js, is_)
    kx, ky = math.ceil(4 * px), math.ceil(2 * px)
    # 2 Kx + 1 and 2 Ky + 1 products and sums of non-negative terms, weights and scale rounded
    bound = 2.0 * (2 * kx + 2 * ky + 8) * 2.0 ** -24 * np.abs(ref) + 1e-30
    assert np.all(np.abs(got[js, is_] - ref) <= bound)


@pytest.mark.parametrize("px", [3.2, 21.6, 37.4, 53.2, 80.0])
@pytest.mark.parametrize("mean", [6.0, 40.0, 60.0])
def test_disk_square_tiles_and_packed_sums(px, mean):
    """A map of enough 64 x 64 tiles but not enough 128 x 64 ones; mean counts whose row totals
    fit 16 bits with room for all rows of the support, with room for a few, and not at all."""
    rng = np.random.default_rng(int(px + mean))
    nx, ny = 1025, 701
    src = W.Grid(0.0, nx * 0.01, 0.0, ny * 0.01, nx, ny)
    c = rng.poisson(mean, (ny, nx)).astype(np.uint32)
    c[300:400, 100:900:7] = int(20 * mean)  # some tiles beyond, their neighbours within
    got = _conv(c, src, M.MLENS_PROFILE_DISK, px * 0.01, 0.7)
    js, is_ = rng.integers(0, ny, 120), rng.integers(0, nx, 120)
    js[:4], is_[:4] = (0, 0, ny - 1, ny - 1), (0, nx - 1, 0, nx - 1)
    ref = LC.convolve_at(c, src, LC.DISK, px * 0.01, 0.7, js, is_).astype(np.float32)
    assert np.array_equal(got[js, is_].view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("nx,ny", [(4, 1), (12, 33), (252, 17), (260, 16), (508, 7), (516, 9), (1028, 5), (2052, 3)])
@pytest.mark.parametrize("px", [1.0, 30.3])
def test_gaussian_rows_of_whole_vectors(nx, ny, px):
    """Widths of whole float4 whose last thread has one of its two; odd row counts; every row
    checked at both ends."""
    rng = np.random.default_rng(nx + ny)
    src = W.Grid(0.0, nx * 0.01, 0.0, ny * 0.01, nx, ny)
    c = _counts(rng, ny, nx, "spikes")
    got = _conv(c, src, M.MLENS_PROFILE_GAUSSIAN, px * 0.01, 0.37)
    edges = np.unique(np.r_[:min(nx, 9), max(nx - 9, 0):nx])
    js, is_ = (v.ravel() for v in np.meshgrid(np.arange(ny), edges, indexing="ij"))
    ref = LC.convolve_at(c, src, LC.GAUSSIAN, px * 0.01, 0.37, js, is_)
    k = math.ceil(4 * px)
    # 2 k + 1 products and sums of non-negative terms per pass, weights and scale rounded
    bound = 2.0 * (4 * k + 8) * 2.0 ** -24 * np.abs(ref) + 1e-30
    assert np.all(np.abs(got[js, is_] - ref) <= bound)
