"""Disks wider than the map: bit for bit against the oracle's exact sums, counts to the edge of 32 bits
included, and no slower than a narrower disk that covers the same columns."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle import lightcurve as LC  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


def _grid(nx, ny, half_width, half_rows):
    """A map of pixels so flat or tall that a disk of half_width + 1/2 columns has half_rows rows on each side."""
    return W.Grid(0.0, float(nx), 0.0, ny * (half_width + 0.5) / (half_rows + 0.5), nx, ny)


@pytest.mark.parametrize("nx", [1, 8, 63, 64, 130])
@pytest.mark.parametrize("hw,hr", [(200, 3), (3000, 20), (800, 60)])
@pytest.mark.parametrize("top", [50, 2 ** 32 - 1, 0])
def test_disks_wider_than_the_map(nx, hw, hr, top):
    ny, rng = 150, np.random.default_rng(nx + hw)
    src = _grid(nx, ny, hw, hr)
    if top == 0:  # the largest count whose sums still fit 32 bits, and one more
        top = (2 ** 32 - 1) // ((2 * hr + 1) * nx)
        c = np.full((ny, nx), top, np.uint32)
        c[ny // 2:] += 1
    else:
        c = rng.integers(0, top, (ny, nx), dtype=np.uint32, endpoint=True)
    out = torch.empty(src.n, dtype=torch.float32, device="cuda")
    M.mlens_convolve(torch.from_numpy(c.view(np.int32).reshape(-1)).cuda(), src, M.MLENS_PROFILE_DISK, hw + 0.5, out, scale=3.0)
    got = out.cpu().numpy().reshape(ny, nx)
    js, is_ = rng.integers(0, ny, 40), rng.integers(0, nx, 40)
    ref = LC.convolve_at(c, src, LC.DISK, hw + 0.5, 3.0, js, is_).astype(np.float32)
    assert np.array_equal(got[js, is_].view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("nx", [8, 20])
def test_a_wide_disk_costs_what_the_map_s_columns_do(nx):
    ny, times = 20000, []
    counts = torch.randint(0, 30, (nx * ny,), device="cuda").to(torch.int32)
    for hw in (300, 3000):
        src = _grid(nx, ny, hw, 20)
        out = torch.empty(src.n, dtype=torch.float32, device="cuda")
        work = torch.empty(M.mlens_convolve_workspace(src, M.MLENS_PROFILE_DISK, hw + 0.5), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(20):
                M.mlens_convolve(counts, src, M.MLENS_PROFILE_DISK, hw + 0.5, out, work=work)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[1] < 1.3 * times[0], f"{50 * times[1]:.1f} us against {50 * times[0]:.1f}"
