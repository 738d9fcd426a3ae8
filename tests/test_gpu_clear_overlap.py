"""The clear of a large map and the kernel that overlaps it: few records binned into a map of 64 MB
take less time than the clear of the map and the binning one after the other."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1703_09707_gb300 import mlens as M  # noqa: E402


def _us(call, n=20):
    """Device time of one call, from a captured run of n: the fastest of five replays."""
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(n):
                call()
        g.replay()
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(s)
            g.replay()
            e1.record(s)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1) * 1e3 / n)
    return best


@pytest.mark.parametrize("order", ["flat", "grid"])
@pytest.mark.parametrize("nr", [256, 512])
def test_few_records_into_a_large_map(order, nr):
    n = 4096
    src, rays = (-8.0, 8.0, -8.0, 8.0, n, n), (-8.0, 8.0, -8.0, 8.0, nr, nr)
    beta = 3.0 * torch.randn((nr * nr, 4), device="cuda", generator=torch.Generator(device="cuda").manual_seed(nr))
    beta[:, 2:] *= 1e-8
    counts = torch.empty(n * n, dtype=torch.int32, device="cuda")

    def run(k, flags=0):
        if order == "flat":
            M.mlens_bin(beta, k * nr, src, counts, flags=flags)
        else:
            M.mlens_bin_grid(beta, (*rays[:5], k), src, counts, flags=flags)

    whole, clear, add = _us(lambda: run(nr)), _us(lambda: run(1)), _us(lambda: run(nr, M.MLENS_ACCUMULATE))
    run(nr)
    px = ((beta[:, :2].double() + beta[:, 2:].double() + 8.0) * (n / 16.0)).floor().long()
    ok = ((px >= 0) & (px < n)).all(1)
    want = torch.bincount(px[ok, 1] * n + px[ok, 0], minlength=n * n)
    assert torch.equal(counts.long(), want)
    assert whole < clear + add, f"{whole:.1f} us against {clear:.1f} + {add:.1f}"
