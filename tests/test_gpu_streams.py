"""Small maps on several streams share the SMs: four streams' maps overlap, and are the maps of the
calls made one after another."""
import time

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from gpu_util import make_ctx  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402

SRC = W.Grid(-10.0, 10.0, -10.0, 10.0, 128, 128)


@pytest.mark.parametrize("prec", [M.MLENS_PREC_FP32, M.MLENS_PREC_FP32_NAIVE])
def test_small_maps_on_four_streams_overlap(prec):
    rays = W.Grid(-5.0, 5.0, -5.0, 5.0, 512, 256)  # half tiles for most SMs, one each
    f = W.random_field(11, 3000, 0.4, 0.1, 0.2, 0.0)
    ctxs = [make_ctx(f, prec, split=1) for _ in range(4)]
    maps = [torch.empty(SRC.n, dtype=torch.int32, device="cuda") for _ in ctxs]
    streams = [torch.cuda.Stream() for _ in ctxs]

    def per_map(n, k=40):
        best = float("inf")
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(k):
                for c, m, s in zip(ctxs[:n], maps, streams):
                    M.mlens_shoot(c, rays, SRC, m, stream=s)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / (k * n))
        return best

    one = per_map(1)
    want = maps[0].clone()
    four = per_map(4)
    assert all(torch.equal(m, want) for m in maps)
    assert four < 0.74 * one, f"{1e6 * four:.1f} us a map on four streams, {1e6 * one:.1f} on one"
    for c in ctxs:
        c.close()
