"""The star stages of the direct sum (y offsets formed once per tile row and star, held
in shared memory) at the edges of their stages, chunks and tiles: every stage size gives
the same beta bit for bit, each within the FP32 error bound of the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from gpu_util import compare_to_oracle, make_ctx, shoot_gpu  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 513])
@pytest.mark.parametrize("rpt", [8, 4])
def test_stage_sizes_agree_at_stage_and_chunk_edges(n, rpt):
    f = W.random_field(W.SEED_BASE + 300 + n, n, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.07)
    src = W.Grid(-2.0, 2.0, -2.0, 2.0, 64, 64)
    # a non-dyadic grid (offsets with low parts) of whole tiles and a ray more, and a dyadic one short of a tile
    for rays in (W.Grid(-3.1, 2.9, -1.7, 2.2, 65, 33), W.Grid(-8.0, 8.0, -8.0, 8.0, 64, 31)):
        ref = None
        for stage in (128, 256, 512):
            ctx = make_ctx(f)
            M.mlens_set_tuning(ctx, rpt, stage)
            c, st, b4 = shoot_gpu(f, rays, src, ctx=ctx)
            ctx.close()
            if ref is None:
                ref = (c, st, b4)
                assert compare_to_oracle(f, rays, src, b4, rays_per_thread=rpt)["bound_ratio"] <= 1.0
            assert np.array_equal(b4.view(np.uint32), ref[2].view(np.uint32)), (stage, rays)
            assert np.array_equal(c, ref[0]) and st == ref[1]


@pytest.mark.parametrize("n", [40, 4095, 4096])
def test_fallback_tiles_equal_the_plain_map_below_and_at_the_first_split(n):
    """Flagged cells run as listed tiles, unsplit below 4096 stars (as padded to chunks of
    32): the plain map bit for bit."""
    f = W.random_field(W.SEED_BASE + 340 + n, n, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.0)
    rays = W.Grid(-2.0, 2.0, -1.0, 1.0, 512, 256)
    src = W.Grid(-1.0, 1.0, -1.0, 1.0, 96, 80)
    ctx = make_ctx(f)
    rep = M.mlens_fit_far_field(ctx, rays, M.fit_params(cells_x=8, order=2, use_network=0, tolerance=0.0))
    assert rep["cells_fallback"] == rep["cells"]
    counts = torch.empty(src.n, dtype=torch.int32, device="cuda")
    beta = torch.empty(rays.n * 4, dtype=torch.float32, device="cuda")
    st = M.mlens_shoot_learned(ctx, rays, src, counts, beta=beta, stats=True)
    ctx.close()
    c, st1, b4 = shoot_gpu(f, rays, src, split=2 if (n + 31) // 32 * 32 >= 4096 else 1)
    assert st == st1
    assert np.array_equal(beta.cpu().numpy().view(np.uint32), b4.reshape(-1).view(np.uint32))
    assert np.array_equal(counts.cpu().numpy().view(np.uint32).reshape(src.ny, src.nx), c)
