"""The learned kernel's tiles from the fit's descriptors: cells with no, one and more than a
stage of near stars, grids that end inside a tile, row ranges, and a reload, each ray within
the fit's own validated error and the FP32 bound of the oracle."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from gpu_util import beta_pair_to_f64, make_ctx, oracle_reference, position_rounding  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


@pytest.mark.parametrize("near", [0, 1, 255, 256, 257, 600])
@pytest.mark.parametrize("ny,lo", [(128, 0), (101, 1)])
def test_near_star_counts_and_ragged_grids(near, ny, lo, tmp_path):
    rng = np.random.default_rng(near + ny)
    w = 0.5 * (1.0 + 0.03 * lo)  # a dyadic cell width, or one whose ray offsets need low parts
    rays = W.Grid(-2 * w, 2 * w, 0.0, w * ny / 64.0, 256, ny)  # four cells across, 64 rows per cell
    far = rng.uniform(3.0, 9.0, (300, 1)) * np.stack([np.cos(a := rng.uniform(0, 2 * np.pi, 300)), np.sin(a)], 1)
    xy = np.concatenate([far, rng.uniform([-2 * w, 0.0], [-w, 0.9 * w], (near, 2))])  # all in the first cell
    xy, m = W.to_f32_exact(xy), W.to_f32_exact(rng.uniform(0.01, 0.02, len(xy)))
    f = W.Field(xy=xy, m=m, kappa_c=0.1, gamma1=0.2, gamma2=0.05)
    src = W.Grid(-2.0, 2.0, -1.0, 3.0, 70, 60)
    ctx = make_ctx(f)
    rep = M.mlens_fit_far_field(ctx, rays, M.fit_params(cells_x=4, order=16, use_network=0, tolerance=1.0))
    assert rep["cells_fallback"] == 0
    counts = torch.empty(src.n, dtype=torch.int32, device="cuda")
    beta = torch.empty(rays.n * 4, dtype=torch.float32, device="cuda")
    st = M.mlens_shoot_learned(ctx, rays, src, counts, beta=beta, stats=True)
    whole, b4 = counts.cpu().numpy().copy(), beta.cpu().numpy().reshape(-1, 4)
    assert st["rays_total"] == rays.n
    ref = oracle_reference(f, rays, np.arange(rays.n, dtype=np.int64))
    err = np.linalg.norm(beta_pair_to_f64(b4) - ref["b64"], axis=1)
    jn = np.sqrt(ref["J"][:, 0] ** 2 + 2 * ref["J"][:, 1] ** 2 + ref["J"][:, 2] ** 2)
    allow = 2 * rep["val_max_err_series"] + 1e-5 * ref["scale"] + jn * math.sqrt(2.0) * position_rounding(rays)
    assert np.max(err / allow) <= 1.0
    # row ranges add up to the whole map, and a saved field shoots it again
    if ny % 32 == 0:
        for k, rows in enumerate(((0, 32), (32, ny))):
            M.mlens_shoot_learned(ctx, rays, src, counts, rows=rows, flags=M.MLENS_ACCUMULATE if k else 0)
        assert np.array_equal(counts.cpu().numpy(), whole)
    path = str(tmp_path / "ff.bin")
    M.mlens_save_far_field(ctx, path)
    M.mlens_load_far_field(ctx, path)
    M.mlens_shoot_learned(ctx, rays, src, counts)
    assert np.array_equal(counts.cpu().numpy(), whole)
    ctx.close()
