"""The direct sum by half tiles and the clears before it: ray grids around a half tile's width
and a tile's rows, star counts with every kind of short last chunk, maps that start off a
16-byte boundary and end between two, accumulation, and replays of a captured call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import workloads as W  # noqa: E402
from gpu_util import compare_to_oracle, make_ctx, shoot_gpu  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 32), (32, 33), (33, 16), (63, 1), (64, 64), (65, 31), (96, 17), (129, 65)])
@pytest.mark.parametrize("rpt", [8, 4])
def test_grids_around_a_half_tile(nx, ny, rpt):
    f = W.random_field(W.SEED_BASE + 500 + nx, 200 + nx, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.07)
    rays, src = W.Grid(-3.0, 3.0, -2.0, 2.0, nx, ny), W.Grid(-2.0, 2.0, -2.0, 2.0, 90, 40)
    for split in (1, 3, 9):
        ctx = make_ctx(f)
        M.mlens_set_tuning(ctx, rpt)
        M.mlens_set_star_split(ctx, split)
        c, st, b4 = shoot_gpu(f, rays, src, ctx=ctx)
        ctx.close()
        c_re, st_re = oracle.rebin_pair(b4, src)
        assert np.array_equal(c, c_re) and st == st_re, split
        assert compare_to_oracle(f, rays, src, b4, rays_per_thread=rpt)["bound_ratio"] <= 1.0, split


@pytest.mark.parametrize("n", list(range(1, 8)) + [30, 34, 35, 36, 62, 125, 131, 159])
def test_short_last_chunks_equal_padded_ones(n):
    """Massless stars add exactly zero: a field filled up with them to whole chunks gives
    the same positions bit for bit as one whose last chunk is short."""
    f = W.random_field(W.SEED_BASE + 600 + n, n, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.07)
    k = -n % 32
    g = W.Field(xy=np.concatenate([f.xy, np.full((k, 2), 3e5)]), m=np.concatenate([f.m, np.zeros(k)]),
                kappa_c=f.kappa_c, gamma1=f.gamma1, gamma2=f.gamma2)
    src = W.Grid(-2.0, 2.0, -2.0, 2.0, 64, 64)
    for rays in (W.Grid(-3.1, 2.9, -1.7, 2.2, 70, 40), W.Grid(-8.0, 8.0, -8.0, 8.0, 64, 64)):
        for split in (1, 2, 20):
            (c0, s0, b0), (c1, s1, b1) = (shoot_gpu(h, rays, src, split=split) for h in (f, g))
            assert np.array_equal(b0.view(np.uint32), b1.view(np.uint32)), split
            assert np.array_equal(c0, c1) and s0 == s1


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 1), (7, 1), (5, 5), (64, 33)])
def test_clears_touch_the_map_alone(off, nx, ny):
    f = W.random_field(W.SEED_BASE + 700, 50, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.0)
    rays, src = W.Grid(-3.0, 3.0, -2.0, 2.0, 100, 60), W.Grid(-2.0, 2.0, -2.0, 2.0, nx, ny)
    want, st, _ = shoot_gpu(f, rays, src)
    buf = torch.full((off + src.n + 9,), 77, dtype=torch.int32, device="cuda")
    counts = buf[off:off + src.n]
    ctx = make_ctx(f)
    assert M.mlens_shoot(ctx, rays, src, counts, stats=True) == st
    assert np.array_equal(counts.cpu().numpy().view(np.uint32).reshape(ny, nx), want)
    assert (buf[:off] == 77).all() and (buf[off + src.n:] == 77).all()
    M.mlens_shoot(ctx, rays, src, counts, flags=M.MLENS_ACCUMULATE)
    assert np.array_equal(counts.cpu().numpy().view(np.uint32).reshape(ny, nx), 2 * want)
    ctx.close()


def test_captured_calls_replay():
    f = W.random_field(W.SEED_BASE + 701, 300, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.0)
    rays, src = W.Grid(-3.0, 3.0, -2.0, 2.0, 200, 160), W.Grid(-2.0, 2.0, -2.0, 2.0, 120, 90)
    want, _, b4 = shoot_gpu(f, rays, src)
    ctx = make_ctx(f)
    counts = torch.empty(src.n, dtype=torch.int32, device="cuda")
    binned = torch.empty(src.n, dtype=torch.int32, device="cuda")
    beta = torch.empty(rays.n * 4, dtype=torch.float32, device="cuda")
    M.mlens_bin_grid(beta.zero_(), rays, src, binned)  # the library's scratch exists before the capture
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        M.mlens_shoot_beta(ctx, rays, src, counts, beta)
        M.mlens_bin_grid(beta, rays, src, binned)
    for _ in range(3):
        counts.fill_(5)
        binned.fill_(6)
        beta.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for c in (counts, binned):
            assert np.array_equal(c.cpu().numpy().view(np.uint32).reshape(src.ny, src.nx), want)
        assert np.array_equal(beta.cpu().numpy().view(np.uint32), b4.reshape(-1).view(np.uint32))
    ctx.close()


@pytest.mark.parametrize("blocks", [1, 4, 5, 8, 9, 12, 13])
@pytest.mark.parametrize("rpt,precision", [(8, "fp32"), (4, "fp32"), (8, "fp32_naive")])
def test_grids_of_few_ctas_equal_their_bands(blocks, rpt, precision):
    """38 half tiles per 32 rows: up to one, two, three or more CTAs on each of 152 SMs, and
    every band of 32 rows, launched with at most one per SM, gives the same positions and map."""
    f = W.random_field(W.SEED_BASE + 700, 300, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.07)
    ny = 32 * blocks - (5 if blocks > 1 else 0)
    rays, src = W.Grid(-3.0, 3.0, -2.0, 2.0, 1200, ny), W.Grid(-2.0, 2.0, -2.0, 2.0, 90, 40)
    ctx = M.mlens_create(f.xy, f.m, f.kappa_c, f.gamma1, f.gamma2, precision)
    M.mlens_set_tuning(ctx, rpt)
    M.mlens_set_star_split(ctx, 1)
    whole, bands = (torch.zeros((40, 90), dtype=torch.int32, device="cuda") for _ in range(2))
    b0, b1 = (torch.zeros((ny, 1200, 4), dtype=torch.float32, device="cuda") for _ in range(2))
    M.mlens_shoot_beta(ctx, rays, src, whole, b0)
    for r in range(0, ny, 32):
        M.mlens_shoot_rows(ctx, rays, (r, min(r + 32, ny)), src, bands, beta=b1, flags=M.MLENS_ACCUMULATE)
    ctx.close()
    assert whole.any() and torch.equal(whole, bands)
    assert torch.equal(b0.view(torch.int32), b1.view(torch.int32))
