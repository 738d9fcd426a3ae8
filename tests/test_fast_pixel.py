"""The fast pixel rule of the binning kernels (mlens_dev.cuh, fast_pixel).

On the CPU the rule is evaluated in IEEE float32 (numpy; the FMAs correctly rounded through
round-to-odd float64) on records on, next to and across pixel edges, in and far outside
maps of many shapes: wherever it decides, its pixel equals the oracle's exact float-pair
rule, non-finite components and large low parts are never decided, and almost every ordinary
record is.  On the GPU the binning kernels' maps and counters equal the oracle's at the edges of
blocks and of the window, for maps smaller than the window, and where the rule never decides."""
import numpy as np
import pytest

import oracle
import workloads as W

f32, f64 = np.float32, np.float64
MAGIC = f32(12582912.0)


def constants(x0, x1, n):
    """The per-axis constants as the library's host code makes them."""
    s = n / (x1 - x0)
    x0h, sh = f32(x0), f32(s)
    cd = -(x0 - float(x0h)) * s - 0.5
    t = 0.5 - 2.0 ** -24 * 1.001 * (3.0 * n + 4.0 * abs(cd) + 8.0)
    bm = 0.25 / abs(float(sh))
    thr = f32(t) if float(f32(t)) <= t else np.nextafter(f32(t), f32(-np.inf))
    bl = f32(bm) if float(f32(bm)) <= bm else np.nextafter(f32(bm), f32(0))
    if not t > 0 or n > 1 << 20 or not abs(x0 * s) <= 2.0 ** 21:
        thr = f32(-1)
    return -x0h, sh, f32(cd), thr, bl


def fma32(a, b, c):
    p, c = a.astype(f64) * b.astype(f64), c.astype(f64)  # the product is exact
    s = p + c
    bb = s - p
    e = (p - (s - bb)) + (c - bb)
    odd = (s.view(np.int64) & 1) == 1
    toward = np.where((e > 0) == (s > 0), 1, -1)
    fix = np.isfinite(s) & (e != 0) & ~odd
    return np.where(fix, (s.view(np.int64) + toward).view(f64), s).astype(f32)


def fast_axis(bh, bl, x0, x1, n, norm=False):
    nx0, sh, c, thr, blmax = constants(x0, x1, n)
    full = lambda v: np.full_like(bh, v)  # noqa: E731
    with np.errstate(all="ignore"):
        d = (bh + nx0).astype(f32)
        u = fma32(d, full(sh), fma32(bl, full(sh), full(c)))
        t = (u + MAGIC).astype(f32)
        k = (t - MAGIC).astype(f32)
        px = t.view(np.int32).astype(np.int64) - int(MAGIC.view(np.int32))
        px = ((px + 2 ** 31) % 2 ** 32 - 2 ** 31)
        ok = np.abs((u - k).astype(f32)) <= thr
        if not norm:
            ok &= np.abs(bl) <= blmax
    return ok, np.where((px >= 0) & (px < n), px, -1)


def exact_axis(bh, bl, x0, x1, n):
    b4 = np.stack([bh, np.full_like(bh, 0.5), bl, np.zeros_like(bh)], 1)
    pix = oracle.pair_pixels(b4, W.Grid(x0, x1, 0.0, 1.0, n, 1))
    return np.where(pix >= 0, pix % n, -1)


MAPS = [(-10.0, 20.0, 1024), (3.25 + 1e-9, 0.1, 4096), (-120.5, 300.0, 37), (-4.0, 8.0, 32768), (-2.0 / 3.0, 4.0 / 3.0, 999),
        (1e3 + 0.3, 1e-3, 64), (-75.0, 150.0, 1 << 20), (0.0, 1e-30, 5), (-1e9, 2e9, 300), (17.0, 1.0, 1)]


@pytest.mark.parametrize("x0,w,n", MAPS)
@pytest.mark.parametrize("norm", [False, True])
def test_decided_pixels_equal_the_exact_rule(x0, w, n, norm):
    rng = np.random.default_rng(n)
    k = 300_000
    edge = x0 + rng.integers(-2, n + 3, k) * (w / n)
    bh = edge.astype(f32)
    mode = rng.integers(0, 5, k)
    ulp = np.spacing(np.abs(bh)).astype(f32)
    bh = np.where(mode == 1, bh + rng.integers(-3, 4, k).astype(f32) * ulp, bh).astype(f32)
    bh = np.where(mode == 3, rng.uniform(x0 - 0.5 * w, x0 + 1.5 * w, k), bh).astype(f32)
    far = rng.choice([-1.0, 1.0], k) * 10.0 ** rng.uniform(-3, 38.4, k)
    bh = np.where(mode == 4, far, bh).astype(f32)
    bl = np.where(mode == 0, edge - bh.astype(f64), rng.uniform(-0.5, 0.5, k) * np.spacing(np.abs(bh))).astype(f32)
    if not norm:  # records need not be normalised pairs
        big = rng.random(k) < 0.1
        bl = np.where(big, rng.choice([-1.0, 1.0], k) * 10.0 ** rng.uniform(-30, 30, k), bl).astype(f32)
    ok, px = fast_axis(bh, bl, x0, x0 + w, n, norm)
    want = exact_axis(bh, bl, x0, x0 + w, n)
    bad = ok & (px != want)
    assert not bad.any(), (int(bad.sum()), bh[bad][:3], bl[bad][:3], px[bad][:3], want[bad][:3])


@pytest.mark.parametrize("x0,w,n", [(-10.0, 20.0, 1024), (-75.0, 150.0, 8192), (3.25 + 1e-9, 0.1, 4096)])
def test_almost_every_ordinary_record_is_decided(x0, w, n):
    rng = np.random.default_rng(n)
    b = rng.uniform(x0 - 0.5 * w, x0 + 1.5 * w, 300_000)
    bh = b.astype(f32)
    ok, _ = fast_axis(bh, (b - bh.astype(f64)).astype(f32), x0, x0 + w, n)
    assert ok.mean() > 1.0 - 4.0 * 2.0 ** -24 * (3 * n + 12) - 1e-3


def test_non_finite_components_are_never_decided():
    bad = np.array([np.nan, np.inf, -np.inf], f32)
    for bh, bl in ((bad, np.zeros(3, f32)), (np.ones(3, f32), bad), (bad, bad)):
        for norm in (False, True):
            assert not fast_axis(bh, bl, -10.0, 10.0, 1024, norm)[0].any()


GPU_MAPS = [W.Grid(-10.0, 10.0, -10.0, 10.0, 1024, 1024), W.Grid(-1.0, 1.0, -2.0, 2.0, 63, 65),
            W.Grid(3.25 + 1e-9, 3.35, 0.0, 1.0, 200, 7), W.Grid(1e3 + 0.3, 1e3 + 0.301, -1.0, 1.0, 64, 64),
            W.Grid(-1.0, 1.0, -1.0, 1.0, 1 << 22, 3), W.Grid(0.0, 1.0, 0.0, 1.0, 1, 1)]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(1, 1), (64, 64), (65, 63), (63, 129), (4097, 1), (700, 301)])
@pytest.mark.parametrize("m", range(len(GPU_MAPS)))
def test_kernels_equal_the_oracle(nx, ny, m):
    torch = pytest.importorskip("torch")
    from paper_1703_09707_gb300 import mlens as M
    src, n = GPU_MAPS[m], nx * ny
    rng = np.random.default_rng(nx * 7 + ny + m)
    b = np.zeros((n, 4), f32)
    for a, (lo, hi, k) in enumerate(((src.x0, src.x1, src.nx), (src.y0, src.y1, src.ny))):
        v = rng.uniform(lo - 0.2 * (hi - lo), hi + 0.2 * (hi - lo), n)
        v = np.where(rng.random(n) < 0.3, lo + rng.integers(0, k + 1, n) * ((hi - lo) / k), v)
        b[:, a] = v
        b[:, a + 2] = v - b[:, a].astype(f64)
    for v in (np.nan, np.inf, -np.inf, 3e38, -1e20):
        q = rng.random(n) < 0.003
        b[q, rng.integers(0, 4, int(q.sum()))] = v
    want, st = oracle.rebin_pair(b, src)
    bd = torch.from_numpy(b).cuda()
    counts = torch.empty(src.n, dtype=torch.int32, device="cuda")
    for call in (lambda: M.mlens_bin(bd, n, src, counts, stats=True),
                 lambda: M.mlens_bin_grid(bd, W.Grid(0.0, 1.0, 0.0, 1.0, nx, ny), src, counts, stats=True)):
        assert call() == st
        assert np.array_equal(counts.cpu().numpy().view(np.uint32).reshape(src.ny, src.nx), want)
