"""Timed cases of the library's work: the calls a user of the binding makes, at the sizes
of the repository's workloads (100 to 1e7 stars, maps of 256^2 to 4096^2 pixels) and
around them.

Every case is a dict of plain values; `kind` names the entry point:

  shoot    mlens_shoot / mlens_shoot_beta (`beta`) of one star field
  batch    mlens_batch_run over independent fields of uneven star counts
  learned  mlens_shoot_learned on a fitted far field
  fit      mlens_fit_far_field and the export of what it fitted
  bin      mlens_bin / mlens_bin_grid on recorded source positions
  convolve mlens_convolve with a caller workspace
  curve    mlens_light_curve

Units: angles in Einstein radii of a 1 M_sun lens, masses in M_sun.  A field of N stars
of mean mass <m> and surface density kappa_* fills a disk of radius sqrt(N <m> / kappa_*).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1703_09707_gb300 import mlens as M

# dN/dm ~ m^-2.35 on [0.1, 1]
_SLOPE, _MLO, _MHI = 2.35, 0.1, 1.0


def listed():
    return [
        # The smallest whole map: 100 unit masses, 1000^2 rays (0.02 spacing, not a dyadic
        # grid; neither axis a multiple of the ray tile), a 256^2 map.  One map takes tens
        # of microseconds: launches, clears and the tile's set-up count.
        dict(name="shoot_100_stars", kind="shoot", stars=100, unit_masses=True, kappa_star=0.45, kappa_c=0.0,
             gamma=0.0, src_half=4.0, ray_hx=10.0, ray_hy=10.0, rays_x=1000, rays_y=1000, map_x=256, map_y=256,
             precision="fp32", beta=False),
        # The headline map: 1e4 stars, 8192^2 rays, 1024^2 pixels.
        dict(name="shoot_1e4_stars", kind="shoot", stars=10_000, unit_masses=False, kappa_star=0.3, kappa_c=0.2,
             gamma=0.3, src_half=10.0, ray_hx=75.0, ray_hy=18.75, rays_x=8192, rays_y=8192, map_x=1024, map_y=1024,
             precision="fp32", beta=False),
        # Very many stars for few rays: the star sum of one ray tile shared by many CTAs.
        dict(name="shoot_1e7_stars", kind="shoot", stars=10_000_000, unit_masses=False, kappa_star=0.45, kappa_c=0.05,
             gamma=0.25, src_half=2.0, ray_hx=12.0, ray_hy=4.0, rays_x=256, rays_y=256, map_x=256, map_y=256,
             precision="fp32", beta=False),
        # The verification path: FP64 source positions of an odd ray grid, and their map.
        dict(name="shoot_fp64", kind="shoot", stars=5000, unit_masses=False, kappa_star=0.3, kappa_c=0.2,
             gamma=0.3, src_half=8.0, ray_hx=60.0, ray_hy=15.0, rays_x=509, rays_y=387, map_x=200, map_y=200,
             precision="fp64", beta=True),
        # A parameter-grid study: 256 independent fields, star counts log-uniform in
        # [1e2, 1e4], 2048^2 rays and a 512^2 map each, in one launch.
        dict(name="batch_256_fields", kind="batch", fields=256, stars_lo=100, stars_hi=10_000, rays=2048, map=512),
        # The far field of 1e6 stars learned, one whole 32768^2-ray map of it.
        dict(name="learned_1e6_stars", kind="learned", stars=1_000_000, cells=256, tiles=2, order=10, network=True,
             samples=1 << 24, epochs=48, map=4096),
        # The exact series alone (no network) on a smaller field and grid.
        dict(name="series_2e5_stars", kind="learned", stars=200_000, cells=128, tiles=2, order=16, network=False,
             samples=1, epochs=1, map=2048),
        # Fitting a far field: cells, coefficients, network training, validation.
        dict(name="fit_2e5_stars", kind="fit", stars=200_000, cells=128, tiles=2, order=10, network=True,
             samples=1 << 22, epochs=24),
        # Binning recorded source positions (8192^2 records in ray order) into a map.
        dict(name="bin_8192sq_records", kind="bin", rays_x=8192, rays_y=8192, map=1024, grid_order=True),
        # A map convolved with a Gaussian source of sigma = 10 pixels.
        dict(name="gaussian_4096sq", kind="convolve", profile="gaussian", map_x=4096, map_y=4096, size_px=10.24),
        # The same map seen by a uniform disk of radius 20 pixels.
        dict(name="disk_4096sq", kind="convolve", profile="disk", map_x=4096, map_y=4096, size_px=20.48),
        # A light curve of 4096 points: the smallest call of the library.
        dict(name="curve_4096_points", kind="curve", map=1024, points=4096),
    ]


def draw(rng):
    """One more case of the listed ranges (odd sizes among them), no dearer than the largest listed one."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["shoot", "shoot", "many", "fp64", "batch", "learned", "fit", "bin", "convolve", "convolve",
                       "curve"])
    kappa_star, kappa_c, gamma = rng.uniform(0.2, 0.45), rng.uniform(0.0, 0.2), rng.uniform(0.0, 0.25)
    if kind == "shoot":
        stars, rays_x, rays_y = log_int(100, 1e5), log_int(200, 8192), log_int(200, 8192)
        while stars * rays_x * rays_y > 6e11:
            rays_y //= 2
        half = _inner_half(stars, kappa_star, kappa_c, gamma, 0.5)
        hx, hy = _lens_box(kappa_star + kappa_c, gamma, half)
        return dict(kind="shoot", stars=stars, unit_masses=rng.random() < 0.2, kappa_star=kappa_star,
                    kappa_c=kappa_c, gamma=gamma, src_half=half, ray_hx=hx, ray_hy=hy, rays_x=rays_x, rays_y=rays_y,
                    map_x=log_int(100, 2048), map_y=log_int(100, 2048), precision="fp32",
                    beta=rng.random() < 0.3 and stars * rays_x * rays_y < 2e9)
    if kind == "many":
        rays_x, rays_y = log_int(100, 512), log_int(100, 512)
        stars = min(log_int(5e5, 1e7), int(6e11 / (rays_x * rays_y)))
        hx, hy = _lens_box(kappa_star + kappa_c, gamma, 2.0)
        return dict(kind="shoot", stars=stars, unit_masses=False, kappa_star=kappa_star, kappa_c=kappa_c, gamma=gamma,
                    src_half=2.0, ray_hx=hx, ray_hy=hy, rays_x=rays_x, rays_y=rays_y, map_x=256, map_y=256,
                    precision="fp32", beta=False)
    if kind == "fp64":
        stars, rays_x, rays_y = log_int(100, 5000), log_int(60, 500), log_int(60, 400)
        half = _inner_half(stars, kappa_star, kappa_c, gamma, 0.5)
        hx, hy = _lens_box(kappa_star + kappa_c, gamma, half)
        return dict(kind="shoot", stars=stars, unit_masses=False, kappa_star=kappa_star, kappa_c=kappa_c, gamma=gamma,
                    src_half=half, ray_hx=hx, ray_hy=hy, rays_x=rays_x, rays_y=rays_y, map_x=log_int(50, 300),
                    map_y=log_int(50, 300), precision="fp64", beta=True)
    if kind == "batch":
        return dict(kind="batch", fields=log_int(4, 200), stars_lo=100, stars_hi=log_int(1000, 10_000),
                    rays=log_int(300, 2048), map=log_int(100, 512))
    if kind == "learned":
        cells, tiles = rng.choice([48, 64, 96, 128]), rng.choice([1, 2])
        net = rng.random() < 0.5
        return dict(kind="learned", stars=log_int(30_000, 300_000), cells=cells, tiles=tiles,
                    order=10 if net else 16, network=net, samples=1 << 22, epochs=24, map=log_int(500, 2048))
    if kind == "fit":
        return dict(kind="fit", stars=log_int(20_000, 200_000), cells=rng.choice([48, 64, 96, 128]),
                    tiles=rng.choice([1, 2]), order=rng.choice([8, 10, 12, 16]), network=rng.random() < 0.6,
                    samples=log_int(1 << 18, 1 << 22), epochs=rng.randrange(4, 24))
    if kind == "bin":
        return dict(kind="bin", rays_x=log_int(300, 8192), rays_y=log_int(300, 8192), map=log_int(128, 2048),
                    grid_order=rng.random() < 0.5)
    if kind == "convolve":
        disk = rng.random() < 0.5
        return dict(kind="convolve", profile="disk" if disk else "gaussian", map_x=log_int(200, 4096),
                    map_y=log_int(200, 4096), size_px=math.exp(rng.uniform(0.0, math.log(80.0 if disk else 30.0))))
    return dict(kind="curve", map=log_int(128, 4096), points=log_int(16, 100_000))


# ---------------------------------------------------------------- star fields
def _mean_mass():
    a, b = 2.0 - _SLOPE, 1.0 - _SLOPE
    return ((_MHI ** a - _MLO ** a) / a) / ((_MHI ** b - _MLO ** b) / b)


def _radius(stars, kappa_star, unit_masses=False):
    return math.sqrt(stars * (1.0 if unit_masses else _mean_mass()) / kappa_star)


def _lens_box(kappa, gamma, src_half):
    """Half sizes of the ray box: the source box, half as large again, mapped back through the macro model."""
    return tuple(math.ceil(64.0 * 1.5 * src_half / abs(1.0 - kappa + s * gamma)) / 64.0 for s in (-1.0, 1.0))


def _inner_half(stars, kappa_star, kappa_c, gamma, share):
    """Half the source box whose ray box stays within `share` of the star disk's radius."""
    half = share * _radius(stars, kappa_star) * abs(1.0 - kappa_star - kappa_c - gamma) / 1.5
    return max(1.0 / 64.0, math.floor(64.0 * half) / 64.0)


def _stars(seed, stars, kappa_star, unit_masses=False):
    """Positions uniform in the field's disk and masses, drawn on the GPU, rounded to float32: host FP64 arrays."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((3, stars), generator=g, device="cuda", dtype=torch.float64)
    r, phi = _radius(stars, kappa_star, unit_masses) * u[0].sqrt(), 2.0 * math.pi * u[1]
    e = 1.0 - _SLOPE
    m = torch.ones_like(u[2]) if unit_masses else (_MLO ** e + u[2] * (_MHI ** e - _MLO ** e)) ** (1.0 / e)
    xy = torch.stack([r * phi.cos(), r * phi.sin()], dim=1)
    return xy.float().double().cpu().numpy(), m.float().double().cpu().numpy()


def _counts(nx, ny):
    return torch.empty(ny * nx, dtype=torch.int32, device="cuda")


def _shot(seed, rays_x, rays_y, map_x, map_y, half=3.25):
    """A 1000-star field with the headline map's lens terms: its context, ray grid and square-pixel source map."""
    kappa_star, kappa_c, gamma = 0.3, 0.2, 0.3
    hx, hy = _lens_box(kappa_star + kappa_c, gamma, half)
    src = (-half, half, -half * map_y / map_x, half * map_y / map_x, map_x, map_y)
    rays = (-hx, hx, -hy, hy, rays_x, rays_y)
    xy, m = _stars(seed, 1000, kappa_star)
    ctx = M.mlens_create(xy, m, kappa_c, gamma, 0.0)
    return ctx, rays, src


def _learned_grid(c):
    """A ray box of the learned workload's shape (three times as wide as high, 0.47 theta_E cells)."""
    w = 0.46875
    nx, rows = 64 * c["tiles"] * c["cells"], -(-c["cells"] // 3)
    hx, hy = 0.5 * w * c["cells"], 0.5 * w * rows
    # square cells: as many 32-ray tile rows per cell as make the workload's ray density along y
    kty = 6 * c["tiles"]
    return (-hx, hx, -hy, hy, nx, 32 * kty * rows)


def _field(c, seed):
    xy, m = _stars(seed, c["stars"], 0.45)
    return M.mlens_create(xy, m, 0.05, 0.25, 0.0)


def _fit_params(c):
    return M.fit_params(cells_x=c["cells"], order=c["order"], use_network=1 if c["network"] else 0,
                        train_samples=c["samples"], epochs=c["epochs"], tolerance=5e-6)


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    c = case
    if c["kind"] == "shoot":
        xy, m = _stars(seed, c["stars"], c["kappa_star"], c["unit_masses"])
        ctx = M.mlens_create(xy, m, c["kappa_c"], c["gamma"], 0.0, c["precision"])
        rays = (-c["ray_hx"], c["ray_hx"], -c["ray_hy"], c["ray_hy"], c["rays_x"], c["rays_y"])
        h = c["src_half"]
        src = (-h, h, -h, h, c["map_x"], c["map_y"])
        beta = None
        if c["beta"]:
            n = c["rays_x"] * c["rays_y"]
            beta = torch.empty((n, 2), dtype=torch.float64, device="cuda") if c["precision"] == "fp64" else \
                torch.empty((n, 4), dtype=torch.float32, device="cuda")
        return dict(kind="shoot", ctx=ctx, rays=rays, src=src, counts=_counts(c["map_x"], c["map_y"]), beta=beta)
    if c["kind"] == "batch":
        rng = np.random.default_rng(seed)
        ctxs, rays, srcs = [], [], []
        maps = torch.empty((c["fields"], c["map"] * c["map"]), dtype=torch.int32, device="cuda")
        while len(ctxs) < c["fields"]:
            stars = int(round(math.exp(rng.uniform(math.log(c["stars_lo"]), math.log(c["stars_hi"])))))
            ks, kc, gm = rng.uniform(0.1, 0.8), rng.uniform(0.0, 0.3), rng.uniform(0.0, 0.6)
            low = min(abs(1.0 - ks - kc - gm), abs(1.0 - ks - kc + gm))
            half = math.floor(64.0 * 0.9 * _radius(stars, ks) * low / (1.5 * math.sqrt(2.0))) / 64.0
            if low < 0.1 or half <= 0.0:
                continue
            xy, m = _stars(int(rng.integers(1 << 31)), stars, ks)
            hx, hy = _lens_box(ks + kc, gm, half)
            ctxs.append(M.mlens_create(xy, m, kc, gm, 0.0))
            rays.append((-hx, hx, -hy, hy, c["rays"], c["rays"]))
            srcs.append((-half, half, -half, half, c["map"], c["map"]))
        return dict(kind="batch", batch=M.mlens_batch_create(ctxs, rays, srcs, list(maps)), maps=maps)
    if c["kind"] == "learned":
        ctx, rays = _field(c, seed), _learned_grid(c)
        M.mlens_fit_far_field(ctx, rays, _fit_params(c))
        h = rays[1] / 6.0
        return dict(kind="learned", ctx=ctx, rays=rays, src=(-h, h, -h, h, c["map"], c["map"]),
                    counts=_counts(c["map"], c["map"]))
    if c["kind"] == "fit":
        return dict(kind="fit", ctx=_field(c, seed), rays=_learned_grid(c), params=_fit_params(c))
    if c["kind"] == "bin":
        ctx, rays, src = _shot(seed, c["rays_x"], c["rays_y"], c["map"], c["map"])
        counts = _counts(c["map"], c["map"])
        beta = torch.empty((rays[4] * rays[5], 4), dtype=torch.float32, device="cuda")
        M.mlens_shoot_beta(ctx, rays, src, counts, beta)
        return dict(kind="bin", beta=beta, rays=rays, src=src, counts=torch.empty_like(counts), grid=c["grid_order"])
    if c["kind"] == "convolve":
        ctx, rays, src = _shot(seed, 4 * c["map_x"], 4 * c["map_y"], c["map_x"], c["map_y"])
        counts = _counts(c["map_x"], c["map_y"])
        M.mlens_shoot(ctx, rays, src, counts)
        size = c["size_px"] * (src[1] - src[0]) / c["map_x"]
        profile = M.MLENS_PROFILE_DISK if c["profile"] == "disk" else M.MLENS_PROFILE_GAUSSIAN
        work = torch.empty(M.mlens_convolve_workspace(src, profile, size), dtype=torch.uint8, device="cuda")
        return dict(kind="convolve", counts=counts, src=src, profile=profile, size=size,
                    out=torch.empty(counts.shape, dtype=torch.float32, device="cuda"), work=work,
                    scale=M.mlens_magnification_scale(rays, src))
    if c["kind"] == "curve":
        ctx, rays, src = _shot(seed, 4 * c["map"], 4 * c["map"], c["map"], c["map"])
        counts = _counts(c["map"], c["map"])
        M.mlens_shoot(ctx, rays, src, counts)
        h = src[1]
        b0, b1 = (-0.9 * h, -0.35 * h), (0.95 * h, 0.55 * h)
        return dict(kind="curve", map=counts.float() * M.mlens_magnification_scale(rays, src), src=src, b0=b0, b1=b1,
                    points=c["points"], out=torch.empty(c["points"], dtype=torch.float32, device="cuda"))
    raise ValueError(c["kind"])


# ----------------------------------------------------------------------- run
def run(state):
    s = state
    if s["kind"] == "shoot":
        if s["beta"] is None:
            M.mlens_shoot(s["ctx"], s["rays"], s["src"], s["counts"])
            return s["counts"]
        M.mlens_shoot_beta(s["ctx"], s["rays"], s["src"], s["counts"], s["beta"])
        return dict(counts=s["counts"], beta=s["beta"])
    if s["kind"] == "batch":
        M.mlens_batch_run(s["batch"])
        return s["maps"]
    if s["kind"] == "learned":
        M.mlens_shoot_learned(s["ctx"], s["rays"], s["src"], s["counts"])
        return s["counts"]
    if s["kind"] == "fit":
        report = M.mlens_fit_far_field(s["ctx"], s["rays"], s["params"])
        state = M.mlens_far_field_export(s["ctx"])
        out = {k: state[k] for k in ("params", "latents", "flags", "coef", "cell_start", "val_max_net",
                                     "val_max_series")}
        out["steps"], out["loss"] = int(report["train_steps"]), float(report["final_loss"])
        return out
    if s["kind"] == "bin":
        if s["grid"]:
            M.mlens_bin_grid(s["beta"], s["rays"], s["src"], s["counts"])
        else:
            M.mlens_bin(s["beta"], s["beta"].shape[0], s["src"], s["counts"])
        return s["counts"]
    if s["kind"] == "convolve":
        M.mlens_convolve(s["counts"], s["src"], s["profile"], s["size"], s["out"], scale=s["scale"], work=s["work"])
        return s["out"]
    M.mlens_light_curve(s["map"], s["src"], s["b0"], s["b1"], s["points"], s["out"])
    return s["out"]


# ---------------------------------------------------------------------- work
def work(case):
    """Bytes every input and output needs once, and floating operations of the method as stated: ten per ray
    and star (two differences, two squares and their sum, m / r^2, two products and two sums), a multiplication and an
    addition per tap and pass of the Gaussian, one subtraction and one addition per row of the disk."""
    c = case
    if c["kind"] == "shoot":
        n, px = c["rays_x"] * c["rays_y"], c["map_x"] * c["map_y"]
        return {"bytes": 16 * c["stars"] + 4 * px + (16 * n if c["beta"] else 0), "flops": 10.0 * n * c["stars"]}
    if c["kind"] == "batch":
        mean = (c["stars_hi"] - c["stars_lo"]) / math.log(c["stars_hi"] / c["stars_lo"])
        return {"bytes": c["fields"] * (16 * mean + 4 * c["map"] ** 2),
                "flops": 10.0 * c["fields"] * c["rays"] ** 2 * mean}
    if c["kind"] == "learned":
        r = _learned_grid(c)
        n, cells = r[4] * r[5], c["cells"] * -(-c["cells"] // 3)
        near = 9 * 0.45 * 0.46875 ** 2 / (math.pi * _mean_mass())  # stars of a 3 x 3 block of cells
        per = 10.0 * near + 8.0 * (c["order"] + 1) + (2.0 * 64 * 68 if c["network"] else 0.0)
        return {"bytes": 16 * c["stars"] + cells * (8 * (c["order"] + 2) + (128 if c["network"] else 0))
                + 4 * c["map"] ** 2, "flops": n * per}
    if c["kind"] == "fit":
        cells = c["cells"] * -(-c["cells"] // 3)
        train = 6.0 * (34 * 64 + 64 * 64 + 128) * c["samples"] * c["epochs"] if c["network"] else 0.0
        return {"bytes": 16 * c["stars"] + cells * (16 * 25 + 140),
                "flops": 25 * 8.0 * cells * c["stars"] + train + 64 * 2.0 * (34 * 64 + 64 * 64 + 128) * cells}
    if c["kind"] == "bin":
        n = c["rays_x"] * c["rays_y"]
        return {"bytes": 16 * n + 4 * c["map"] ** 2, "flops": 4 * n}
    if c["kind"] == "convolve":
        n = c["map_x"] * c["map_y"]
        taps = 2 * math.ceil(4 * c["size_px"]) + 1 if c["profile"] == "gaussian" else 2 * int(c["size_px"]) + 1
        return {"bytes": 8 * n, "flops": (4.0 if c["profile"] == "gaussian" else 2.0) * taps * n}
    return {"bytes": 4 * min(4 * c["points"], c["map"] ** 2) + 4 * c["points"], "flops": 25 * c["points"]}


# --------------------------------------------------------------------- exact
def _exact_beta(c, seed):
    n = c["rays_x"] * c["rays_y"]
    if not c["beta"] or n * c["stars"] > 4e9:
        return None
    xy, m = (torch.from_numpy(a).cuda() for a in _stars(seed, c["stars"], c["kappa_star"], c["unit_masses"]))

    def centres(h, k):
        return -h + (torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) * (2.0 * h / k)

    tx = centres(c["ray_hx"], c["rays_x"]).repeat(c["rays_y"])
    ty = centres(c["ray_hy"], c["rays_y"]).repeat_interleave(c["rays_x"])
    ax, ay = torch.zeros_like(tx), torch.zeros_like(ty)
    for k in range(0, c["stars"], 256):
        for i in range(0, n, 1 << 19):
            dx, dy = (t[i:i + (1 << 19), None] - xy[None, k:k + 256, d] for d, t in ((0, tx), (1, ty)))
            f = m[None, k:k + 256] / (dx * dx + dy * dy)
            ax[i:i + (1 << 19)] += (f * dx).sum(1)
            ay[i:i + (1 << 19)] += (f * dy).sum(1)
    bx = (1.0 - c["kappa_c"] - c["gamma"]) * tx - ax
    by = (1.0 - c["kappa_c"] + c["gamma"]) * ty - ay
    b = torch.stack([bx, by], dim=1)
    if c["precision"] == "fp64":
        return dict(counts=None, beta=b)
    hi = b.float().double()
    return dict(counts=None, beta=torch.cat([hi, b - hi], dim=1))


def _exact_coef(c, seed):
    """The far field's series coefficients -sum m s^p / (z - z_c)^(p + 1) over the stars outside the 3 x 3 block."""
    cells, rows = c["cells"], -(-c["cells"] // 3)
    if cells * rows * c["stars"] > 2e9:
        return None
    r = _learned_grid(c)
    w = (r[1] - r[0]) / cells
    xy, m = (torch.from_numpy(a).cuda() for a in _stars(seed, c["stars"], 0.45))
    x0, y0 = r[0] - w, r[2] - w
    cx, cy = ((xy[:, 0] - x0) / w).floor(), ((xy[:, 1] - y0) / w).floor()
    outside = (cx < 0) | (cx >= cells + 2) | (cy < 0) | (cy >= rows + 2)
    z = torch.complex(xy[:, 0], xy[:, 1])
    s = w * math.sqrt(0.5)
    out = torch.zeros((rows * cells, 25), dtype=torch.complex128, device="cuda")
    ex = torch.arange(cells * rows, device="cuda") % cells + 1
    ey = torch.arange(cells * rows, device="cuda") // cells + 1
    step = max(1, int(4e7 // c["stars"]))
    for b in range(0, rows * cells, step):
        ix, iy = ex[b:b + step, None], ey[b:b + step, None]
        near = ((cx[None] - ix).abs() <= 1) & ((cy[None] - iy).abs() <= 1) & ~outside[None]
        zc = torch.complex(x0 + (ix + 0.5) * w, y0 + (iy + 0.5) * w)
        v = s / torch.where(near, torch.full_like(zc, 1e30), z[None] - zc)
        t = -(m[None] / s) * v * (~near)
        for p in range(25):
            out[b:b + step, p] = t.sum(1)
            t = t * v
    return torch.view_as_real(out)


def _exact_convolution(c, seed):
    s = prepare(c, seed)
    nx, ny = c["map_x"], c["map_y"]
    a = s["counts"].view(ny, nx)
    dx, dy = (s["src"][1] - s["src"][0]) / nx, (s["src"][3] - s["src"][2]) / ny
    if c["profile"] == "gaussian":
        a = a.double()
        for axis, d in ((1, dx), (0, dy)):
            k = math.ceil(4.0 * s["size"] / d)
            w = torch.exp(-(torch.arange(-k, k + 1, dtype=torch.float64) * d) ** 2 / (2.0 * s["size"] ** 2))
            w = (w / w.sum()).tolist()
            n = a.shape[axis]
            out = torch.zeros_like(a)
            for q, wq in zip(range(-k, k + 1), w):
                lo, hi = max(0, -q), min(n, n - q)
                if hi > lo:
                    out.narrow(axis, lo, hi - lo).add_(a.narrow(axis, lo + q, hi - lo), alpha=wq)
            a = out
        return (a * s["scale"]).reshape(-1)
    p = torch.zeros((ny, nx + 1), dtype=torch.int64, device="cuda")
    p[:, 1:] = a.long().cumsum(1)
    i = torch.arange(nx, device="cuda")
    total, count = torch.zeros((ny, nx), dtype=torch.int64, device="cuda"), 0
    for dj in range(-int(s["size"] / dy) - 1, int(s["size"] / dy) + 2):
        if (dj * dy) * (dj * dy) > s["size"] * s["size"]:
            continue
        h = int(math.sqrt(s["size"] ** 2 - (dj * dy) ** 2) / dx) + 1
        while h >= 0 and (h * dx) * (h * dx) + (dj * dy) * (dj * dy) > s["size"] * s["size"]:
            h -= 1
        if h < 0:
            continue
        count += 2 * h + 1
        lo, hi = max(0, -dj), min(ny, ny - dj)
        if hi > lo:
            rows = p[lo + dj:hi + dj]
            total[lo:hi] += rows[:, (i + h + 1).clamp(max=nx)] - rows[:, (i - h).clamp(min=0)]
    return (total.double() * (s["scale"] / count)).reshape(-1)


def _exact_curve(c, seed):
    s = prepare(c, seed)
    n = c["map"]
    a = s["map"].view(n, n).double()
    t = torch.arange(c["points"], device="cuda", dtype=torch.float64) / max(1, c["points"] - 1)

    def axis(lo, hi, b0, b1):
        u = (b0 + t * (b1 - b0) - lo) / ((hi - lo) / n) - 0.5
        k = u.floor()
        return k.long().clamp(0, n - 1), (k.long() + 1).clamp(0, n - 1), u - k

    i0, i1, fx = axis(s["src"][0], s["src"][1], s["b0"][0], s["b1"][0])
    j0, j1, fy = axis(s["src"][2], s["src"][3], s["b0"][1], s["b1"][1])
    return (1 - fy) * ((1 - fx) * a[j0, i0] + fx * a[j0, i1]) + fy * ((1 - fx) * a[j1, i0] + fx * a[j1, i1])


def exact(case, seed):
    """What run() returns for these inputs, evaluated in 64 bits (maps are whole numbers: none)."""
    c = case
    if c["kind"] == "shoot":
        return _exact_beta(c, seed)
    if c["kind"] == "fit":
        coef = _exact_coef(c, seed)
        return None if coef is None else dict(coef=coef)
    if c["kind"] == "convolve":
        return _exact_convolution(c, seed)
    if c["kind"] == "curve":
        return _exact_curve(c, seed)
    return None
