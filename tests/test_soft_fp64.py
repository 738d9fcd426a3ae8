"""The FP64 direct sum's products and quotients on the integer pipes (csrc/soft64.cuh).

On the CPU the same integer steps are evaluated with Python integers and compared with the
IEEE operations of the machine, on random significands, on ones with long runs of zeros or
ones and on quotients next to rounding midpoints, with reciprocal estimates anywhere within
their allowed error.  On the GPU the FP64 source positions equal the oracle's bit for bit
where the kernel changes path: rays level with stars and on them, massless and subnormal
masses, positions of extreme magnitude, star counts around its stage."""
import struct

import numpy as np
import pytest

M64, TOP = (1 << 64) - 1, 1 << 63


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def f32_bits(x):
    return struct.unpack("<I", struct.pack("<f", x))[0]


def i32(x):
    x &= 0xffffffff
    return x - (1 << 32) if x >> 31 else x


def i64(x):
    x &= M64
    return x - (1 << 64) if x >> 63 else x


def soft_of(b):
    return ((b << 11) & M64) | TOP, ((b >> 52) & 0x7ff) - 1023


def soft_bits(n, e):
    return (((e + 1022) << 52) + (n >> 11)) & M64


def soft_round(n, e):
    r = (n + 0x3ff + ((n >> 11) & 1)) & M64
    return (r & ~0x7ff & M64) | TOP, e + 1 - (r >> 63)


def soft_product(hi, rest, e):
    n = hi | (1 if rest else 0)
    top = n >> 63
    return soft_round((n << (1 - top)) & M64, e + top)


def soft_square(n, e):
    p = n * n
    return soft_product(p >> 64, p & M64, 2 * e)


def soft_mul32(n, e, m, em):
    lo = (n & 0xffffffff) * m
    return soft_product((n >> 32) * m + (lo >> 32), lo & 0xffffffff, e + em)


def soft_reciprocal(b, y):
    r0 = ((y << 8) | 0x80000000) & 0xffffffff
    lo = (b & 0xffffffff) * r0
    e0 = i32(i64(TOP - ((b >> 32) * r0 + (lo >> 32))) >> 11)
    r1 = ((r0 << 32) + ((i32(r0 >> 1) * e0) >> 19)) & M64
    e1 = i32(i64(TOP - (b * r1 >> 64)))
    return (r1 + ((i32(r1 >> 33) * e1) >> 30) - 3) & M64


def soft_div(a, ea, b, eb, r):
    q = a * r >> 64
    top = q >> 63
    n, e = (q << (1 - top)) & M64, ea - eb - 1 + top
    low = n & 0x7ff
    n &= ~0x7ff
    up = low >= 0x400
    if 0x400 - 12 <= low < 0x400:
        mid = (n >> 10) | 1
        up = i64(((a >> 11) << (54 - top)) - mid * (b >> 11)) > 0
    n = (n + (0x800 if up else 0)) & M64
    return n | TOP, e + 1 - (n >> 63)


def operands(rng, k, span):
    m = rng.integers(0, 1 << 52, k, dtype=np.uint64)
    s = rng.integers(0, 52, k, dtype=np.uint64)
    kind = rng.integers(0, 6, k)
    one = np.uint64(1)
    m = np.where(kind == 0, m & ~((one << s) - one), m)
    m = np.where(kind == 1, m | ((one << s) - one), m)
    m = np.where(kind == 2, one << s, m)
    m = np.where(kind == 3, ((one << np.uint64(52)) - one) ^ (one << s), m)
    e = rng.integers(1023 - span, 1023 + span + 1, k).astype(np.uint64)
    return ((e << np.uint64(52)) | (m & np.uint64((1 << 52) - 1))).view(np.float64)


def estimate(rng, n):
    """A float within its allowed error of 2^63 / n, clamped as the kernel clamps it."""
    y = np.float32((TOP / n) * (1.0 + rng.uniform(-1, 1) * 2.0 ** -22))
    return f32_bits(min(max(float(y), 0.5), float(np.float32(1.0 - 2.0 ** -24))))


def test_products_equal_the_ieee_ones():
    rng = np.random.default_rng(1)
    for a, b in zip(operands(rng, 20000, 200).tolist(), operands(rng, 20000, 100).astype(np.float32).tolist()):
        sa = soft_of(bits(a))
        assert soft_bits(*soft_square(*sa)) == bits(a * a), a
        n, e = soft_of(bits(b))
        assert soft_bits(*soft_mul32(*sa, n >> 32, e)) == bits(a * b), (a, b)


def test_quotients_equal_the_ieee_ones():
    rng = np.random.default_rng(2)
    a, b = operands(rng, 20000, 200), operands(rng, 20000, 200)
    # numerators whose quotient lies next to a midpoint: b (q + half an ulp), rounded
    q = operands(rng, 20000, 1)
    near = np.array([float(int(x * 2.0 ** 60) * (int(bits(y) & ((1 << 52) - 1)) * 2 + (1 << 53) + 1)) * 2.0 ** -114
                     for x, y in zip(b / 2.0 ** np.floor(np.log2(b)), q)])
    for x, y in list(zip(a.tolist(), b.tolist())) + list(zip(near.tolist(), (b / 2.0 ** np.floor(np.log2(b))).tolist())):
        (na, ea), (nb, eb) = soft_of(bits(x)), soft_of(bits(y))
        r = soft_reciprocal(nb, estimate(rng, nb))
        assert 0 <= (1 << 127) - nb * r < 5 * nb, y
        assert soft_bits(*soft_div(na, ea, nb, eb, r)) == bits(x / y), (x, y)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
def test_gpu_positions_equal_the_oracle(n):
    import oracle
    import workloads as W
    from gpu_util import shoot_gpu
    from paper_1703_09707_gb300 import mlens as M
    f = W.random_field(W.SEED_BASE + 400 + n, n, kappa_star=0.35, kappa_c=0.1, gamma1=0.2, gamma2=0.07)
    rays, src = W.Grid(-4.0, 4.0, -4.0, 4.0, 67, 35), W.Grid(-2.0, 2.0, -2.0, 2.0, 50, 40)
    th = oracle.ray_theta(rays, np.arange(rays.n, dtype=np.int64))
    f.xy[0] = np.float32(th[100])          # as near a ray as a float is
    f.xy[-1, 1] = np.float32(th[700, 1])
    if n > 2:
        f.m[1], f.m[2] = 0.0, float(np.float32(1e-41))
    c, st, b = shoot_gpu(f, rays, src, prec=M.MLENS_PREC_FP64)
    want = oracle.beta_rays(rays, np.arange(rays.n, dtype=np.int64), f)
    same = b.view(np.uint64) == want.view(np.uint64)
    assert (same | (np.isnan(b) & np.isnan(want))).all()
    rng = np.random.default_rng(n)
    t = rng.normal(0.0, 1.0, (200, 2)) * 10.0 ** rng.uniform(-60, 140, (200, 1))
    t[:4] = [f.xy[0], f.xy[0] + [1e-13, 0.0], [f.xy[-1, 0], 3.0], [0.0, 0.0]]
    ctx = M.mlens_create(f.xy, f.m, f.kappa_c, f.gamma1, f.gamma2)
    got, ref = M.mlens_trace(ctx, t), oracle.beta(t, f)
    ctx.close()
    assert ((got.view(np.uint64) == ref.view(np.uint64)) | (np.isnan(got) & np.isnan(ref))).all()
