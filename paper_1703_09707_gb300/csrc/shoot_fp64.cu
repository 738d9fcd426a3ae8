// shoot_fp64.cu -- IEEE FP64 variant of the direct sum (Eq. 3), the source
// position (Eq. 2) and the FP64 binning rule, with every operation correctly rounded
// in the order the equations state it, stars visited in input order.  Its beta and its
// maps therefore equal a plain IEEE FP64 evaluation of the same formulas bit for bit.
// This path exists for verification (mlens_trace), for the precision study and for exact
// per-ray references.
#include <cuda_runtime.h>
#include <stdint.h>

#include "mlens_dev.cuh"
#include "soft64.cuh"

namespace mlens {

constexpr int kT64 = 128;

// One staged star: its position in FP64 (converted once per CTA), its mass as a float and as
// a normalised significand and exponent; mant = 0 where the mass is zero or not normal.
struct Star64 {
    double2 xy;
    uint32_t mant;
    int em;
    float m;
};

__device__ __forceinline__ Star64 star64(float4 q)
{
    Star64 s;
    s.xy = make_double2((double)q.x, (double)q.y);
    const uint32_t b = __float_as_uint(q.z), e = b >> 23;  // masses are not negative
    const bool normal = e - 1u < 254u;
    s.mant = normal ? (b << 8) | 0x80000000u : 0u;
    s.em = (int)e - 127;
    s.m = q.z;
    return s;
}

// s += m d / r2 for both components of one star: the reference operations.
__device__ __noinline__ void add_star_fp64(double dx, double dy, float m, double &sx, double &sy)
{
    const double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), md = (double)m;
    sx = __dadd_rn(sx, __ddiv_rn(__dmul_rn(md, dx), r2));
    sy = __dadd_rn(sy, __ddiv_rn(__dmul_rn(md, dy), r2));
}

// The same sum with products and quotients formed on the integer pipes (soft64.cuh:
// the same roundings, so the same bits) wherever both differences lie within 2^+-200 and
// the mass is normal; every intermediate is then far from overflow and underflow.  Other
// stars (a ray level with a star or on it, massless stars) take the FP64 instructions.
// The five additions left to the FP64 unit hold it for 380 cycles per star and warp while
// the integer work takes about 330 issue slots; 509 x 387 rays of 5000 stars 54.3 ->
// 12.2 ms.  Also on the FP64 unit: one square, 12.9 ms; the products m d, 14.8 ms.  The sum
// of the squares on the integer pipes too: 15.2 ms.
__device__ __forceinline__ void alpha_fp64(double tx, double ty, const Star64 *st, int cnt, double &sx, double &sy)
{
    for (int k = 0; k < cnt; ++k) {
        const Star64 &q = st[k];
        const double dx = __dsub_rn(tx, q.xy.x), dy = __dsub_rn(ty, q.xy.y);
        const uint64_t bx = (uint64_t)__double_as_longlong(dx), by = (uint64_t)__double_as_longlong(dy);
        const uint32_t ex = (uint32_t)(bx >> 52) & 0x7ffu, ey = (uint32_t)(by >> 52) & 0x7ffu;
        if (ex - 823u <= 400u && ey - 823u <= 400u && q.mant != 0u) {
            const Soft64 x = soft_of(bx), y = soft_of(by);
            const double dx2 = __longlong_as_double((long long)soft_bits(soft_square(x), 0));
            const double dy2 = __longlong_as_double((long long)soft_bits(soft_square(y), 0));
            const Soft64 r2 = soft_of((uint64_t)__double_as_longlong(__dadd_rn(dx2, dy2)));
            const float f = __uint_as_float(0x3f800000u | ((uint32_t)(r2.n >> 40) & 0x7fffffu));
            const float e = fminf(fmaxf(rcp_approx(f), 0.5f), 0x1.fffffep-1f);
            const uint64_t r = soft_reciprocal(r2.n, __float_as_uint(e));
            const Soft64 ax = soft_div(soft_mul32(x, q.mant, q.em), r2, r);
            const Soft64 ay = soft_div(soft_mul32(y, q.mant, q.em), r2, r);
            sx = __dadd_rn(sx, __longlong_as_double((long long)soft_bits(ax, bx & uint64_t(1) << 63)));
            sy = __dadd_rn(sy, __longlong_as_double((long long)soft_bits(ay, by & uint64_t(1) << 63)));
        } else {
            add_star_fp64(dx, dy, q.m, sx, sy);
        }
    }
}

__device__ __forceinline__ double ray_coord(double x0, double x1, int n, int i)
{
    return __dadd_rn(x0, __dmul_rn(__dadd_rn((double)i, 0.5), __ddiv_rn(__dsub_rn(x1, x0), (double)n)));
}

__device__ __forceinline__ int pixel_fp64(double bx, double by, const BinGrid &g)
{
    if (!isfinite(bx) || !isfinite(by)) return -2;
    const double ux = floor(__dmul_rn(__dsub_rn(bx, g.x0), __ddiv_rn((double)g.nx, __dsub_rn(g.x1, g.x0))));
    const double uy = floor(__dmul_rn(__dsub_rn(by, g.y0), __ddiv_rn((double)g.ny, __dsub_rn(g.y1, g.y0))));
    if (ux < 0.0 || ux >= (double)g.nx || uy < 0.0 || uy >= (double)g.ny) return -1;
    return (int)uy * g.nx + (int)ux;
}

// GRID: rays of a grid (one per thread, 32 x 4 threads per CTA), binned;
// otherwise: k arbitrary positions from `theta`, beta written, nothing binned.
template <bool GRID>
__global__ void __launch_bounds__(kT64, 8) k_fp64(ShootArgs a, const double2 *theta, double2 *beta, int64_t k, int by0)
{
    __shared__ Star64 sq[kT64];
    __shared__ unsigned sred[3];
    const int tid = threadIdx.x;
    if (tid == 0) sred[0] = sred[1] = sred[2] = 0u;

    int i = 0, j = 0;
    int64_t r = 0;
    bool ok;
    double tx, ty;
    if (GRID) {
        i = blockIdx.x * 32 + (tid & 31);
        j = (by0 + (int)blockIdx.y) * 4 + (tid >> 5);
        ok = i < a.rays.nx && j < a.rays.ny;
        tx = ray_coord(a.rays.x0, a.rays.x1, a.rays.nx, i);
        ty = ray_coord(a.rays.y0, a.rays.y1, a.rays.ny, j);
    } else {
        r = (int64_t)blockIdx.x * kT64 + tid;
        ok = r < k;
        const double2 t = ok ? theta[r] : make_double2(0.0, 0.0);
        tx = t.x;
        ty = t.y;
    }
    const double kc = a.lens.kc, g1 = a.lens.g1, g2 = a.lens.g2;
    double sx = __dadd_rn(__dmul_rn(__dadd_rn(kc, g1), tx), __dmul_rn(g2, ty));
    double sy = __dadd_rn(__dmul_rn(g2, tx), __dmul_rn(__dsub_rn(kc, g1), ty));
    for (int64_t s0 = 0; s0 < a.nstars; s0 += kT64) {
        const int cnt = (int)min((int64_t)kT64, a.nstars - s0);
        __syncthreads();
        if (tid < cnt) sq[tid] = star64(a.stars[s0 + tid]);
        __syncthreads();
        alpha_fp64(tx, ty, sq, cnt, sx, sy);
    }
    const double bx = __dsub_rn(tx, sx), by = __dsub_rn(ty, sy);
    if (!GRID) {
        if (ok) beta[r] = make_double2(bx, by);
        return;
    }
    unsigned nb = 0, no = 0, nn = 0;
    if (ok) {
        const int p = pixel_fp64(bx, by, a.bin);
        if (p >= 0) {
            atomicAdd(&a.counts[p], 1u);
            nb = 1;
        } else if (p == -1) {
            no = 1;
        } else {
            nn = 1;
        }
        if (a.beta_out) reinterpret_cast<double2 *>(a.beta_out)[(int64_t)j * a.rays.nx + i] = make_double2(bx, by);
    }
    __syncthreads();
    stats_add_block(nb, no, nn, sred, a.stats);
}

cudaError_t launch_shoot_fp64(const ShootArgs &a, cudaStream_t s, int row0, int row1)
{
    // blocks of 32 x 4 rays: rows [row0, row1) in block rows (row0 a multiple of 4)
    const int tx = (a.rays.nx + 31) / 32;
    const int r1 = row1 < 0 || row1 > a.rays.ny ? a.rays.ny : row1;
    const int ty = (r1 + 3) / 4;
    for (int by0 = row0 / 4; by0 < ty; by0 += 65535) {
        const dim3 grid((unsigned)tx, (unsigned)min(65535, ty - by0));
        k_fp64<true><<<grid, kT64, 0, s>>>(a, nullptr, nullptr, 0, by0);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_trace_fp64(const float4 *stars, int64_t nstars, const LensTerms &lens, const double2 *theta,
                              double2 *beta, int64_t k, cudaStream_t s)
{
    if (k <= 0) return cudaSuccess;
    ShootArgs a{};
    a.stars = stars;
    a.nstars = nstars;
    a.lens = lens;
    int64_t nb = (k + kT64 - 1) / kT64;
    if (nb > 0x7fffffff) return cudaErrorInvalidConfiguration;
    k_fp64<false><<<(unsigned)nb, kT64, 0, s>>>(a, theta, beta, k, 0);
    return cudaGetLastError();
}

}  // namespace mlens
