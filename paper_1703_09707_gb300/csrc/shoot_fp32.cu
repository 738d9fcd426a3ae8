// shoot_fp32.cu -- the FP32 direct-sum ray-shooting kernels (Algorithm 1 with
// the deflection of Eq. 3 and the source position of Eq. 2), fused with the
// binning step, for one field (a grid of tiles) and for many fields (one
// persistent launch over a work queue of (field, tile) items).
//
// One CTA of 128 threads owns half a 64 x (8*NP) tile of the ray grid; each thread
// owns 2*NP rays of one grid column, processed as NP packed pairs with the
// Blackwell f32x2 instructions (FMUL2/FFMA2), so one instruction serves two rays.
// Stars stream through shared memory in stages of 128; a stage holds, per star, the
// differences y_ray - y_star of the tile's rows, the mass and the re-centred x
// (tile.cuh RowStage), read as broadcasts.  Per star and ray the work is FFMA (r^2),
// MUFU.RCP, FMUL (m/r^2), 2 FFMA (accumulate): the MUFU reciprocal (16 per SM per
// clock) is the unit nearest saturation (shoot_half has the count of both pipes).
// A CTA takes 37 KB: four per SM.  (The API's star stage of 256 or 512 would not fit
// four; every setting stages 128, which never changes the arithmetic.)
//
// Precision (MLENS_PREC_FP32): rays and stars are relative to an FP32 tile
// centre c, so differences of nearby positions carry no absolute-coordinate
// rounding.  Terms are accumulated in plain FP32 over 32 stars and each 32-star
// partial is added to the running sum with Kahan compensation.  The
// smooth+shear part A c of the tile centre is formed in FP64 once per tile, and
// beta = A c + A delta - S is assembled as a float pair, so the only rounding
// left at the full coordinate scale is the exact binning rule's.  The tile shape NP
// changes the last bits (it moves the tile centres).
// MLENS_PREC_FP32_NAIVE keeps absolute coordinates and one running FP32 sum
// (Algorithm 1 written in single precision).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "tile.cuh"

namespace mlens {

template <int NP, bool NAIVE, int NRP>
__global__ void __launch_bounds__(kHalfThreads, 4) k_shoot_fp32(ShootArgs a, int by0)
{
    __shared__ __align__(16) ShootSmem<NP, NAIVE> sm;
    __shared__ TileShared ts;
    shoot_half<NP, NAIVE, NRP>(a, blockIdx.x, by0 + (int)blockIdx.y, sm, ts);
}

// Persistent kernel over many fields: CTAs pull (field, half tile) items from one
// atomic counter until the queue is empty.  Items are numbered field by field in
// the order `order` (heaviest field first, so the tail is made of light items);
// begin[k] is the first item of the k-th field in that order (begin[nf] = total).
template <int NP, int NRP>
__global__ void __launch_bounds__(kHalfThreads, 4)
    k_shoot_batch(const ShootArgs *fields, const int *order, const int64_t *begin, int nf, int64_t total,
                  unsigned long long *counter)
{
    __shared__ __align__(16) ShootSmem<NP> sm;
    __shared__ TileShared ts;
    __shared__ long long s_item;
    for (;;) {
        __syncthreads();  // everyone has finished with the previous item number
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const int64_t item = s_item;
        if (item >= total) break;
        int lo = 0, hi = nf - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (begin[mid] <= item) lo = mid;
            else hi = mid - 1;
        }
        const ShootArgs &A = fields[order[lo]];
        const int64_t t = item - begin[lo];
        const int hx = halves_x(A.rays);
        shoot_half<NP, false, NRP>(A, (int)(t % hx), (int)(t / hx), sm, ts);
    }
}

// Tile rows [ty0, ty1) of the grid; ty1 < 0 means through the last tile row.
static inline int tile_row_end(const ShootArgs &a, int np, int ty1)
{
    const int ty = (a.rays.ny + tile_rows(np) - 1) / tile_rows(np);
    return ty1 < 0 || ty1 > ty ? ty : ty1;
}

// Dynamic shared memory that spreads a grid of few CTAs evenly.  Where ceil(CTAs / SMs) = c
// is below the four that fit an SM, c + 1 are made not to fit: left to themselves the CTAs
// do not always spread (440 on 152 SMs: four on some SMs; 256 behind other work on the
// stream: three), and an SM's reciprocals take the time of all its CTAs.
// 1e7 stars x 512^2 rays, unsplit (256 CTAs): 981 -> 651 ms;
// 3000 stars x 704 x 640 rays (440): 334 -> 308 us.
// c = 1 leaves room for two: such grids spread by themselves behind a clear of the same
// carveout (clear.cu), and one CTA keeps an SM less than two thirds busy, which maps on
// other streams can use.  512 x 256 rays of 3000 stars (128 CTAs), a map on each of four
// streams 105 -> 83 us a map, on two 108 -> 100, on one 127 either way.
static cudaError_t spread_smem(int64_t ctas, size_t used, size_t *dyn, size_t *most)
{
    *dyn = 0;
    int dev = 0, nsm = 0, sm_bytes = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || ctas > 3 * (int64_t)nsm) return e;
    e = cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess) return e;
    // c of these bytes fit an SM, c + 1 do not
    auto pad = [&](int c) { return (size_t)sm_bytes / (c + 1) + 128 - used - (size_t)reserved; };
    *dyn = pad(ctas <= nsm ? 2 : (int)((ctas + nsm - 1) / nsm));
    *most = pad(2);
    return cudaSuccess;
}

template <int NP, bool NAIVE, int NRP>
static cudaError_t launch_t(const ShootArgs &a, cudaStream_t s, int ty0, int ty1, bool pdl)
{
    // tile rows in launches of at most 65535 (the grid's y limit)
    const int ty = tile_row_end(a, NP, ty1);
    if (ty <= ty0) return cudaSuccess;
    auto *const k = k_shoot_fp32<NP, NAIVE, NRP>;
    size_t dyn = 0, most = 0;
    cudaError_t e = spread_smem((int64_t)halves_x(a.rays) * (ty - ty0),
                                sizeof(ShootSmem<NP, NAIVE>) + sizeof(TileShared), &dyn, &most);
    if (e == cudaSuccess && dyn > 0) e = allow_dynamic_smem(k, dyn, most);
    if (e != cudaSuccess) return e;
    for (int by0 = ty0; by0 < ty; by0 += 65535) {
        const dim3 grid((unsigned)halves_x(a.rays), (unsigned)min(65535, ty - by0));
        if (pdl && by0 == ty0) {
            e = launch_pdl(k, grid, dim3(kHalfThreads), dyn, s, a, by0);
        } else {
            k<<<grid, kHalfThreads, dyn, s>>>(a, by0);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <bool NAIVE, int NRP>
static cudaError_t launch_sel(const ShootArgs &a, int np, cudaStream_t s, int ty0, int ty1, bool pdl)
{
    return np == 2 ? launch_t<2, NAIVE, NRP>(a, s, ty0, ty1, pdl) : launch_t<4, NAIVE, NRP>(a, s, ty0, ty1, pdl);
}

cudaError_t launch_shoot_fp32(const ShootArgs &a, int pairs_per_thread, bool naive, cudaStream_t s, int fma_pairs,
                              int ty0, int ty1, bool pdl)
{
    if (naive) return launch_sel<true, 0>(a, pairs_per_thread, s, ty0, ty1, pdl);
    return fma_pairs ? launch_sel<false, 1>(a, pairs_per_thread, s, ty0, ty1, pdl)
                     : launch_sel<false, 0>(a, pairs_per_thread, s, ty0, ty1, pdl);
}

int64_t tiles_of(const RayGrid &r, int pairs_per_thread)
{
    const int ty = tile_rows(pairs_per_thread);
    return (int64_t)((r.nx + kTileX - 1) / kTileX) * (int64_t)((r.ny + ty - 1) / ty);
}

template <int NP, int NRP>
static cudaError_t grid_b(int *grid)
{
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_shoot_batch<NP, NRP>, kHalfThreads, 0);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    *grid = nsm * (per_sm > 0 ? per_sm : 1);
    return cudaSuccess;
}

cudaError_t batch_grid_size(int pairs_per_thread, int *grid, int fma_pairs)
{
    if (pairs_per_thread == 2) return fma_pairs ? grid_b<2, 1>(grid) : grid_b<2, 0>(grid);
    return fma_pairs ? grid_b<4, 1>(grid) : grid_b<4, 0>(grid);
}

template <int NP, int NRP>
static cudaError_t launch_b(const BatchLaunch &b, cudaStream_t s)
{
    const int64_t want = b.grid > 0 ? b.grid : 1;
    const unsigned grid = (unsigned)(b.total < want ? (b.total > 0 ? b.total : 1) : want);
    k_shoot_batch<NP, NRP><<<grid, kHalfThreads, 0, s>>>(b.fields, b.order, b.begin, b.nfields, b.total, b.counter);
    return cudaGetLastError();
}

cudaError_t launch_shoot_batch(const BatchLaunch &b, int pairs_per_thread, cudaStream_t s, int fma_pairs)
{
    if (pairs_per_thread == 2) return fma_pairs ? launch_b<2, 1>(b, s) : launch_b<2, 0>(b, s);
    return fma_pairs ? launch_b<4, 1>(b, s) : launch_b<4, 0>(b, s);
}

}  // namespace mlens
