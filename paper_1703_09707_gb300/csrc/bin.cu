// bin.cu -- the binning step of Algorithm 1 on its own: float-pair source
// positions -> exact pixel -> shared-memory-privatised window histogram -> global
// uint32 counts.  Same pixel rule, window and atomics as the fused shooting kernels.
//
// Two record orders.  Flat: a CTA takes 4096 consecutive records.  Grid: the
// records are a row-major nx x ny ray grid and a CTA takes a 64 x 64 block of
// it; neighbouring rays land on neighbouring pixels, so most of the block's
// records hit its 64 x 64 window, placed on the block's middle record (consecutive
// records of one grid row would instead spread along a strip of the map far longer
// than the window).
//
// Bound by HBM in grid order: 8192^2 records (1.07 GB) into 1024^2 pixels in 0.160 ms
// = 6.7 TB/s, 0.99 of the measured copy rate; 0.292 ms, bound by its 114 instructions a
// record, before the fast pixel rule (mlens_dev.cuh), 0.164 before the clears ran
// alongside the first loads (clear.cu).  Flat order 0.271 -> 0.214 ms, bound by the global
// atomics of records outside the window.  Four records in flight per thread and eight
// CTAs of 32 registers per SM; against 0.164: eight records and four CTAs 0.181 ms, eight
// and five 0.170, sixteen and three 0.210; 8192 records per CTA 0.167.
#include <cuda_runtime.h>
#include <stdint.h>

#include "mlens_dev.cuh"

namespace mlens {

constexpr int kBinThreads = 256;
constexpr int kBinPer = 4;                                    // records per thread and round
constexpr int kBinRounds = 4;
constexpr int kBinCnt = kBinPer * kBinRounds;                 // records per thread
constexpr int kBinRecs = kBinThreads * kBinCnt;               // 4096 records per CTA
constexpr int kBinTileX = 64;                                 // grid order: 64 x 64 records per CTA
constexpr int kBinTileY = kBinRecs / kBinTileX;
constexpr int kBinRowStep = kBinThreads / kBinTileX;          // rows between a thread's records

template <bool GRID>
__device__ __forceinline__ void bin_block(const BinArgs &a)
{
    __shared__ __align__(16) uint32_t hist[kWin * kWin];
    __shared__ unsigned sred[3];
    const int tid = threadIdx.x;
    // record r of this thread is first[r * step], r < cnt; in grid order r counts rows of
    // the block (kBinRowStep apart), in flat order runs of kBinThreads records
    const float4 *first, *centre;
    int64_t step;
    int cnt;
    if (GRID) {
        const int c0 = blockIdx.x * kBinTileX, col = c0 + tid % kBinTileX;
        const int r0 = blockIdx.y * kBinTileY, row = r0 + tid / kBinTileX;
        first = a.beta + (int64_t)row * a.rnx + col;
        step = (int64_t)kBinRowStep * a.rnx;
        cnt = col < a.rnx ? min(kBinCnt, (a.rny - row + kBinRowStep - 1) / kBinRowStep) : 0;
        centre = a.beta + (int64_t)min(r0 + kBinTileY / 2, a.rny - 1) * a.rnx + min(c0 + kBinTileX / 2, a.rnx - 1);
    } else {
        const int64_t i0 = (int64_t)blockIdx.x * kBinRecs;
        first = a.beta + i0 + tid;
        step = kBinThreads;
        cnt = (int)min((int64_t)kBinCnt, (a.n - i0 - tid + kBinThreads - 1) / kBinThreads);
        centre = a.beta + min(i0 + kBinRecs / 2, a.n - 1);
    }
    cnt = max(cnt, 0);
    float4 v[kBinPer];
    auto load = [&](int r0) {
#pragma unroll
        for (int r = 0; r < kBinPer; ++r)
            if (r0 + r < cnt) v[r] = __ldcs(first + (r0 + r) * step);
    };
    load(0);
    const float4 vc = *centre;
    hist_zero(hist);
    if (tid == 0) sred[0] = sred[1] = sred[2] = 0u;
    const WinHist<> W = make_window(hist, win_origin(pair_axis_rough(vc.x, a.bin.ax), a.bin.nx),
                                  win_origin(pair_axis_rough(vc.y, a.bin.ay), a.bin.ny), a.bin);
    __syncthreads();
    pdl_wait();  // the map's and the counters' clears
    unsigned no = 0, nn = 0;
#pragma unroll
    for (int r0 = 0; r0 < kBinCnt; r0 += kBinPer) {
        if (r0 > 0) load(r0);
#pragma unroll
        for (int r = 0; r < kBinPer; ++r)
            if (r0 + r < cnt) bin_pair<false>(v[r].x, v[r].y, v[r].z, v[r].w, a.bin, W, a.counts, no, nn);
    }
    __syncthreads();
    hist_flush(W, a.bin, a.counts);
    stats_add_block((unsigned)cnt - no - nn, no, nn, sred, a.stats);
}

__global__ void __launch_bounds__(kBinThreads, 8) k_bin_grid(BinArgs a) { bin_block<true>(a); }
__global__ void __launch_bounds__(kBinThreads, 8) k_bin_flat(BinArgs a) { bin_block<false>(a); }

// 72 %: eight CTAs of a 16 KB window and 1 KB reserved, 137 of 228 KB, in the next size there
// is.  2^16 random records into 4096^2 pixels 29.8 -> 15.4 us (with the clear and the kernel
// one after the other 16.0), 500^2 rays in order 23.6 -> 16.1 us.  Below four CTAs per SM;
// more fill the chip however they are placed, and then do better behind any clear: 2^22
// records into 2900^2 pixels 31 us, 33 us behind the same carveout, 8192^2 rays into 1024^2 pixels
// 158.8 and 160.1 us.  (The largest carveout spreads them too, but leaves the kernel little L1:
// 8192^2 rays into 4096^2 pixels 224 -> 238 us.)
int bin_clear_carveout(int64_t n)
{
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return -1;
    return n <= (int64_t)kBinRecs * 4 * nsm ? 72 : -1;
}

cudaError_t launch_bin(const BinArgs &a, cudaStream_t s)
{
    if (a.n <= 0) return cudaSuccess;
    if (a.rnx > 0) {
        const int64_t tx = (a.rnx + kBinTileX - 1) / kBinTileX, ty = (a.rny + kBinTileY - 1) / kBinTileY;
        if (tx > 0x7fffffff || ty > 65535) return cudaErrorInvalidConfiguration;
        return launch_pdl(k_bin_grid, dim3((unsigned)tx, (unsigned)ty), dim3(kBinThreads), 0, s, a);
    }
    const int64_t nb = (a.n + kBinRecs - 1) / kBinRecs;
    if (nb > 0x7fffffff) return cudaErrorInvalidConfiguration;
    return launch_pdl(k_bin_flat, dim3((unsigned)nb), dim3(kBinThreads), 0, s, a);
}

}  // namespace mlens
