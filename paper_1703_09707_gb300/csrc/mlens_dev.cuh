// mlens_dev.cuh -- device helpers shared by the libmlens kernels:
// float-pair arithmetic, the exact float-pair binning rule (the source-pixel
// conversion of Algorithm 1) and the privatised, warp-aggregated histogram
// epilogue that performs its "mag[j_s, i_s] += 1".
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mlens_internal.h"

namespace mlens {

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialisation may begin while the one before it finishes; pdl_wait() returns once that
// one has completed and its writes are visible, and pdl_launch_next() lets the next
// kernel begin launching once every CTA of this one has called it.  Both do nothing in a
// kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------ float pairs
// Knuth's error-free TwoSum: s + e == a + b exactly, s = fl(a + b).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    float x = __fadd_rn(a, b);
    float bb = __fsub_rn(x, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(x, bb)), __fsub_rn(b, bb));
    s = x;
}

// MUFU reciprocal (max error 1 ulp; 1/0 = +inf).
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ------------------------------------------------------- exact binning rule
// Pixel of one axis for beta = bh + bl (an unevaluated float pair):
// floor((bh + bl - x0) * s) with x0 = x0h + x0l, s = sh + sl, evaluated as
// float pairs and floored exactly; -1 when outside [0, n).  The operation
// sequence is part of the library's contract (a CPU re-binning with the same
// float32 operations reproduces the GPU map bit for bit).
__device__ __forceinline__ int pair_axis_exact(float bh, float bl, const AxisPair &A)
{
    float dh, dl;
    two_sum(bh, -A.x0h, dh, dl);
    float t = __fsub_rn(bl, A.x0l);
    dl = __fadd_rn(dl, t);
    two_sum(dh, dl, dh, dl);
    float uh = __fmul_rn(dh, A.sh);
    float ul = __fmaf_rn(dh, A.sh, -uh);
    ul = __fmaf_rn(dh, A.sl, ul);
    ul = __fmaf_rn(dl, A.sh, ul);
    two_sum(uh, ul, uh, ul);
    if (!(uh == uh) || isinf(uh)) return -1;
    float p = floorf(uh);
    if (p == uh && ul < 0.0f) p = __fsub_rn(p, 1.0f);
    if (p < 0.0f || p >= (float)A.n) return -1;
    return (int)p;
}

// The same pixels, usually without the pair arithmetic, for both axes at once in
// packed f32x2.  With V = (bh + bl - x0) s the value pair_axis_exact floors (to about
// 2^-45 relative), the rule forms u ~ V - 1/2 as
//     d = fl(bh - x0h),  w = fl(bl sh + c),  u = fl(d sh + w),  c = fl(-x0l s - 1/2),
// and takes the integer nearest u, k, which is floor(V) unless V lies within the error
// of a pixel edge.  Error of u against V - 1/2, for |bl sh| <= 1/4: rounding d and
// leaving out d sl, 2 2^-24 |d sh|; leaving out bl sl, 2^-24 / 4; rounding c and w,
// 2^-24 (2 |c| + 1/4); rounding u, 2^-24 |u|; with |d sh| <= |u| + |c| + 1/2 together
//     B <= 2^-24 (3 |u| + 4 |c| + 1.5) (1 + 2^-20) + 2^-45 |V|.
// The host's del = 1.001 2^-24 (3 n + 4 |c| + 8) is above B for -2 <= u <= n + 2, and
// beyond that range B stays below u's distance from the map (n <= 2^20), so there the
// pixel is outside the map as the exact rule's is.  k comes from the magic number
// M = 1.5 2^23: t = fl(u + M) has k in its low bits where |u| < 2^22, so k =
// bits(t) - bits(M) without a conversion instruction; t - M and u - k are exact, and
// u is decided when |u - k| <= 1/2 - del.  Where |u| >= 2^22, bits(t) - bits(M) is at
// least 2^22 as an unsigned number: outside the map.  A non-finite component makes
// u - k a NaN, which is never decided.
// NORM: the pair is normalised (|bl| <= 2^-24 |bh|), so |bl sh| <= 1/4 needs no test
// (make_fast refuses origins beyond 2^21 pixels).
// Decides all but about 4 del of the records (7e-4 on a 1024^2 map) without a
// conversion or a rounding instruction (both run at the MUFU's rate).  Against a test of
// each axis with two floors and scalar bounds: a series-only map of 2.7e8 rays 2.94 ->
// 2.47 ms, 1000^2 rays of 100 stars 51.3 -> 48.9 us, the standalone kernel 0.292 ->
// 0.181 ms before its own launch shape was set.
constexpr float kMagic = 12582912.0f;
template <bool NORM>
__device__ __forceinline__ bool fast_pixel(float xh, float yh, float xl, float yl, const FastBin &F, int &px, int &py)
{
    const float2 d = __fadd2_rn(make_float2(xh, yh), F.nx0);
    const float2 w = __ffma2_rn(make_float2(xl, yl), F.s, F.c);
    const float2 u = __ffma2_rn(d, F.s, w);
    const float2 t = __fadd2_rn(u, make_float2(kMagic, kMagic));
    const float2 k = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
    px = __float_as_int(t.x) - __float_as_int(kMagic);
    py = __float_as_int(t.y) - __float_as_int(kMagic);
    const bool ok = fabsf(__fsub_rn(u.x, k.x)) <= F.thr.x && fabsf(__fsub_rn(u.y, k.y)) <= F.thr.y;
    return NORM ? ok : ok && fabsf(xl) <= F.blmax.x && fabsf(yl) <= F.blmax.y;
}

// The exact rule for a record the fast one leaves undecided, out of line so that the
// unrolled record loops stay small.
struct BinPix {
    int px, py;  // -1: outside the map on that axis
    bool finite;
};

static __device__ __noinline__ BinPix exact_pixel(float xh, float yh, float xl, float yl, AxisPair ax, AxisPair ay)
{
    BinPix p{-1, -1, isfinite(xh) && isfinite(yh) && isfinite(xl) && isfinite(yl)};
    if (!p.finite) return p;
    p.px = pair_axis_exact(xh, xl, ax);
    p.py = pair_axis_exact(yh, yl, ay);
    return p;
}

// Unclamped floor of the hi part (used only to place the histogram window).
__device__ __forceinline__ int pair_axis_rough(float bh, const AxisPair &A)
{
    float u = (bh - A.x0h) * A.sh;
    u = fminf(fmaxf(u, -1.0e9f), 1.0e9f);
    return (int)floorf(u);
}

// ------------------------------------------------ privatised histogram epilogue
// A CTA's rays come from one compact tile of the lens plane, so almost all of
// them land in a small patch of the source map.  The CTA counts that patch in
// a W x W shared-memory window (placed around the pixel of one of its rays, inside the
// map) and adds the window to the global map at the end; rays outside the window go
// straight to global atomics.  W is 64, or 32 for the direct sum's half tiles and the
// learned tiles.  One atomic per ray: the shared-memory increment merges a warp's equal pixels in hardware, which
// cost less than finding runs of equal pixels with a shuffle, a vote and a branch per ray.
constexpr int kWin = 64;

template <int W = kWin>
struct WinHist {
    uint32_t *h;         // W*W counters in shared memory
    int wx0, wy0;        // window origin in pixels, within the map
    unsigned nwx, nwy;   // window extent: W, or the map's where that is smaller
};

// Origin of the window on one axis, for a window centred on pixel p.
template <int W = kWin>
__device__ __forceinline__ int win_origin(int p, int n)
{
    return min(max(p - W / 2, 0), max(n - W, 0));
}

template <int W = kWin>
__device__ __forceinline__ WinHist<W> make_window(uint32_t *h, int wx0, int wy0, const BinGrid &g)
{
    return {h, wx0, wy0, (unsigned)min(W, g.nx), (unsigned)min(W, g.ny)};
}

// One float-pair beta into the histogram; counts it in `out` (finite, outside the map)
// or `nan` otherwise.
template <bool NORM, int WN>
__device__ __forceinline__ void bin_pair(float xh, float yh, float xl, float yl, const BinGrid &g,
                                         const WinHist<WN> &W, uint32_t *counts, unsigned &out, unsigned &nan)
{
    int px, py;
    if (!fast_pixel<NORM>(xh, yh, xl, yl, g.fast, px, py)) {
        const BinPix p = exact_pixel(xh, yh, xl, yl, g.ax, g.ay);
        if (!p.finite) {
            ++nan;
            return;
        }
        px = p.px;
        py = p.py;
    }
    const unsigned wx = (unsigned)(px - W.wx0), wy = (unsigned)(py - W.wy0);
    if (wx < W.nwx && wy < W.nwy)
        atomicAdd(&W.h[wy * WN + wx], 1u);
    else if ((unsigned)px < (unsigned)g.nx && (unsigned)py < (unsigned)g.ny)
        atomicAdd(&counts[py * g.nx + px], 1u);
    else
        ++out;
}

// Clear the window (uint4 stores; the window is 16-byte aligned).
template <int W = kWin>
__device__ __forceinline__ void hist_zero(uint32_t *h)
{
    uint4 *h4 = reinterpret_cast<uint4 *>(h);
    for (int b = threadIdx.x; b < W * W / 4; b += blockDim.x) h4[b] = make_uint4(0u, 0u, 0u, 0u);
}

// Add the window to the global map (bins outside the map are never filled).
// CLEAR: and leave it cleared for the next tile.
template <bool CLEAR = false, int WN>
__device__ __forceinline__ void hist_flush(const WinHist<WN> &W, const BinGrid &g, uint32_t *counts)
{
    uint4 *h4 = reinterpret_cast<uint4 *>(W.h);
    for (int b = threadIdx.x; b < WN * WN / 4; b += blockDim.x) {
        const uint4 v = h4[b];
        if ((v.x | v.y | v.z | v.w) == 0u) continue;
        if (CLEAR) h4[b] = make_uint4(0u, 0u, 0u, 0u);
        const int64_t base = (int64_t)(W.wy0 + b / (WN / 4)) * g.nx + (W.wx0 + 4 * (b % (WN / 4)));
        if (v.x) atomicAdd(&counts[base + 0], v.x);
        if (v.y) atomicAdd(&counts[base + 1], v.y);
        if (v.z) atomicAdd(&counts[base + 2], v.z);
        if (v.w) atomicAdd(&counts[base + 3], v.w);
    }
}

// Block-wide sum of three per-thread counters into global 64-bit stats.
__device__ __forceinline__ void stats_add_block(unsigned binned, unsigned out, unsigned nan, unsigned *sred,
                                                unsigned long long *stats)
{
    binned = __reduce_add_sync(0xffffffffu, binned);
    out = __reduce_add_sync(0xffffffffu, out);
    nan = __reduce_add_sync(0xffffffffu, nan);
    if ((threadIdx.x & 31u) == 0) {
        if (binned) atomicAdd(&sred[0], binned);
        if (out) atomicAdd(&sred[1], out);
        if (nan) atomicAdd(&sred[2], nan);
    }
    __syncthreads();
    if (threadIdx.x == 0 && stats) {
        if (sred[0]) atomicAdd(&stats[0], (unsigned long long)sred[0]);
        if (sred[1]) atomicAdd(&stats[1], (unsigned long long)sred[1]);
        if (sred[2]) atomicAdd(&stats[2], (unsigned long long)sred[2]);
    }
}

// The same for the counts of a persistent CTA, which may add up to 2^32 and more over its
// threads (2^21 tiles of 2048 rays): sums in 64 bits.
__device__ __forceinline__ void stats_add_cta(unsigned binned, unsigned out, unsigned nan, unsigned long long *sred,
                                              unsigned long long *stats)
{
    const unsigned v[3] = {binned, out, nan};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const unsigned lo = __reduce_add_sync(0xffffffffu, v[k] & 0xffffu), hi = __reduce_add_sync(0xffffffffu, v[k] >> 16);
        if ((threadIdx.x & 31u) == 0) atomicAdd(&sred[k], ((unsigned long long)hi << 16) + lo);
    }
    __syncthreads();
    if (threadIdx.x < 3 && stats && sred[threadIdx.x]) atomicAdd(&stats[threadIdx.x], sred[threadIdx.x]);
}

}  // namespace mlens
