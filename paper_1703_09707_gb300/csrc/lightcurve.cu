// lightcurve.cu -- the magnification map convolved with a source's intensity
// profile, and light curves sampled from it (Section 1: given a model of the
// background source's size and intensity profile, the magnification pattern
// yields simulated light curves).  Declared in include/mlens.h.
//
//   out[j][i] = scale * sum_{(di,dj) in K} w(di,dj) counts[j+dj][i+di],
//   counts = 0 outside the map, weights normalised to sum 1 over K.
//
// Gaussian profile: separable, so two passes over the map -- rows
// (uint32 counts -> FP32) and columns (FP32 -> FP32 x scale) -- each staging a
// tile plus its halo in shared memory and taking every tap from there.
// Uniform disk: each row of the disk's support is one contiguous run of pixels,
// so with per-row inclusive prefix sums P an output is
// sum over the support's rows of P[row][i+h] - P[row][i-h-1]: O(rows) work per
// pixel, exact integer sums, then (float)(sum * (scale / |K|)) as FP64 rounds it.
// One kernel with the prefixes in shared memory where a tile fits, else prefixes in
// int64 in global memory.
// Light curve: bilinear interpolation between pixel centres along a straight
// source track, in FP64 with explicit round-to-nearest operations.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "mlens_internal.h"
#include "soft64.cuh"

namespace mlens {
namespace {

constexpr int kThr = 256;
constexpr size_t kConvSmemMost = 226 * 1024;  // above every convolution kernel's dynamic shared memory
constexpr int kColX = 64;       // column pass: tile columns
constexpr int kColY = 128;      // column pass: tile rows
constexpr int kMaxTaps = 256;   // Gaussian half-width limit (pixels)
constexpr int kMaxDiskRows = 4096;
constexpr size_t kDiskTileSmem3 = 74 * 1024;   // three CTAs per SM
constexpr size_t kDiskTileSmem1 = 220 * 1024;  // one

// Asynchronous global -> shared copy of N = 4 or 16 bytes (cp.async: no register round
// trip, so all of a thread's copies are in flight at once); ok = false writes zeros
// and reads nothing.
template <int N>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem, bool ok)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(s), "l"(gmem), "n"(N), "r"(ok ? N : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__host__ __device__ constexpr int taps_padded(int K) { return (2 * K + 1 + 3) / 4 * 4; }

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// The normalised 1-D weights, zero-padded to a multiple of four (adding exact zeros),
// passed by value with the launch: every thread of the grid takes the same weight at
// the same time, so they come from the constant bank.  From shared memory, duplicated
// for the packed arithmetic, they took as much of its bandwidth as the pixels did and
// bound both passes.
struct GaussTaps {
    float w[taps_padded(kMaxTaps)];
};

// acc[q] += sum_t w_t x[q + t] for N outputs and one step of four taps, every output's taps
// in ascending order.  Tap by tap over the outputs, so that consecutive packed
// operations share the weight operand (three distinct operand pairs cost a third
// cycle).
template <int N>
__device__ __forceinline__ void gauss_step(float2 (&acc)[N], const float2 (&x)[N + 3], const float *w)
{
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2 wt = make_float2(w[t], w[t]);
#pragma unroll
        for (int q = 0; q < N; ++q) acc[q] = ffma2(wt, x[q + t], acc[q]);
    }
}

// Row pass.  TX threads take 8 TX consecutive outputs of two adjacent rows, thread t
// outputs 8t .. 8t+7 of both, the rows packed into the lanes of f32x2 registers, with
// a sliding window of 11 inputs stepped four taps at a time: four 8-byte shared-memory
// loads per 32 packed multiply-adds.  A CTA holds kThr / TX row pairs.  The staged
// inputs are de-interleaved by index mod 8 (plane e % 8, slot e / 8) so that the lanes'
// loads of element 8t + k are consecutive.  TX follows the map's width (run_convolution):
// 1024 outputs per row pair need the least halo, narrower maps would leave threads
// without outputs.
// Where rows start on 16 bytes a thread stores its outputs itself, as two float4 a row;
// else they go through the planes, so that the lanes store consecutive pixels.
// Bound by the FP32 pipe and the staging's latency: 83 taps over 4096^2 pixels 83 -> 61
// us (the multiply-adds alone take 35 us); the whole call 182 -> 119 us.
// Five CTAs an SM and three elements in flight: against 121 us in one timing, four or six
// CTAs 126, two or five elements 134 and 130, all outputs through the planes 126 us.
template <int TX>
__global__ void __launch_bounds__(kThr, 5) k_gauss_rows(const uint32_t *__restrict__ in, int nx, int ny,
                                                        const __grid_constant__ GaussTaps W, int K,
                                                        float *__restrict__ out)
{
    extern __shared__ float2 sm2[];
    const int Kp = taps_padded(K);
    const int E = 8 * TX + Kp + 7;  // staged inputs per row
    const int P = E / 8 + 1;
    const int t = threadIdx.x % TX, g = threadIdx.x / TX;
    float2 *xs = sm2 + g * 8 * P;
    const int i0 = blockIdx.x * 8 * TX;
    constexpr int kPairs = kThr / TX;
    for (int64_t jb = 2 * kPairs * (int64_t)blockIdx.y; jb < ny; jb += 2 * kPairs * (int64_t)gridDim.y) {
        const int64_t j = jb + 2 * g;
        const bool one = j < ny, two = j + 1 < ny;
        const uint32_t *row0 = in + j * nx, *row1 = row0 + nx;
        __syncthreads();  // previous rows' taps are done
        constexpr int kB = 3;  // elements of each row in flight per thread
        for (int e0 = t; e0 < E; e0 += kB * TX) {
            uint32_t v0[kB], v1[kB];
#pragma unroll
            for (int q = 0; q < kB; ++q) {
                const int e = e0 + q * TX, i = i0 - K + e;
                const bool inside = e < E && i >= 0 && i < nx;
                v0[q] = inside && one ? row0[i] : 0u;
                v1[q] = inside && two ? row1[i] : 0u;
            }
#pragma unroll
            for (int q = 0; q < kB; ++q) {
                const int e = e0 + q * TX;
                if (e < E) xs[(e & 7) * P + (e >> 3)] = make_float2((float)v0[q], (float)v1[q]);
            }
        }
        __syncthreads();
        const int o = i0 + 8 * t;  // this thread's first output
        float2 acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = make_float2(0.f, 0.f);
        if (o < nx && one) {
            const float2 *b = xs + t;  // element 8t + n: plane n % 8, slot t + n / 8
            float2 x[11];
#pragma unroll
            for (int q = 0; q < 7; ++q) x[q] = b[q * P];
            auto step = [&](int m, int half) {  // taps m .. m + 3, m = 4 half mod 8
#pragma unroll
                for (int q = 7; q < 11; ++q) {
                    const int n = q + 4 * half;  // plane and slot of element m + q, relative to m's eight
                    x[q] = b[(n & 7) * P + (m >> 3) + (n >> 3)];
                }
                gauss_step<8>(acc, x, W.w + m);
#pragma unroll
                for (int q = 0; q < 7; ++q) x[q] = x[q + 4];
            };
            int m = 0;
#pragma unroll 2
            for (; m + 8 <= Kp; m += 8) {
                step(m, 0);
                step(m + 4, 1);
            }
            if (m < Kp) step(m, 0);
        }
        if (nx % 4 == 0) {  // of a thread's two groups of four outputs the first is in the row, the second may not be
            if (o < nx && one) {
                float4 *d = reinterpret_cast<float4 *>(out + j * nx + o);
                const bool both = o + 4 < nx;
                d[0] = make_float4(acc[0].x, acc[1].x, acc[2].x, acc[3].x);
                if (both) d[1] = make_float4(acc[4].x, acc[5].x, acc[6].x, acc[7].x);
                if (two) {
                    d += nx / 4;
                    d[0] = make_float4(acc[0].y, acc[1].y, acc[2].y, acc[3].y);
                    if (both) d[1] = make_float4(acc[4].y, acc[5].y, acc[6].y, acc[7].y);
                }
            }
            continue;
        }
        // outputs through the planes, so that the lanes store consecutive pixels (a
        // thread's own eight would touch a sector per lane and store)
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 8; ++q) xs[q * P + t] = acc[q];
        __syncthreads();
        if (one)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = q * TX + t, i = i0 + e;
                if (i < nx) {
                    const float2 v = xs[(e & 7) * P + (e >> 3)];
                    out[j * nx + i] = v.x;
                    if (two) out[(j + 1) * nx + i] = v.y;
                }
            }
    }
}

// Column pass.  A CTA stages kColY + Kp + 3 rows of 64 columns; thread (p, g)
// computes rows 16g .. 16g+15 of the adjacent columns 2p and 2p + 1 (packed into
// f32x2 lanes) in blocks of eight consecutive rows, with the same window (the lanes of a
// warp read 32 consecutive column pairs of one staged row).  As in the row pass, every
// output's taps keep their order.  VEC: rows of 16-byte-aligned chunks, staged 16 bytes at
// a time.  Bound by the FP32 pipe (74 % busy): 80 -> 57 us at the size above.
template <bool VEC>
__global__ void __launch_bounds__(kThr) k_gauss_cols(const float *__restrict__ in, int nx, int ny,
                                                     const __grid_constant__ GaussTaps W, int K, float scale,
                                                     float *__restrict__ out)
{
    extern __shared__ __align__(16) float tile[];  // (kColY + Kp + 3) rows x kColX columns
    const int Kp = taps_padded(K);
    const int tid = threadIdx.x;
    const int cp = tid % (kColX / 2), g = tid / (kColX / 2);  // column pair, group of kColY / 8 rows
    const int ib = blockIdx.x * kColX;
    const int i = ib + 2 * cp;                                // first column of this thread's pair
    const int rows = kColY + Kp + 3;
    const int tiles_y = (ny + kColY - 1) / kColY;
    for (int ty = blockIdx.y; ty < tiles_y; ty += gridDim.y) {
        const int64_t j0 = (int64_t)ty * kColY;
        __syncthreads();
        constexpr int kChunk = VEC ? 4 : 1, kPerRow = kColX / kChunk;
        const int lc = kChunk * (tid % kPerRow);
        for (int r = tid / kPerRow; r < rows; r += kThr / kPerRow) {
            const int64_t j = j0 - K + r;
            const bool ok = ib + lc < nx && j >= 0 && j < ny;
            cp_async<4 * kChunk>(tile + r * kColX + lc, ok ? in + j * nx + ib + lc : in, ok);
        }
        cp_async_wait_all();
        __syncthreads();
        if (i >= nx) continue;
        const bool two = i + 1 < nx;
        for (int r = g * (kColY / 8); r < (g + 1) * (kColY / 8); r += 8) {
            if (j0 + r >= ny) break;
            const float2 *T = reinterpret_cast<const float2 *>(tile + r * kColX + 2 * cp);
            constexpr int S = kColX / 2;  // float2 per staged row
            float2 acc[8], x[11];
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 7; ++q) x[q] = T[q * S];
#pragma unroll 4
            for (int k = 0; k < Kp; k += 4) {
#pragma unroll
                for (int q = 7; q < 11; ++q) x[q] = T[(k + q) * S];
                gauss_step<8>(acc, x, W.w + k);
#pragma unroll
                for (int q = 0; q < 7; ++q) x[q] = x[q + 4];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + r + q < ny) {
                    float *dst = out + (j0 + r + q) * nx + i;
                    dst[0] = __fmul_rn(acc[q].x, scale);
                    if (two) dst[1] = __fmul_rn(acc[q].y, scale);
                }
        }
    }
}

// Inclusive prefix sums of each row (int64): one CTA per row, 8 elements per thread
// per chunk, warp shuffles then one shared-memory step across the 8 warps.  A
// chunk's counts are read, and its sums written, through shared memory so that
// the global accesses are coalesced (a thread's own 8 elements are consecutive).
__global__ void __launch_bounds__(kThr) k_row_prefix(const uint32_t *__restrict__ in, int nx, int ny,
                                                     int64_t *__restrict__ P)
{
    constexpr int kPer = 8, kChunk = kThr * kPer;
    __shared__ int64_t wsum[kThr / 32];
    __shared__ int64_t carry_s;
    __shared__ __align__(16) uint32_t cin[kChunk];
    __shared__ __align__(16) int64_t cout[kChunk + kChunk / kPer];  // element e at e + e / 8: no bank conflicts
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int64_t j = blockIdx.x; j < ny; j += gridDim.x) {
        const uint32_t *row = in + j * nx;
        int64_t *prow = P + j * nx;
        int64_t carry = 0;
        for (int64_t base = 0; base < nx; base += kChunk) {
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int64_t i = base + k * kThr + tid;
                cin[k * kThr + tid] = i < nx ? row[i] : 0u;
            }
            __syncthreads();
            const uint4 c0 = reinterpret_cast<const uint4 *>(cin)[2 * tid];
            const uint4 c1 = reinterpret_cast<const uint4 *>(cin)[2 * tid + 1];
            const uint32_t cv[kPer] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
            int64_t v[kPer];
            int64_t run = 0;
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                run += (int64_t)cv[k];  // zero past the row's end
                v[k] = run;
            }
            int64_t x = run;  // inclusive scan of the thread totals across the warp
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int64_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            if (lane == 31) wsum[warp] = x;
            __syncthreads();
            int64_t before = 0;
            for (int q = 0; q < warp; ++q) before += wsum[q];
            const int64_t off = carry + before + (x - run);
#pragma unroll
            for (int k = 0; k < kPer; ++k) cout[tid * (kPer + 1) + k] = off + v[k];
            if (tid == kThr - 1) carry_s = off + run;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int64_t i = base + k * kThr + tid;
                const int e = k * kThr + tid;
                if (i < nx) prow[i] = cout[e + e / kPer];
            }
            carry = carry_s;
            __syncthreads();  // wsum, carry_s, cin and cout are reused by the next chunk
        }
    }
}

__global__ void __launch_bounds__(kThr) k_disk(const int64_t *__restrict__ P, int nx, int ny,
                                               const int *__restrict__ half, int H, double f,
                                               float *__restrict__ out)
{
    extern __shared__ int hs[];  // 2H+1 half-widths
    const int tid = threadIdx.x;
    for (int k = tid; k <= 2 * H; k += kThr) hs[k] = half[k];
    __syncthreads();
    const int i = blockIdx.x * kThr + tid;
    for (int64_t j = blockIdx.y; j < ny; j += gridDim.y) {
        if (i >= nx) continue;
        int64_t s = 0;
        for (int d = -H; d <= H; ++d) {
            const int64_t jj = j + d;
            if (jj < 0 || jj >= ny) continue;
            const int h = hs[d + H];
            const int64_t *pr = P + jj * nx;
            const int hi = min(i + h, nx - 1);
            const int lo = i - h - 1;
            s += pr[hi] - (lo >= 0 ? pr[lo] : 0);
        }
        out[j * nx + i] = __double2float_rn(__dmul_rn((double)s, f));
    }
}

// The same sums for disks of moderate size, in one kernel straight from the counts: a
// CTA takes TX x TY outputs, stages the counts they need (TY + 2H rows, TX + 2W + 1
// columns; zero outside the map) and turns each staged row into its prefix sums in
// place.  An output is the sum over the support's rows of two prefix values' difference;
// thread (c, g) computes column c, eight rows at a time, taking the support's rows in
// groups of equal half-width: m such rows need m + 7 run sums for the eight outputs, not 8 m.
// The row stride S is a template parameter, so that the rows' loads have immediate
// addresses; S = 4 x odd, four segments of S / 4 words: the scan's 8 rows x 4 segments
// per warp fall on 32 different banks.
// Where every staged row's total fits 13 bits (47 rays a pixel at R = 20 pixels) the prefixes are kept as 16-bit numbers, two
// neighbouring ones a word, and a thread sums two columns at once (disk_sums): half the
// loads and additions.  Elsewhere sums are exact in 32 bits, modulo 2^32 in the prefixes,
// while the largest staged count times |K|, or the part of K that the
// map's columns leave, is below 2^32 (`limit`; 3.2e6 rays in a pixel for
// 1317 pixels).  A tile with larger counts takes the sums modulo 2^32 and, staged once
// more, those of the counts' high halves, which together give the 64-bit sums: 2048^2 pixels
// with counts up to 4e6 at R = 20 104.5 us (53 with counts up to 1e5), 201 us in two passes
// per eight rows, 104.5 us with int64 prefixes; R = 62 623 -> 367 us.
// Bound by issue slots (77 %) and shared-memory loads (30 words an output at R = 20 pixels
// packed, 59 not): 4096^2 pixels in 130 us; 164 us unpacked; 373 us with int64 prefixes made
// by a kernel of their own and staged with their halo (8 bytes a load, three FP64 operations
// per output).  R = 45 1959 -> 316 us, R = 79 2788 -> 871 us.
constexpr int kMaxGroups = 256;  // runs of support rows of one half-width that a plan carries
struct DiskGroups {
    int n;
    uint16_t half[kMaxGroups], rows[kMaxGroups];
};

// The groups cut into blocks of 8, 4, 2 and 1 rows (integer sums take any order): the
// stage offset of a block's first row and its half-width; passed by value with
// the launch and read from the constant bank.
constexpr int kMaxBlocks = 384;  // plans of more take the 64-bit prefixes (none that fits a tile's shared memory has as many)
struct DiskBlocks {
    int n8, n4, n2, n1;  // ends of the blocks of each kind
    int2 at[kMaxBlocks];
};
static_assert(sizeof(DiskBlocks) <= 3584, "fits the launch's parameters");

// Columns of the support a tile of TX outputs and row stride S (words) has room for.
constexpr int disk_tile_w(int TX, int S) { return (S - TX - 1) / 2; }

// (float)((double)s * f), each operation rounded to nearest, without the FP64 pipe (two
// conversions and a product cost more there than the sum itself).  With f = fh + fl + O(2^-48)
// and s = sh + sl exact, p + t is s f to 2^-44 relative; r = fl(p + t) is the double
// product's rounding to float whenever p + t (1 +- 2^-40 |p|) round to the same float, which
// then holds of the double between them.  `fast` = |f| within 2^+-60.
__device__ __noinline__ float scale_sum_fp64(uint32_t s, double f)  // out of line: never evaluated speculatively
{
    return __double2float_rn(__dmul_rn((double)s, f));
}
__device__ __forceinline__ float scale_sum(uint32_t s, double f, float fh, float fl, bool fast)
{
    const float sh = __uint2float_rn(s);
    const float sl = (float)(int)(s - (sh >= 4294967296.0f ? 0u : (uint32_t)sh));
    const float p = __fmul_rn(sh, fh);
    const float e = __fmaf_rn(sh, fh, -p);
    const float t = __fmaf_rn(sh, fl, __fmaf_rn(sl, fh, e));
    const float z = __fmul_rn(fabsf(p), 0x1p-40f);
    const float up = __fadd_rn(p, __fadd_rn(t, z)), dn = __fadd_rn(p, __fsub_rn(t, z));
    if (s == 0u && fast) return p;  // the zero's sign is f's
    if (fast && up == dn) return up;
    return scale_sum_fp64(s, f);
}

// Sums of R output rows of one staged column (PACKED: of two adjacent ones, in the halves
// of a word) over the support's blocks.  base: the column in the first of the rows.
// PACKED words hold two neighbouring prefix values each, in two copies of a row: word k of
// the first S / 2 is (P[2k], P[2k+1]), of the others (P[2k+1], P[2k+2]), so that a pair of
// columns reads one word at any offset.  The prefixes do not decrease and are below 2^16, so
// a word's difference is both columns' runs; `room` rows of runs fit a half, then the sums
// move to lo and hi.
template <int S, int W, int R, bool PACKED>
__device__ __forceinline__ void disk_sums(const uint32_t *base, const DiskBlocks &B, int room, uint32_t (&sum)[R],
                                          uint32_t (&lo_s)[R], uint32_t (&hi_s)[R])
{
#pragma unroll
    for (int k = 0; k < R; ++k) sum[k] = lo_s[k] = hi_s[k] = 0;
    const uint32_t *hi = nullptr, *lo = nullptr;
    auto run = [&](int q) { return hi[q * S] - lo[q * S]; };  // row q of the block
    auto at = [&](int n) {
        const int2 e = B.at[n];
        const int xh = W + 1 + e.y, xl = W - e.y;
        hi = base + e.x + (PACKED ? (xh >> 1) + (xh & 1) * (S / 2) : xh);
        lo = base + e.x + (PACKED ? (xl >> 1) + (xl & 1) * (S / 2) : xl);
    };
    int left = room;
    auto make_room = [&](int m) {
        if (!PACKED) return;
        if (left < m) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                lo_s[k] += sum[k] & 0xffffu;
                hi_s[k] += sum[k] >> 16;
                sum[k] = 0;
            }
            left = room;
        }
        left -= m;
    };
    int n = 0;
    for (; n < B.n8; ++n) {
        at(n);
        make_room(8);
        uint32_t r[R + 7];
#pragma unroll
        for (int q = 0; q < R + 7; ++q) r[q] = run(q);
#pragma unroll
        for (int q = 0; q < R + 6; ++q) r[q] += r[q + 1];
#pragma unroll
        for (int q = 0; q < R + 4; ++q) r[q] += r[q + 2];
#pragma unroll
        for (int k = 0; k < R; ++k) sum[k] += r[k] + r[k + 4];
    }
    for (; n < B.n4; ++n) {
        at(n);
        make_room(4);
        uint32_t r[R + 3];
#pragma unroll
        for (int q = 0; q < R + 3; ++q) r[q] = run(q);
#pragma unroll
        for (int q = 0; q < R + 2; ++q) r[q] += r[q + 1];
#pragma unroll
        for (int k = 0; k < R; ++k) sum[k] += r[k] + r[k + 2];
    }
    for (; n < B.n2; ++n) {
        at(n);
        make_room(2);
        uint32_t r[R + 1];
#pragma unroll
        for (int q = 0; q < R + 1; ++q) r[q] = run(q);
#pragma unroll
        for (int k = 0; k < R; ++k) sum[k] += r[k] + r[k + 1];
    }
#pragma unroll 2
    for (; n < B.n1; ++n) {
        at(n);
        make_room(1);
#pragma unroll
        for (int k = 0; k < R; ++k) sum[k] += run(k);
    }
    if (PACKED) {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            lo_s[k] += sum[k] & 0xffffu;
            hi_s[k] += sum[k] >> 16;
        }
    }
}

template <int TX, int TY, int S>
__global__ void __launch_bounds__(kThr) k_disk_tile(const uint32_t *__restrict__ in, int nx, int ny,
                                                    const __grid_constant__ DiskBlocks B, int H, uint32_t limit,
                                                    double f, float fh, float fl, bool fast, float *__restrict__ out)
{
    extern __shared__ __align__(16) uint32_t T[];
    __shared__ uint32_t s_top, s_row;  // the largest staged count and row total
    constexpr int kGroup = kThr / TX, kRows = 8, kPer = TY / kGroup;  // output rows per thread, kRows at a time
    constexpr int kSeg = S / 4;
    // packed pairs of columns: the segment of a scan is held in registers
    constexpr bool kPacks = kSeg <= 51;
    constexpr int kGroup2 = 2 * kGroup, kPer2 = TY / kGroup2, kRows2 = kPer2 < 8 ? kPer2 : 8;
    static_assert(kThr % TX == 0 && kPer % kRows == 0 && kPer2 % kRows2 == 0, "whole batches");
    static_assert(S % 8 == 4, "conflict-free scan");
    constexpr int W = disk_tile_w(TX, S);  // the staged columns start at i0 - W - 1
    const int rows = TY + 2 * H;
    const int tid = threadIdx.x;
    const int i0 = blockIdx.x * TX;
    const int64_t tiles_y = ((int64_t)ny + TY - 1) / TY;
    for (int64_t by = blockIdx.y; by < tiles_y; by += gridDim.y) {
        const int64_t j0 = by * TY;
        // stage the counts
        auto stage = [&]() {
            __syncthreads();  // the previous reads are done
            for (int r = tid / 32; r < rows; r += kThr / 32) {  // a warp per row, its lanes along it
                const int64_t jj = j0 - H + r;
                const bool in_y = jj >= 0 && jj < ny;
                const uint32_t *row = in + jj * nx;
                for (int q = tid % 32; q < S; q += 32) {
                    const int64_t col = (int64_t)i0 - W - 1 + q;
                    const bool ok = in_y && col >= 0 && col < nx;
                    cp_async<4>(&T[r * S + q], ok ? row + col : in, ok);
                }
            }
            cp_async_wait_all();
            __syncthreads();
        };
        // rows to prefix sums of (count >> shift) & mask, four lanes per row; the largest
        // count seen to s_top
        auto scan = [&](int shift, uint32_t mask) {
            uint32_t top = 0;
            for (int base = 0; base < rows; base += kThr / 4) {
                const int r = base + tid / 4;
                uint32_t *p = T + r * S + (tid & 3) * kSeg;
                uint32_t sum = 0;
                if (r < rows) {
#pragma unroll 8
                    for (int k = 0; k < kSeg; ++k) {
                        top = max(top, p[k]);
                        sum += (p[k] >> shift) & mask;
                    }
                }
                uint32_t inc = sum;  // inclusive over the row's four lanes
#pragma unroll
                for (int d = 1; d < 4; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(0xffffffffu, inc, d, 4);
                    if ((tid & 3) >= d) inc += o;
                }
                uint32_t run = inc - sum;
                if (r < rows) {
#pragma unroll 8
                    for (int k = 0; k < kSeg; ++k) {
                        run += (p[k] >> shift) & mask;
                        p[k] = run;
                    }
                }
            }
            top = __reduce_max_sync(0xffffffffu, top);
            if ((tid & 31) == 0) atomicMax(&s_top, top);
            __syncthreads();
        };
        // rows to packed prefix sums, in place: a row's four lanes (one warp) have read it
        // before they write
        auto scan_packed = [&]() {
            for (int base = 0; base < rows; base += kThr / 4) {
                const int r = base + tid / 4, seg = tid & 3;
                uint32_t *row = T + r * S;
                uint32_t v[kSeg + 1], sum = 0;
#pragma unroll
                for (int k = 0; k < kSeg; ++k) {
                    v[k] = r < rows ? row[seg * kSeg + k] : 0u;
                    sum += v[k];
                }
                uint32_t inc = sum;
#pragma unroll
                for (int d = 1; d < 4; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(0xffffffffu, inc, d, 4);
                    if (seg >= d) inc += o;
                }
                v[kSeg] = __shfl_down_sync(0xffffffffu, v[0], 1, 4);  // the next segment's first (unread behind the last)
                __syncwarp();
                if (r < rows) {
                    uint32_t run = inc - sum + v[0];  // P at the segment's first element
                    const int odd = (seg * kSeg) & 1;
                    uint32_t *even_w = row + (seg * kSeg + odd) / 2, *odd_w = row + S / 2 + (seg * kSeg - odd) / 2;
                    // element g = seg kSeg + k goes, with its successor, to word g / 2 of the even or the odd copy
#pragma unroll
                    for (int k = 0; k < kSeg; ++k) {
                        const uint32_t nxt = run + v[k + 1], w = run | nxt << 16;
                        if (((k ^ odd) & 1) == 0)
                            even_w[(k - odd + (k & 1)) / 2] = w;
                        else
                            odd_w[(k + odd - (odd ? 0 : 1)) / 2] = w;
                        run = nxt;
                    }
                }
            }
            __syncthreads();
        };
        if (tid == 0) s_top = s_row = 0u;
        stage();
        uint32_t most = 0xffffffffu;
        if (kPacks) {  // the largest row total (counts saturate at 16 bits: it is only compared with 8191)
            most = 0;
            for (int base = 0; base < rows; base += kThr / 4) {
                const int r = base + tid / 4;
                const uint32_t *p = T + r * S + (tid & 3) * kSeg;
                uint32_t sum = 0;
                if (r < rows) {
#pragma unroll 8
                    for (int k = 0; k < kSeg; ++k) sum += min(p[k], 0xffffu);
                }
                sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                most = max(most, sum);
            }
            most = __reduce_max_sync(0xffffffffu, most);
            if ((tid & 31) == 0) atomicMax(&s_row, most);
            __syncthreads();
            most = s_row;
        }
        if (kPacks && most <= 8191u) {
            // eight rows of runs fit 16 bits (with one count above 0xffff the total is above too)
            scan_packed();
            const int c = 2 * (tid % (TX / 2)), g = tid / (TX / 2), i = i0 + c;
            const int room = (int)min(65535u / max(most, 1u), 1u << 20);
            for (int b = 0; b < kPer2; b += kRows2) {
                const int rt = g * kPer2 + b;
                if (i >= nx || j0 + rt >= ny) break;
                uint32_t sum[kRows2], lo[kRows2], hi[kRows2];
                disk_sums<S, W, kRows2, true>(T + rt * S + c / 2, B, room, sum, lo, hi);
#pragma unroll
                for (int k = 0; k < kRows2; ++k)
                    if (j0 + rt + k < ny) {
                        float *dst = out + (j0 + rt + k) * nx + i;
                        dst[0] = scale_sum(lo[k], f, fh, fl, fast);
                        if (i + 1 < nx) dst[1] = scale_sum(hi[k], f, fh, fl, fast);
                    }
            }
        } else {
            const int c = tid % TX, g = tid / TX, i = i0 + c;
            scan(0, 0xffffffffu);
            const bool large = s_top > limit;
            // this thread's rows: their sums (0), or the sums modulo 2^32, kept in the output (1)
            // until those of the counts' high halves complete them (2)
            auto rows_of = [&](auto part) {
#pragma unroll 1
                for (int b = 0; b < kPer; b += kRows) {
                    const int rt = g * kPer + b;
                    uint32_t sum[kRows], lo[kRows], hi[kRows];
                    if (i < nx && j0 + rt < ny) {
                        disk_sums<S, W, kRows, false>(T + rt * S + c, B, 0, sum, lo, hi);
#pragma unroll
                        for (int k = 0; k < kRows; ++k)
                            if (j0 + rt + k < ny) {
                                float *dst = out + (j0 + rt + k) * nx + i;
                                if (part == 0) {
                                    *dst = scale_sum(sum[k], f, fh, fl, fast);
                                } else if (part == 1) {
                                    *dst = __uint_as_float(sum[k]);
                                } else {  // the low halves add less than 2^32 to high 2^16
                                    const uint64_t from = (uint64_t)sum[k] << 16;
                                    const uint64_t t = from + (__float_as_uint(*dst) - (uint32_t)from);
                                    *dst = __double2float_rn(__dmul_rn((double)(int64_t)t, f));
                                }
                            }
                    }
                }
            };
            // (a loop for each part, or for the widest strides one loop for all three: each 3 %
            // faster than the other way round)
            if constexpr (kPacks) {
                if (!large) {
                    rows_of(std::integral_constant<int, 0>{});
                } else {
                    rows_of(std::integral_constant<int, 1>{});
                    stage();
                    scan(16, 0xffffu);
                    rows_of(std::integral_constant<int, 2>{});
                }
            } else {
                for (int pass = 0; pass < (large ? 2 : 1); ++pass) {
                    if (pass > 0) {
                        stage();
                        scan(16, 0xffffu);
                    }
                    rows_of(large ? pass + 1 : 0);
                }
            }
        }
        __syncthreads();  // s_top and s_row are set again
    }
}

// Half-width of each row dj = q - H of the disk support: the largest h with
// (h dx)^2 + (dj dy)^2 <= R^2 in FP64 without contraction (the definition of the
// support), capped at nx (a longer run changes nothing: both ends clamp).
__global__ void __launch_bounds__(kThr) k_disk_halves(double R, double dx, double dy, int H, int nx,
                                                      int *__restrict__ half)
{
    const int q = blockIdx.x * kThr + threadIdx.x;
    if (q > 2 * H) return;
    const double dj = (double)(q - H);
    const double yy = __dmul_rn(__dmul_rn(dj, dy), __dmul_rn(dj, dy));
    const double rr = __dmul_rn(R, R);
    auto inside = [&](long long h) {
        const double x = __dmul_rn((double)h, dx);
        return __dadd_rn(__dmul_rn(x, x), yy) <= rr;
    };
    long long h = (long long)floor(__ddiv_rn(__dsqrt_rn(fmax(__dsub_rn(rr, yy), 0.0)), dx));
    while (h > 0 && !inside(h)) --h;
    while (h < nx && inside(h + 1)) ++h;
    half[q] = (int)min(h, (long long)nx);
}

// A constant divisor: its value and, where it lies within 2^+-200, its significand and
// reciprocal for soft_div (ok).
struct Divisor {
    double d;
    Soft64 b;
    uint64_t r;
    bool ok;
};

struct Track {
    double o[2], b0[2], b1[2];  // map origin, first and last point of the track, per axis
    Divisor w[2], last;         // pixel widths, n - 1
    int size[2];                // map size
    int n;
};

// a / D, correctly rounded.
__device__ __forceinline__ double divide(double a, const Divisor &D)
{
    const uint64_t bits = (uint64_t)__double_as_longlong(a);
    const uint32_t e = (uint32_t)(bits >> 52) & 0x7ffu;
    if (!D.ok || e - 823u > 400u) return __ddiv_rn(a, D.d);
    return __longlong_as_double((long long)soft_bits(soft_div(soft_of(bits), D.b, D.r), bits & uint64_t(1) << 63));
}

// Two lanes per point, one per axis: the even lane takes x and the lower row's
// interpolation, the odd lane y, the upper row's and the point's value.  Bound by FP64
// latency (76 cycles an instruction and warp): the divisions run on the integer pipes
// (soft64.cuh), the axes side by side, and CTAs are small so that a short curve spreads
// over the SMs.  4096 points 7.1 -> 3.7 us.
constexpr int kCurveThreads = 64;
__global__ void __launch_bounds__(kCurveThreads) k_curve(const float *__restrict__ m,
                                                         const __grid_constant__ Track T, float *__restrict__ out)
{
    const int64_t lin = (int64_t)blockIdx.x * kCurveThreads + threadIdx.x;
    const int ax = threadIdx.x & 1, k = (int)min(lin >> 1, (int64_t)T.n - 1);
    double t = 0.0;
    if (T.n > 1 && k > 0) {  // k / (n - 1)
        const int z = __clz(k);
        t = __longlong_as_double((long long)soft_bits(soft_div({(uint64_t)k << (32 + z), 31 - z}, T.last.b, T.last.r), 0));
    }
    const double b0 = T.b0[ax], b1 = T.b1[ax];
    const double b = __dadd_rn(b0, __dmul_rn(t, __dsub_rn(b1, b0)));
    const double u = __dsub_rn(divide(__dsub_rn(b, T.o[ax]), T.w[ax]), 0.5);
    const double fl = floor(u);
    const double f = __dsub_rn(u, fl);
    // corner indices clamped before the conversion (only the map's edges matter)
    const int n = T.size[ax], i = (int)fmin(fmax(fl, -2.0), (double)n + 1.0);
    const int ia = min(max(i, 0), n - 1), ib = min(max(i + 1, 0), n - 1);
    // the even lane needs the lower row, the odd lane the upper row and x's columns and fraction
    constexpr unsigned kAll = 0xffffffffu;
    const int ja = __shfl_xor_sync(kAll, ia, 1), oa = __shfl_xor_sync(kAll, ib, 1);
    const double of = __shfl_xor_sync(kAll, f, 1);
    const int row = ax ? ib : ja, c0 = ax ? ja : ia, c1 = ax ? oa : ib;
    const double fx = ax ? of : f, gx = __dsub_rn(1.0, fx);
    const double m0 = m[(int64_t)row * T.size[0] + c0], m1 = m[(int64_t)row * T.size[0] + c1];
    const double s = __dadd_rn(__dmul_rn(gx, m0), __dmul_rn(fx, m1));
    const double s0 = __shfl_xor_sync(kAll, s, 1);
    if (ax && lin >> 1 < T.n) {  // gy s0 + fy s1
        const double gy = __dsub_rn(1.0, f);
        out[k] = __double2float_rn(__dadd_rn(__dmul_rn(gy, s0), __dmul_rn(f, s)));
    }
}

Divisor make_divisor(double d)
{
    Divisor D{};
    D.d = d;
    uint64_t bits;
    std::memcpy(&bits, &d, sizeof(bits));
    D.ok = d > 0x1p-200 && d < 0x1p200;
    if (D.ok) {
        D.b = soft_of(bits);
        D.r = (uint64_t)((((unsigned __int128)1 << 127) - 1) / D.b.n);
    }
    return D;
}

int lc_cuda(cudaError_t e, const char *what)
{
    set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
    clear_pending_error();
    return e == cudaErrorMemoryAllocation ? MLENS_ERR_NOMEM : MLENS_ERR_CUDA;
}

int lc_fail(int code, const std::string &msg)
{
    set_last_error(msg);
    return code;
}

int check_map(const mlens_grid *g)
{
    if (!g) return lc_fail(MLENS_ERR_ARG, "source grid is NULL");
    if (!std::isfinite(g->x0) || !std::isfinite(g->x1) || !std::isfinite(g->y0) || !std::isfinite(g->y1) ||
        !(g->x1 > g->x0) || !(g->y1 > g->y0))
        return lc_fail(MLENS_ERR_ARG, "source box must be finite with x1 > x0 and y1 > y0");
    if (g->nx < 1 || g->ny < 1 || (int64_t)g->nx * g->ny > (int64_t(1) << 30))
        return lc_fail(MLENS_ERR_ARG, "source map needs nx, ny >= 1 and nx*ny <= 2^30");
    return MLENS_OK;
}

// Largest di >= 0 with (di dx)^2 + (dj dy)^2 <= R^2, or -1 if none (FP64, as the
// definition of the support).
int half_width(double R, double dx, double dy, int dj)
{
    const double yy = ((double)dj * dy) * ((double)dj * dy);
    if (yy > R * R) return -1;
    auto inside = [&](int64_t h) { return ((double)h * dx) * ((double)h * dx) + yy <= R * R; };
    int64_t h = (int64_t)std::floor(std::sqrt(R * R - yy) / dx);  // within a step or two of the answer
    while (h > 0 && !inside(h)) --h;
    while (inside(h + 1)) ++h;
    return (int)h;
}

}  // namespace
}  // namespace mlens

using namespace mlens;

namespace mlens {
namespace {

// Shape of one convolution: taps / support rows and the workspace layout.
struct ConvPlan {
    int Kx = 0, Ky = 0;    // Gaussian half-widths (pixels)
    int Hs = 0;            // disk: support rows |dj| <= Hs
    int Ws = 0;            // disk: the largest half-width, capped at nx
    int64_t count = 0;     // disk: |K|
    int64_t terms = 0;     // disk: the most pixels of the map that K covers (rows capped at nx)
    DiskGroups groups{};   // disk: runs of support rows of one half-width (capped at nx); n = 0: too many
    int blocks = 0;        // disk: the blocks of 8, 4, 2 and 1 rows they are cut into (DiskBlocks)
    size_t off_map = 0;    // workspace offset of the map-sized buffer
    size_t bytes = 0;      // workspace size
};

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

int plan_convolution(const mlens_grid *src, int32_t profile, double size, ConvPlan *pl)
{
    int rc;
    if ((rc = check_map(src))) return rc;
    if (!std::isfinite(size) || size < 0.0) return lc_fail(MLENS_ERR_ARG, "size must be finite and >= 0");
    const int nx = src->nx, ny = src->ny;
    const size_t npix = (size_t)nx * (size_t)ny;
    const double dx = (src->x1 - src->x0) / nx, dy = (src->y1 - src->y0) / ny;
    if (profile == MLENS_PROFILE_GAUSSIAN) {
        if (!(size > 0.0)) return lc_fail(MLENS_ERR_ARG, "a Gaussian profile needs size > 0");
        if (4.0 * size / dx > kMaxTaps || 4.0 * size / dy > kMaxTaps)
            return lc_fail(MLENS_ERR_ARG, "Gaussian profile wider than 4 sigma = 256 pixels");
        pl->Kx = (int)std::ceil(4.0 * size / dx);
        pl->Ky = (int)std::ceil(4.0 * size / dy);
        pl->off_map = round256((size_t)(2 * pl->Kx + 1 + 2 * pl->Ky + 1) * sizeof(float));
        pl->bytes = pl->off_map + round256(npix * sizeof(float));
        return MLENS_OK;
    }
    if (profile == MLENS_PROFILE_DISK) {
        const int H = (int)std::floor(size / dy) + 1;
        if (H > kMaxDiskRows) return lc_fail(MLENS_ERR_ARG, "disk profile taller than 4096 pixels");
        if (size / dx > 1e9) return lc_fail(MLENS_ERR_ARG, "disk profile wider than 1e9 pixels");
        int64_t count = 0;
        int Hs = 0;
        for (int dj = -H; dj <= H; ++dj) {
            const int h = half_width(size, dx, dy, dj);
            if (h >= 0) {
                count += 2 * (int64_t)h + 1;
                pl->terms += std::min<int64_t>(2 * (int64_t)h + 1, nx);
                Hs = std::max(Hs, std::abs(dj));
                pl->Ws = std::max(pl->Ws, std::min(h, nx));
            }
        }
        pl->Hs = Hs;
        pl->count = count;
        DiskGroups &G = pl->groups;
        for (int dj = -Hs; dj <= Hs; ++dj) {
            const int h = std::min(half_width(size, dx, dy, dj), nx);
            if (G.n > 0 && G.half[G.n - 1] == h) {
                ++G.rows[G.n - 1];
            } else if (G.n < kMaxGroups && h <= 0xffff) {
                G.half[G.n] = (uint16_t)h;
                G.rows[G.n++] = 1;
            } else {
                G.n = 0;
                break;
            }
        }
        for (int q = 0; q < G.n; ++q) {
            const int r = G.rows[q];
            pl->blocks += r / 8 + (r >> 2 & 1) + (r >> 1 & 1) + (r & 1);
        }
        pl->off_map = round256((size_t)(2 * Hs + 1) * sizeof(int));
        pl->bytes = pl->off_map + round256(npix * sizeof(int64_t));
        return MLENS_OK;
    }
    return lc_fail(MLENS_ERR_ARG, "unknown profile");
}

// Normalised 1-D Gaussian weights exp(-((k-K) d)^2 / (2 sigma^2)) / sum: FP64 terms
// and sum, float results, zero-padded.
GaussTaps gauss_taps(double sigma, double d, int K)
{
    GaussTaps t{};
    std::vector<double> e((size_t)(2 * K + 1));
    double sum = 0.0;
    for (int k = 0; k <= 2 * K; ++k) {
        const double off = (double)(k - K) * d;
        e[(size_t)k] = std::exp(-(off * off) / (2.0 * (sigma * sigma)));
        sum += e[(size_t)k];
    }
    for (int k = 0; k <= 2 * K; ++k) t.w[k] = (float)(e[(size_t)k] / sum);
    return t;
}

template <int TX>
cudaError_t launch_gauss_rows(const uint32_t *in, int nx, int ny, const GaussTaps &w, int K, float *out, cudaStream_t s)
{
    constexpr int kPairs = kThr / TX;
    const size_t smem = (size_t)kPairs * 8 * ((8 * TX + taps_padded(K) + 7) / 8 + 1) * sizeof(float2);
    const cudaError_t e = allow_dynamic_smem(k_gauss_rows<TX>, smem, kConvSmemMost);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((nx + 8 * TX - 1) / (8 * TX)),
                    (unsigned)std::min<int64_t>((ny + 2 * kPairs - 1) / (2 * kPairs), 65535));
    k_gauss_rows<TX><<<grid, kThr, smem, s>>>(in, nx, ny, w, K, out);
    return cudaGetLastError();
}

template <bool VEC>
cudaError_t launch_gauss_cols(const float *in, int nx, int ny, const GaussTaps &w, int K, float scale, float *out,
                              cudaStream_t s)
{
    const size_t smem = (size_t)(kColY + taps_padded(K) + 3) * kColX * sizeof(float);
    const cudaError_t e = allow_dynamic_smem(k_gauss_cols<VEC>, smem, kConvSmemMost);
    if (e != cudaSuccess) return e;
    const int64_t tiles_y = (ny + kColY - 1) / kColY;
    const dim3 grid((unsigned)((nx + kColX - 1) / kColX), (unsigned)std::min<int64_t>(tiles_y, 65535));
    k_gauss_cols<VEC><<<grid, kThr, smem, s>>>(in, nx, ny, w, K, scale, out);
    return cudaGetLastError();
}

template <int TX, int TY, int S>
cudaError_t launch_disk_tile(const uint32_t *in, int nx, int ny, const ConvPlan &pl, double f, float *out,
                             cudaStream_t s)
{
    const size_t smem = (size_t)(TY + 2 * pl.Hs) * S * sizeof(uint32_t);
    const cudaError_t e = allow_dynamic_smem(k_disk_tile<TX, TY, S>, smem, kConvSmemMost);
    if (e != cudaSuccess) return e;
    DiskBlocks B{};
    int n = 0, *end[4] = {&B.n8, &B.n4, &B.n2, &B.n1};
    for (int kind = 0; kind < 4; ++kind) {
        const int m = 8 >> kind;
        for (int g = 0, row = 0; g < pl.groups.n; row += pl.groups.rows[g++]) {
            const int h = pl.groups.half[g], all = pl.groups.rows[g];
            // 8s first, then at most one block of each smaller kind, from the group's first row on
            const int r0 = m == 8 ? 0 : all / (2 * m) * (2 * m), k = m == 8 ? all / 8 : all / m % 2;
            for (int q = 0; q < k; ++q) {
                const int r = (row + r0 + q * m) * S;
                B.at[n++] = make_int2(r, h);
            }
        }
        *end[kind] = n;
    }
    const uint32_t limit = (uint32_t)(0xffffffffull / (uint64_t)pl.terms);
    const bool fast = std::fabs(f) > 0x1p-60 && std::fabs(f) < 0x1p60;
    const float fh = (float)f, fl = (float)(f - (double)fh);
    const dim3 grid((unsigned)((nx + TX - 1) / TX), (unsigned)std::min<int64_t>(((int64_t)ny + TY - 1) / TY, 65535));
    k_disk_tile<TX, TY, S><<<grid, kThr, smem, s>>>(in, nx, ny, B, pl.Hs, limit, f, fh, fl, fast, out);
    return cudaGetLastError();
}

// The disk in one kernel: 128 x 64 outputs (the least halo) where three CTAs fit an SM
// and the tiles fill the SMs twice, else 64 x 64 where they fill them once, else 64 x 32; the
// smallest row stride with room for the support.  *done = false: no tile fits its shared memory,
// or the support is wider than the longest row (half-width 117).  Such supports of few rows
// (pixels much higher than wide) take the int64 prefixes, which there are faster than the tiles of int64
// prefixes that took them before: 4096^2 pixels, half-width 145, five rows 280 -> 194 us.
template <int TX, int TY, int S, int... More>
cudaError_t disk_tile_of(const uint32_t *in, int nx, int ny, const ConvPlan &pl, double f, float *out, cudaStream_t s,
                         size_t most, bool *done)
{
    if (pl.Ws <= disk_tile_w(TX, S)) {
        if ((size_t)(TY + 2 * pl.Hs) * S * sizeof(uint32_t) > most) return cudaSuccess;
        *done = true;
        return launch_disk_tile<TX, TY, S>(in, nx, ny, pl, f, out, s);
    }
    if constexpr (sizeof...(More) > 0) return disk_tile_of<TX, TY, More...>(in, nx, ny, pl, f, out, s, most, done);
    return cudaSuccess;
}

int run_convolution(const uint32_t *counts_dev, const mlens_grid *src, int32_t profile, double size, double scale,
                    float *out_dev, const ConvPlan &pl, char *work, cudaStream_t s)
{
    const int nx = src->nx, ny = src->ny;
    const double dx = (src->x1 - src->x0) / nx, dy = (src->y1 - src->y0) / ny;
    cudaError_t e;
    if (profile == MLENS_PROFILE_GAUSSIAN) {
        float *t = reinterpret_cast<float *>(work + pl.off_map);
        const GaussTaps wx = gauss_taps(size, dx, pl.Kx), wy = gauss_taps(size, dy, pl.Ky);
        e = nx > 512 ? launch_gauss_rows<128>(counts_dev, nx, ny, wx, pl.Kx, t, s)
                     : nx > 256 ? launch_gauss_rows<64>(counts_dev, nx, ny, wx, pl.Kx, t, s)
                                : launch_gauss_rows<32>(counts_dev, nx, ny, wx, pl.Kx, t, s);
        if (e != cudaSuccess) return lc_cuda(e, "row pass launch");
        // the workspace is 256-byte aligned: rows of whole 16-byte chunks start on one
        e = nx % 4 == 0 ? launch_gauss_cols<true>(t, nx, ny, wy, pl.Ky, (float)scale, out_dev, s)
                        : launch_gauss_cols<false>(t, nx, ny, wy, pl.Ky, (float)scale, out_dev, s);
        if (e != cudaSuccess) return lc_cuda(e, "column pass launch");
        return MLENS_OK;
    }
    int dev = 0, nsm = 1;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return lc_cuda(e, "cudaGetDevice");
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return lc_cuda(e, "cudaDeviceGetAttribute");
    const double f = scale / (double)pl.count;
    // One kernel from the counts wherever a tile fits (sums of 16-bit halves beyond 32
    // bits need the 64-bit prefixes).  On maps narrower than the disk only the columns there are
    // count: 20 x 20000 pixels under a half-width of 3000 and 41 rows 118.9 us with the
    // 64-bit prefixes -> 24.6 us.
    if (pl.groups.n > 0 && pl.blocks <= kMaxBlocks && pl.terms <= 65536) {
        bool done = false;
        if ((int64_t)((nx + 127) / 128) * ((ny + 63) / 64) >= 2 * (int64_t)nsm)
            e = disk_tile_of<128, 64, 140, 172, 204>(counts_dev, nx, ny, pl, f, out_dev, s, kDiskTileSmem3, &done);
        if (e == cudaSuccess && !done && (int64_t)((nx + 63) / 64) * ((ny + 63) / 64) >= (int64_t)nsm)
            e = disk_tile_of<64, 64, 76, 108, 140, 172, 236, 300>(counts_dev, nx, ny, pl, f, out_dev, s, kDiskTileSmem1,
                                                                  &done);
        if (e == cudaSuccess && !done)
            e = disk_tile_of<64, 32, 76, 108, 140, 172, 236, 300>(counts_dev, nx, ny, pl, f, out_dev, s, kDiskTileSmem1,
                                                                  &done);
        if (e != cudaSuccess) return lc_cuda(e, "disk launch");
        if (done) return MLENS_OK;
    }
    int *half = reinterpret_cast<int *>(work);
    int64_t *P = reinterpret_cast<int64_t *>(work + pl.off_map);
    k_disk_halves<<<(unsigned)((2 * pl.Hs + 1 + kThr - 1) / kThr), kThr, 0, s>>>(size, dx, dy, pl.Hs, nx, half);
    const unsigned gp = (unsigned)std::min<int64_t>(ny, (int64_t)nsm * 8);
    k_row_prefix<<<gp, kThr, 0, s>>>(counts_dev, nx, ny, P);
    const dim3 gd((unsigned)((nx + kThr - 1) / kThr), (unsigned)std::min<int64_t>(ny, 65535));
    k_disk<<<gd, kThr, (size_t)(2 * pl.Hs + 1) * sizeof(int), s>>>(P, nx, ny, half, pl.Hs, f, out_dev);
    if ((e = cudaGetLastError()) != cudaSuccess) return lc_cuda(e, "disk launches");
    return MLENS_OK;
}

}  // namespace
}  // namespace mlens

extern "C" {

int mlens_convolve_workspace(const mlens_grid *src, int32_t profile, double size, uint64_t *bytes_out)
{
    if (!bytes_out) return lc_fail(MLENS_ERR_ARG, "bytes_out is NULL");
    ConvPlan pl;
    int rc;
    if ((rc = plan_convolution(src, profile, size, &pl))) return rc;
    *bytes_out = pl.bytes;
    return MLENS_OK;
}

int mlens_convolve(const uint32_t *counts_dev, const mlens_grid *src, int32_t profile, double size, double scale,
                   float *out_dev, void *work_dev, uint64_t work_bytes, void *stream)
{
    ConvPlan pl;
    int rc;
    if ((rc = plan_convolution(src, profile, size, &pl))) return rc;
    if (!counts_dev || !out_dev) return lc_fail(MLENS_ERR_ARG, "counts_dev and out_dev must be non-NULL");
    if (((uintptr_t)counts_dev & 3u) || ((uintptr_t)out_dev & 3u))
        return lc_fail(MLENS_ERR_ARG, "counts_dev and out_dev must be 4-byte aligned");
    if (!std::isfinite(scale)) return lc_fail(MLENS_ERR_ARG, "scale must be finite");
    const int64_t npix = (int64_t)src->nx * src->ny;
    const uintptr_t a0 = (uintptr_t)counts_dev, a1 = a0 + 4 * (uintptr_t)npix;
    const uintptr_t b0 = (uintptr_t)out_dev, b1 = b0 + 4 * (uintptr_t)npix;
    if (a0 < b1 && b0 < a1) return lc_fail(MLENS_ERR_ARG, "out_dev must not overlap counts_dev");
    if (work_dev) {
        if (((uintptr_t)work_dev & 255u) != 0) return lc_fail(MLENS_ERR_ARG, "work_dev must be 256-byte aligned");
        if (work_bytes < pl.bytes) return lc_fail(MLENS_ERR_ARG, "work_bytes is below mlens_convolve_workspace's size");
        const uintptr_t w0 = (uintptr_t)work_dev, w1 = w0 + pl.bytes;
        if ((w0 < a1 && a0 < w1) || (w0 < b1 && b0 < w1))
            return lc_fail(MLENS_ERR_ARG, "work_dev must not overlap counts_dev or out_dev");
        return run_convolution(counts_dev, src, profile, size, scale, out_dev, pl, (char *)work_dev,
                               (cudaStream_t)stream);
    }
    cudaStream_t s = (cudaStream_t)stream;
    char *work = nullptr;
    cudaError_t e = dmalloc(&work, pl.bytes);
    if (e != cudaSuccess) return lc_cuda(e, "cudaMalloc(convolution workspace)");
    rc = run_convolution(counts_dev, src, profile, size, scale, out_dev, pl, work, s);
    e = cudaStreamSynchronize(s);
    dfree(work);
    if (rc == MLENS_OK && e != cudaSuccess) rc = lc_cuda(e, "cudaStreamSynchronize");
    return rc;
}

int mlens_light_curve(const float *map_dev, const mlens_grid *src, double bx0, double by0, double bx1, double by1,
                      int32_t npts, float *out_dev, void *stream)
{
    int rc;
    if ((rc = check_map(src))) return rc;
    if (npts < 1) return lc_fail(MLENS_ERR_ARG, "npts must be >= 1");
    if (!map_dev || !out_dev) return lc_fail(MLENS_ERR_ARG, "map_dev and out_dev must be non-NULL");
    if (((uintptr_t)map_dev & 3u) || ((uintptr_t)out_dev & 3u))
        return lc_fail(MLENS_ERR_ARG, "map_dev and out_dev must be 4-byte aligned");
    if (!std::isfinite(bx0) || !std::isfinite(by0) || !std::isfinite(bx1) || !std::isfinite(by1))
        return lc_fail(MLENS_ERR_ARG, "track end points must be finite");
    Track T{};
    T.o[0] = src->x0;
    T.o[1] = src->y0;
    T.b0[0] = bx0;
    T.b0[1] = by0;
    T.b1[0] = bx1;
    T.b1[1] = by1;
    T.w[0] = make_divisor((src->x1 - src->x0) / src->nx);
    T.w[1] = make_divisor((src->y1 - src->y0) / src->ny);
    T.last = make_divisor((double)std::max(1, npts - 1));
    T.size[0] = src->nx;
    T.size[1] = src->ny;
    T.n = npts;
    const int64_t blocks = (2 * (int64_t)npts + kCurveThreads - 1) / kCurveThreads;
    k_curve<<<(unsigned)blocks, kCurveThreads, 0, (cudaStream_t)stream>>>(map_dev, T, out_dev);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return lc_cuda(e, "light curve launch");
    return MLENS_OK;
}

int mlens_magnification_scale(const mlens_grid *rays, const mlens_grid *src, double *scale_out)
{
    if (!rays || !src || !scale_out) return lc_fail(MLENS_ERR_ARG, "rays, src and scale_out must be non-NULL");
    int rc;
    if ((rc = check_map(src))) return rc;
    if (!(rays->x1 > rays->x0) || !(rays->y1 > rays->y0) || rays->nx < 1 || rays->ny < 1 ||
        !std::isfinite(rays->x1 - rays->x0) || !std::isfinite(rays->y1 - rays->y0))
        return lc_fail(MLENS_ERR_ARG, "rays grid needs a finite box with x1 > x0, y1 > y0 and nx, ny >= 1");
    const double a_lens = (rays->x1 - rays->x0) * (rays->y1 - rays->y0);
    const double dx = (src->x1 - src->x0) / src->nx, dy = (src->y1 - src->y0) / src->ny;
    *scale_out = a_lens / ((double)rays->nx * (double)rays->ny * dx * dy);
    return MLENS_OK;
}

}  // extern "C"
