// tile.cuh -- the FP32 shooting routine (Algorithm 1 on half a 64 x 8*NP tile of the
// ray grid: prologue, star stages, beta, binning), shared by the single-field, the
// split, the persistent multi-field and the fallback-tile kernels.  See shoot_fp32.cu for the design notes.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mlens_dev.cuh"

namespace mlens {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;              // the learned kernel's CTA: a whole tile
constexpr int kTileX = 64;                 // rays per tile row
constexpr int kGroups = 4;                 // row groups of a tile, 2 NP rows each
// The direct sum's CTA takes half a tile, 32 of its columns (a warp per row group): the
// arithmetic is the tile's (its centre), while grids of few tiles fill the SMs more evenly
// and four small CTAs per SM leave fewer warps waiting at a barrier than two large ones
// (100 stars x 1000^2 rays 48.6 -> 34.8 us together with the short last chunk and the one
// clear, clear.cu; 256 fields 490 -> 472 ms; 1e4 stars x 8192^2 rays, many tiles, 132.2 ->
// 132.6 ms).
constexpr int kHalfX = 32;
constexpr int kHalfThreads = kHalfX * kGroups;
constexpr int kStage = kHalfThreads;       // stars per stage: one per thread
constexpr int kHalfWin = 32;               // binning window of a half tile
constexpr int kKahan = 32;                 // stars per compensated partial

static_assert(kStarPad % kKahan == 0, "star padding must be whole Kahan chunks");

// Shared memory of one tile: two star stages (double buffered), whose bytes then
// hold the binning window.
//
// Re-centred kernels (RowStage): the y offsets ray - star of a tile depend only on
// the ray's row and the star, so a stage holds them ready: per star the tile's 8 NP
// row offsets, then (m, m, -dx, 0) relative to the tile centre.  A thread reads its
// 2 NP rows' offsets as NP / 2 broadcast LDS.128 instead of forming them with NP
// packed additions.  An odd number of float4 per star keeps the staging threads'
// stores (one star each) free of bank conflicts.
//
// Naive kernel (StarStage): absolute coordinates, duplicated for packed arithmetic.
template <int NP, int SC>
struct RowStage {
    static constexpr int kStride = 2 * NP + 1;  // float4 per star
    float4 s[2][SC * kStride];
};

template <int SC>
struct StarStage {
    float4 q[2][SC];   // (-x, -x, -y, -y)
    float2 mm[2][SC];  // (m, m)
};

template <int NP, bool NAIVE = false>
union ShootSmem {
    std::conditional_t<NAIVE, StarStage<kStage>, RowStage<NP, kStage>> st;
    uint32_t hist[kHalfWin * kHalfWin];
};

constexpr int kMaxRows = 32;  // ray rows of the largest tile (NP = 4)

struct TileShared {
    float tc[10];      // cx, cy, ex, ey, B0h.x, B0h.y, B0l.x, B0l.y, exl, eyl
    int win[2];
    unsigned sred[3];
    __align__(16) float ro[kMaxRows], rl[kMaxRows];  // the rows' offsets from the tile centre: high, low parts
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// v - c for packed pairs, with one rounding (fma with -1 is exact in the product)
__device__ __forceinline__ float2 sub2(float2 v, float2 c) { return __ffma2_rn(c, f2(-1.0f, -1.0f), v); }

// The tile centre on one axis, chosen so that the offset of every star near the
// tile from it is exact in float32: 0 when the tile lies within 4 tile extents of
// the axis' zero (a star offset is then the star's own coordinate), else the
// middle of the tile rounded to a multiple of q, the largest power of two not
// above the ray spacing (RayGrid qx, qy).  A float star coordinate s and a centre
// c that are both multiples of ulp(s), or both of q, differ by a float whenever
// |s - c| < |s| (or |s - c| < 2^24 q), which holds for the stars within an extent
// of the tile (|s| >= 2.5 extents > |s - c|).  Farther stars round as before,
// with errors small against their distance.
__device__ __forceinline__ float tile_centre(double mid, double extent, double q, double qinv)
{
    if (fabs(mid) < 4.0 * extent) return 0.0f;
    const double c = rint(mid * qinv) * q;
    return (float)c == c ? (float)c : (float)mid;
}

// Offset of ray k of the tile from the tile centre, e + k d with the first ray's
// offset e = eh + el and the ray spacing d = dh + dl, as a float pair (hi, lo):
// TwoProduct for k dh (exact with the FMA), TwoSum with eh, the small terms
// added to the error and the pair renormalised; about 2^-44 relative.  The
// star loop adds lo after the subtraction of the star's offset, which is exact
// for the stars close to the ray (tile_centre): there the deflection m/r would
// magnify the rounding of a float32 offset.  On grids whose ray offsets are
// exact floats (a dyadic spacing and origin, RayGrid lo = 0) lo is zero and the
// loop skips the addition, which then changes nothing.
__device__ __forceinline__ void ray_offset(float k, float eh, float el, float dh, float dl, float &hi, float &lo)
{
    const float p = __fmul_rn(k, dh);
    const float pe = __fmaf_rn(k, dh, -p);
    const float s = __fadd_rn(eh, p);
    const float bb = __fsub_rn(s, eh);
    const float se = __fadd_rn(__fsub_rn(eh, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    const float t = __fadd_rn(__fadd_rn(se, pe), __fmaf_rn(k, dl, el));
    hi = __fadd_rn(s, t);
    lo = __fsub_rn(t, __fsub_rn(hi, s));
}

// Kahan step on packed pairs: S + v with compensation C (true sum ~ S - C).
__device__ __forceinline__ void kahan2(float2 &S, float2 &C, float2 v)
{
    float2 y = sub2(v, C);
    float2 t = __fadd2_rn(S, y);
    C = sub2(sub2(t, S), y);
    S = t;
}

constexpr int tile_rows(int np) { return kGroups * 2 * np; }

// Reciprocal on the FMA pipe for a packed pair: an initial guess read off the
// float bits (seed - bits(x), seed chosen by a minimax search over one binade:
// relative error <= 5.1%) refined by three Newton-Raphson steps
// y <- y + y (1 - x y), each squaring the relative error (5.1e-2 -> 2.6e-3 ->
// 6.5e-6 -> 4e-11, below float32 resolution).  x = 0 gives a non-finite result,
// as the hardware reciprocal does.  Used for a share of the interactions so that
// the FMA pipe takes part of the reciprocal load off the MUFU unit.
constexpr int kRcpSeed = 0x7EF311C2;

__device__ __forceinline__ float2 rcp_nr2(float2 x)
{
    float2 y = f2(__int_as_float(kRcpSeed - __float_as_int(x.x)), __int_as_float(kRcpSeed - __float_as_int(x.y)));
    const float2 nx = f2(-x.x, -x.y);
    const float2 one = f2(1.0f, 1.0f);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float2 e = __ffma2_rn(nx, y, one);
        y = __ffma2_rn(y, e, y);
    }
    return y;
}

// Half hx of tile row by (half hx % 2 of tile hx / 2) of the ray grid of `a`, start to finish: prologue, star
// stages, beta, binning, counters.  Every thread of the CTA must call it.
// NRP = 1: ray pair 0 takes its reciprocals from rcp_nr2 (FMA pipe) on every third
// star of a 32-star chunk (stars 2, 5, .., 29: 10 of the 128 reciprocals a thread
// forms per chunk, 7.8 %); all others come from the MUFU unit.
// NRP = 0: MUFU alone.
//
// What bounds the re-centred star loop, per star and warp (8 rays a thread) on one of
// the SM's four schedulers: MUFU, 59 cycles (8 reciprocals of 8 cycles, less the
// Newton share), against the FP32 pipe.  A packed FP32 operation holds the pipe for 2
// cycles, and 3 when its three operands are all different register pairs (measured; the
// operand ports deliver two 32-bit registers a cycle), which the accumulations
// f dx + px and f dy + py are.  Forming dx, dx^2 and dy in packed form in every thread
// put the FP32 pipe level with MUFU: 66.6 cycles a star, 138.8 ms for 1e4 stars x
// 8192^2 rays.  dx and dx^2 are the same in both lanes, so scalar operations and a copy
// replace the packed ones (135 ms); dy comes ready from the stage (RowStage): 132.2 ms,
// 63.4 cycles a star, 0.93 of the MUFU bound, and on grids whose offsets carry low parts
// 21.87 -> 18.49 ms (9999 stars x 3001 x 2999 rays), since dy's low part is added once
// per row instead of once per ray.  More warps per SM (80 or 64 registers, the Kahan
// sums in shared memory) ran slower (145 ms): spills, and the same two pipes.
//
// SPLIT > 1 (re-centred FP32 only): the CTA is rank r of a cluster of SPLIT CTAs
// that share the tile; it sums the r-th of SPLIT consecutive 32-aligned slices
// of the stars.  Ranks 1.. leave their (S, C) partials in their own stage memory
// (2 NP float4 per thread); rank 0 reads them through distributed shared memory in
// rank order, folds each in with two Kahan steps (S_r, then -C_r) and alone goes on
// to beta and binning.
// GS (re-centred FP32 only, SPLIT = 1): the split star sum through global memory.
// GS = 1: the CTA sums slice `gslice` of a.gslices consecutive 32-aligned slices of
// the stars (the same slices as a cluster split of that many CTAs) and stores its
// partials (S, C) as 2 NP float4 per thread at a.gpart, block ghalf * a.gslices +
// gslice, then returns.  GS = 2: the CTA sums no stars; it takes slice 0's partials
// as its own, folds the others in slice order (two Kahan steps each, S_r then -C_r,
// as the cluster fold does) and goes on to beta and binning.
template <int NP, bool NAIVE, int NRP = 0, int SPLIT = 1, int GS = 0>
__device__ __forceinline__ void shoot_half(const ShootArgs &a, int hx, int by, ShootSmem<NP, NAIVE> &sm,
                                           TileShared &ts, int64_t ghalf = 0, int gslice = 0)
{
    static_assert(SPLIT == 1 || !NAIVE, "the split sum is for the re-centred kernel");
    static_assert(GS == 0 || (!NAIVE && SPLIT == 1), "the global split is for the re-centred kernel");
    constexpr int kTileY = tile_rows(NP);
    static_assert(kTileY <= kMaxRows, "TileShared holds the tile's rows");
    const int tid = threadIdx.x;
    const int tx = hx % 2 * kHalfX + tid % kHalfX;  // column within the tile
    const int tg = tid / kHalfX;                    // row group: one warp
    const int i0 = hx / 2 * kTileX;
    const int j0 = by * kTileY;
    const RayGrid &R = a.rays;
    if (i0 + hx % 2 * kHalfX >= R.nx) return;  // the whole half is beyond the grid

    if (tid < 2 && !NAIVE) {
        // one axis per lane: the tile centre (tile_centre: star offsets near the tile
        // exact), offsets of the first ray and A c in FP64, split into float pairs
        const bool y = tid == 1;
        const double o = y ? R.y0 : R.x0, d = y ? R.dy : R.dx;
        const double first = (double)(y ? j0 : i0), span = (double)(y ? kTileY : kTileX);
        const double mid = o + (first + 0.5 * span) * d;
        const float c = tile_centre(mid, span * d, y ? R.qy : R.qx, y ? R.qyinv : R.qxinv);
        const double e = (o + (first + 0.5) * d) - (double)c;
        const float other = __shfl_xor_sync(0x3u, c, 1);
        const double cx = (double)(y ? other : c), cy = (double)(y ? c : other);
        const double ax = y ? a.lens.a12 : a.lens.a11, ay = y ? a.lens.a22 : a.lens.a12;
        const double bd = ax * cx + ay * cy;
        const float bh = (float)bd, eh = (float)e;
        ts.tc[tid] = c;
        ts.tc[2 + tid] = eh;
        ts.tc[4 + tid] = bh;
        ts.tc[6 + tid] = (float)(bd - (double)bh);
        ts.tc[8 + tid] = (float)(e - (double)eh);
    }
    if (tid < 3) ts.sred[tid] = 0u;
    __syncthreads();

    // ------------------------------------------------------- this thread's rays
    float rxh = 0.f, rxl = 0.f;        // the column's offset from the tile centre (NAIVE: its coordinate): high, low part
    float2 px[NP], py[NP];             // partial sums (NAIVE: the whole running sum)
    float2 Sx[NP], Sy[NP], Cx[NP], Cy[NP];
    const float kx = (float)tx;
    const bool lo = !NAIVE && R.lo;
    if (!NAIVE) {
        if (lo) {
            ray_offset(kx, ts.tc[2], ts.tc[8], R.dxh, R.dxl, rxh, rxl);
        } else {
            // exact float offsets (RayGrid lo = 0): e + k d with every step exact
            rxh = __fmaf_rn(kx, R.dxh, ts.tc[2]);
        }
        if (tid < kTileY) {  // the rows' offsets
            float h, l = 0.0f;
            if (lo) ray_offset((float)tid, ts.tc[3], ts.tc[9], R.dyh, R.dyl, h, l);
            else h = __fmaf_rn((float)tid, R.dyh, ts.tc[3]);
            ts.ro[tid] = h;
            ts.rl[tid] = l;
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) px[p] = py[p] = Sx[p] = Sy[p] = Cx[p] = Cy[p] = f2(0.f, 0.f);
        __syncthreads();
    } else {
        rxh = (float)R.x0 + ((float)(i0 + tx) + 0.5f) * (float)R.dx;
    }

    // ---------------------------------------------------------- star stages
    const float4 *stars = a.stars;
    int64_t nst = a.nstars;   // multiple of kKahan: the slices are whole chunks
    int64_t real = a.n;       // of which stars: the padding adds exactly zero and is left out
    if (SPLIT > 1) {
        const int64_t chunk = ((nst + SPLIT - 1) / SPLIT + kKahan - 1) / kKahan * kKahan;
        const int64_t s0 = min(nst, (int64_t)cg::this_cluster().block_rank() * chunk);
        stars += s0;
        nst = min(chunk, nst - s0);
        real -= s0;
    }
    if (GS == 1) {
        const int64_t chunk = ((nst + a.gslices - 1) / a.gslices + kKahan - 1) / kKahan * kKahan;
        const int64_t s0 = min(nst, (int64_t)gslice * chunk);
        stars += s0;
        nst = min(chunk, nst - s0);
        real -= s0;
    }
    if (GS == 2) nst = 0;
    nst = max(min(nst, real), (int64_t)0);
    constexpr int SC = kStage;
    const int nstage = (int)((nst + SC - 1) / SC);
    float4 nxt;
    auto stage_load = [&](int s) {
        const int64_t k = (int64_t)s * SC + tid;
        nxt = k < nst ? __ldg(&stars[k]) : make_float4(kPadCoord, kPadCoord, 0.f, 0.f);
    };
    if constexpr (NAIVE) {
        const float y0f = (float)R.y0, dyf = (float)R.dy;
        const float2 rx = f2(rxh, rxh);
        float2 ry[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float y0 = y0f + ((float)(j0 + tg * 2 * NP + 2 * p) + 0.5f) * dyf;
            const float y1 = y0f + ((float)(j0 + tg * 2 * NP + 2 * p + 1) + 0.5f) * dyf;
            ry[p] = f2(y0, y1);
            // alpha_0 first (Algorithm 1), then every star is added to it
            px[p] = f2(a.lens.fm11 * rxh + a.lens.fm12 * y0, a.lens.fm11 * rxh + a.lens.fm12 * y1);
            py[p] = f2(a.lens.fm12 * rxh + a.lens.fm22 * y0, a.lens.fm12 * rxh + a.lens.fm22 * y1);
        }
        auto stage_store = [&](int buf) {
            sm.st.q[buf][tid] = make_float4(-nxt.x, -nxt.x, -nxt.y, -nxt.y);
            sm.st.mm[buf][tid] = f2(nxt.z, nxt.z);
        };
        if (nstage > 0) {
            stage_load(0);
            stage_store(0);
        }
        __syncthreads();
        for (int s = 0; s < nstage; ++s) {
            const int buf = s & 1;
            const int cnt = (int)min((int64_t)SC, nst - (int64_t)s * SC);
            if (s + 1 < nstage) stage_load(s + 1);
            const float4 *Q = sm.st.q[buf];
            const float2 *M = sm.st.mm[buf];
#pragma unroll 1
            for (int k0 = 0; k0 < cnt; k0 += kKahan) {  // (a short last chunk is staged full, with massless stars)
#pragma unroll
                for (int k = k0; k < k0 + kKahan; ++k) {
                    const float4 q = Q[k];
                    const float2 m2 = M[k];
                    const float2 dx = __fadd2_rn(rx, f2(q.x, q.y));
                    const float2 dx2 = __fmul2_rn(dx, dx);
                    const float2 nyv = f2(q.z, q.w);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const float2 dy = __fadd2_rn(ry[p], nyv);
                        const float2 r2 = __ffma2_rn(dy, dy, dx2);
                        const float2 f = __fmul2_rn(m2, f2(rcp_approx(r2.x), rcp_approx(r2.y)));
                        px[p] = __ffma2_rn(f, dx, px[p]);
                        py[p] = __ffma2_rn(f, dy, py[p]);
                    }
                }
            }
            if (s + 1 < nstage) stage_store(buf ^ 1);
            __syncthreads();
        }
    } else {
        constexpr int kStride = RowStage<NP, SC>::kStride;
        auto stage_store = [&](int buf) {  // thread t: star t against every row of the tile
            const float ny = __fsub_rn(ts.tc[1], nxt.y);
            float4 *dst = sm.st.s[buf] + tid * kStride;
#pragma unroll
            for (int r = 0; r < kTileY / 4; ++r) {
                const float4 o = reinterpret_cast<const float4 *>(ts.ro)[r];
                float4 d = make_float4(__fadd_rn(o.x, ny), __fadd_rn(o.y, ny), __fadd_rn(o.z, ny), __fadd_rn(o.w, ny));
                if (lo) {  // after the subtraction of the star's offset (ray_offset)
                    const float4 l = reinterpret_cast<const float4 *>(ts.rl)[r];
                    d = make_float4(__fadd_rn(d.x, l.x), __fadd_rn(d.y, l.y), __fadd_rn(d.z, l.z), __fadd_rn(d.w, l.w));
                }
                dst[r] = d;
            }
            dst[kTileY / 4] = make_float4(nxt.z, nxt.z, __fsub_rn(ts.tc[0], nxt.x), 0.0f);
        };
        if (nstage > 0) {
            stage_load(0);
            stage_store(0);
        }
        __syncthreads();
        for (int s = 0; s < nstage; ++s) {
            const int buf = s & 1;
            const int cnt = (int)min((int64_t)SC, nst - (int64_t)s * SC);
            if (s + 1 < nstage) stage_load(s + 1);
            // the chunks of the stage; LO: the column's low part is added after the
            // subtraction (grids whose ray offsets are not exact floats, RayGrid lo)
            auto chunks = [&](auto lo_tag) {
                constexpr bool LO = decltype(lo_tag)::value;
                // star k of a chunk (Q: the chunk's first); NR: ray pair 0 by rcp_nr2
                auto star = [&](const float4 *Q, int k, bool NR) {
                    const float4 q = Q[k * kStride + kTileY / 4];
                    float d = __fadd_rn(rxh, q.z);
                    if (LO) d = __fadd_rn(d, rxl);
                    const float d2 = __fmul_rn(d, d);
                    const float2 dx = f2(d, d), dx2 = f2(d2, d2), m2 = f2(q.x, q.y);
                    float4 row[NP / 2];
#pragma unroll
                    for (int h = 0; h < NP / 2; ++h) row[h] = Q[k * kStride + tg * (NP / 2) + h];
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const float2 dy = p % 2 ? f2(row[p / 2].z, row[p / 2].w) : f2(row[p / 2].x, row[p / 2].y);
                        const float2 r2 = __ffma2_rn(dy, dy, dx2);
                        const float2 inv =
                            NRP > 0 && p == 0 && NR ? rcp_nr2(r2) : f2(rcp_approx(r2.x), rcp_approx(r2.y));
                        const float2 f = __fmul2_rn(m2, inv);
                        px[p] = __ffma2_rn(f, dx, px[p]);
                        py[p] = __ffma2_rn(f, dy, py[p]);
                    }
                };
                auto chunk_end = [&]() {
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        kahan2(Sx[p], Cx[p], px[p]);
                        kahan2(Sy[p], Cy[p], py[p]);
                        px[p] = py[p] = f2(0.f, 0.f);
                    }
                };
                const float4 *Q = sm.st.s[buf], *end = Q + cnt / kKahan * kKahan * kStride;
#pragma unroll 1
                for (; Q != end; Q += kKahan * kStride) {
#pragma unroll
                    for (int k = 0; k < kKahan; ++k) star(Q, k, k % 3 == 2);
                    chunk_end();
                }
                const int rest = cnt % kKahan;  // the stars' last, short chunk
                if (rest) {
                    int k = 0;
#pragma unroll 1
                    for (; k + 3 <= rest; k += 3) {
                        star(Q, k, false);
                        star(Q, k + 1, false);
                        star(Q, k + 2, true);
                    }
#pragma unroll 1
                    for (; k < rest; ++k) star(Q, k, false);
                    chunk_end();
                }
            };
            if (lo)
                chunks(std::true_type{});
            else
                chunks(std::false_type{});
            if (s + 1 < nstage) stage_store(buf ^ 1);
            __syncthreads();
        }
    }

    if constexpr (GS == 1) {
        float4 *dst = a.gpart + (ghalf * a.gslices + gslice) * (int64_t)(2 * NP * kHalfThreads);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            dst[(2 * p) * kHalfThreads + tid] = make_float4(Sx[p].x, Sx[p].y, Sy[p].x, Sy[p].y);
            dst[(2 * p + 1) * kHalfThreads + tid] = make_float4(Cx[p].x, Cx[p].y, Cy[p].x, Cy[p].y);
        }
        return;
    }
    if constexpr (GS == 2) {
        const float4 *src = a.gpart + ghalf * a.gslices * (int64_t)(2 * NP * kHalfThreads);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float4 s0 = src[(2 * p) * kHalfThreads + tid], c0 = src[(2 * p + 1) * kHalfThreads + tid];
            Sx[p] = f2(s0.x, s0.y);
            Sy[p] = f2(s0.z, s0.w);
            Cx[p] = f2(c0.x, c0.y);
            Cy[p] = f2(c0.z, c0.w);
        }
#pragma unroll 1
        for (int r = 1; r < a.gslices; ++r) {
            const float4 *rp = src + (int64_t)r * (2 * NP * kHalfThreads);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float4 sr = rp[(2 * p) * kHalfThreads + tid], cr = rp[(2 * p + 1) * kHalfThreads + tid];
                kahan2(Sx[p], Cx[p], f2(sr.x, sr.y));
                kahan2(Sy[p], Cy[p], f2(sr.z, sr.w));
                kahan2(Sx[p], Cx[p], f2(-cr.x, -cr.y));
                kahan2(Sy[p], Cy[p], f2(-cr.z, -cr.w));
            }
        }
    }

    if constexpr (SPLIT > 1) {
        static_assert(sizeof(sm) >= 2 * NP * kHalfThreads * sizeof(float4), "the partials fit the stage memory");
        cg::cluster_group cl = cg::this_cluster();
        const unsigned rank = cl.block_rank();
        float4 *part = reinterpret_cast<float4 *>(&sm);  // the stages are dead (the loop's last barrier)
        if (rank != 0) {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                part[(2 * p) * kHalfThreads + tid] = make_float4(Sx[p].x, Sx[p].y, Sy[p].x, Sy[p].y);
                part[(2 * p + 1) * kHalfThreads + tid] = make_float4(Cx[p].x, Cx[p].y, Cy[p].x, Cy[p].y);
            }
        }
        cl.sync();  // every rank's partials are in place
        if (rank == 0) {
#pragma unroll 1
            for (int r = 1; r < SPLIT; ++r) {
                const float4 *rp = cl.map_shared_rank(part, r);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const float4 sr = rp[(2 * p) * kHalfThreads + tid], cr = rp[(2 * p + 1) * kHalfThreads + tid];
                    kahan2(Sx[p], Cx[p], f2(sr.x, sr.y));
                    kahan2(Sy[p], Cy[p], f2(sr.z, sr.w));
                    kahan2(Sx[p], Cx[p], f2(-cr.x, -cr.y));
                    kahan2(Sy[p], Cy[p], f2(-cr.z, -cr.w));
                }
            }
        }
        cl.sync();  // rank 0 has read them: the other ranks may exit
        if (rank != 0) return;
    }

    // ------------------------------------------------ beta as float pairs
    float bxh[2 * NP], byh[2 * NP], bxl[2 * NP], byl[2 * NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = 2 * p + h;
            if (!NAIVE) {
                const float sx = h ? Sx[p].y : Sx[p].x, sy = h ? Sy[p].y : Sy[p].x;
                const float ccx = h ? Cx[p].y : Cx[p].x, ccy = h ? Cy[p].y : Cy[p].x;
                const float dxr = rxh, dyr = ts.ro[tg * 2 * NP + r];
                const float dxl = rxl, dyl = ts.rl[tg * 2 * NP + r];
                // A delta for this ray (small), the offsets' low parts included
                const float lx = __fmaf_rn(a.lens.fa11, dxr, __fmaf_rn(a.lens.fa12, dyr,
                                           __fmaf_rn(a.lens.fa11, dxl, __fmul_rn(a.lens.fa12, dyl))));
                const float ly = __fmaf_rn(a.lens.fa12, dxr, __fmaf_rn(a.lens.fa22, dyr,
                                           __fmaf_rn(a.lens.fa12, dxl, __fmul_rn(a.lens.fa22, dyl))));
                float th, tl;
                two_sum(ts.tc[4], -sx, th, tl);
                tl = __fadd_rn(tl, __fadd_rn(__fadd_rn(ts.tc[6], ccx), lx));
                two_sum(th, tl, bxh[r], bxl[r]);
                two_sum(ts.tc[5], -sy, th, tl);
                tl = __fadd_rn(tl, __fadd_rn(__fadd_rn(ts.tc[7], ccy), ly));
                two_sum(th, tl, byh[r], byl[r]);
            } else {
                const float thy = (float)R.y0 + ((float)(j0 + tg * 2 * NP + r) + 0.5f) * (float)R.dy;
                bxh[r] = __fsub_rn(rxh, h ? px[p].y : px[p].x);
                byh[r] = __fsub_rn(thy, h ? py[p].y : py[p].x);
                bxl[r] = 0.0f;
                byl[r] = 0.0f;
            }
        }
    }

    // ----------------------------------------------------------- binning
    pdl_wait();  // the map's and the counters' clears
    const int ix = i0 + tx;
    const bool col_ok = ix < R.nx;
    __syncthreads();  // star stages are dead: reuse the memory as the window
    hist_zero<kHalfWin>(sm.hist);
    if (tid == kHalfThreads / 2 + kHalfX / 2) {  // the half tile's middle ray
        ts.win[0] = win_origin<kHalfWin>(pair_axis_rough(bxh[0], a.bin.ax), a.bin.nx);
        ts.win[1] = win_origin<kHalfWin>(pair_axis_rough(byh[0], a.bin.ay), a.bin.ny);
    }
    __syncthreads();
    const WinHist<kHalfWin> W = make_window<kHalfWin>(sm.hist, ts.win[0], ts.win[1], a.bin);
    const int nrow = col_ok ? min(2 * NP, R.ny - (j0 + tg * 2 * NP)) : 0;  // this thread's rays in the grid
    unsigned no = 0, nn = 0;
#pragma unroll
    for (int r = 0; r < 2 * NP; ++r) {
        if (r < nrow) {
            bin_pair<true>(bxh[r], byh[r], bxl[r], byl[r], a.bin, W, a.counts, no, nn);
            if (a.beta_out) {
                float4 *bo = reinterpret_cast<float4 *>(a.beta_out);
                bo[(int64_t)(j0 + tg * 2 * NP + r) * R.nx + ix] = make_float4(bxh[r], byh[r], bxl[r], byl[r]);
            }
        }
    }
    const unsigned nb = (unsigned)max(nrow, 0) - no - nn;
    __syncthreads();
    hist_flush(W, a.bin, a.counts);
    stats_add_block(nb, no, nn, ts.sred, a.stats);
}

}  // namespace mlens
