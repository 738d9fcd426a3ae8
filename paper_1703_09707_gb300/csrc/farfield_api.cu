// farfield_api.cu -- host side of the learned-far-field variant: fitting
// (cell CSR, FP64 far-field expansion, network training on the GPU,
// validation, fallback flags, work list), shooting, export, save / load, and
// the network verification entry point.  Every computation runs in the kernels
// of farfield.cu; this file sizes buffers, sequences launches and schedules.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <string>
#include <vector>

#include "farfield.h"
#include "mlp.cuh"

using namespace mlens;

struct FarState {
    bool ready = false;
    mlens_grid rays{};
    CellGrid cg{};
    int pe = 8, pt = 24, use_net = 1;
    double tol = 0.0;
    int nrc = 0, next = 0;
    int *scell = nullptr, *count = nullptr, *start = nullptr, *fill = nullptr, *perm = nullptr;
    float4 *cstars = nullptr;
    double *coef64 = nullptr;
    float *coef = nullptr, *tail = nullptr, *sc = nullptr;
    float *params = nullptr, *m = nullptr, *v = nullptr, *grads = nullptr, *loss = nullptr;  // params then Z
    float *gpart = nullptr, *dzs = nullptr;  // per-CTA gradient rows and per-sample latent gradients of a step
    __nv_bfloat16 *w1zb = nullptr, *w2b = nullptr;
    unsigned char *wimg = nullptr;  // the training kernel's weight operands, as in its shared memory
    float *ec = nullptr;
    int *flags = nullptr;
    unsigned *vmax_net = nullptr, *vmax_series = nullptr;
    double *vsum = nullptr;
    int *items = nullptr;
    int64_t nitems = 0, nfallback_tiles = 0;
    std::vector<int> h_items;      // host copy of the work list
    int *sub_items = nullptr;      // row-restricted calls: fallback tiles, then learned tiles' descriptors
    TileDesc *desc = nullptr;      // the learned tiles, in the work list's order
    CellRec *cells = nullptr;      // the ray cells
    unsigned long long *counter = nullptr;
    int *d_err = nullptr;  // learned kernel: a tensor-core wait gave up
    int grid = 0;
    NetConsts net{};  // the network's shared constants, passed with each learned launch
    char *arena = nullptr;  // the one allocation behind every device pointer above but sub_items
    size_t arena_bytes = 0;
    mlens_fit_report report{};
};

namespace {

int ffail(int code, const std::string &m)
{
    set_last_error(m);
    return code;
}

int fcuda(cudaError_t e, const char *what)
{
    set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
    clear_pending_error();
    return e == cudaErrorMemoryAllocation ? MLENS_ERR_NOMEM : MLENS_ERR_CUDA;
}

#define FCUDA(call, what)                              \
    do {                                               \
        cudaError_t e_ = (call);                       \
        if (e_ != cudaSuccess) return fcuda(e_, what); \
    } while (0)

template <class T>
void ffree(T *&p)
{
    if (p) dfree((void *)p);
    p = nullptr;
}

void free_state(FarState *f)
{
    ffree(f->arena), ffree(f->sub_items);
    f->ready = false;
}

double now_s()
{
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

bool same_grid(const mlens_grid &a, const mlens_grid &b)
{
    return a.x0 == b.x0 && a.x1 == b.x1 && a.y0 == b.y0 && a.y1 == b.y1 && a.nx == b.nx && a.ny == b.ny;
}

// Cells aligned with the 64 x 32-ray tiles: cells_x cells across the ray box.
int make_layout(const mlens_grid &r, int cells_x, CellGrid &cg)
{
    if (cells_x < 1) return ffail(MLENS_ERR_ARG, "cells_x must be >= 1");
    if (r.nx % (64 * cells_x) != 0)
        return ffail(MLENS_ERR_ARG, "rays.nx must be a multiple of 64 * cells_x (cells hold whole 64-ray tiles)");
    const double dx = (r.x1 - r.x0) / r.nx, dy = (r.y1 - r.y0) / r.ny;
    cg.ktx = r.nx / (64 * cells_x);
    cg.w = 64.0 * cg.ktx * dx;
    const double ky = cg.w / (32.0 * dy);
    cg.kty = (int)std::lround(ky);
    if (cg.kty < 1 || std::fabs(ky - cg.kty) > 1e-9 * ky)
        return ffail(MLENS_ERR_ARG, "square cells need the cell width to be a whole number of 32-ray tiles in y");
    cg.ncx = cells_x;
    cg.ncy = (r.ny + 32 * cg.kty - 1) / (32 * cg.kty);
    cg.nx = cg.ncx + 2;
    cg.ny = cg.ncy + 2;
    cg.x0 = r.x0 - cg.w;
    cg.y0 = r.y0 - cg.w;
    cg.rays_nx = r.nx;
    cg.rays_ny = r.ny;
    if ((int64_t)cg.nx * cg.ny > (int64_t(1) << 26)) return ffail(MLENS_ERR_ARG, "too many cells");
    return MLENS_OK;
}

int64_t ray_tiles(const mlens_grid &r) { return (int64_t)((r.nx + 63) / 64) * ((r.ny + 31) / 32); }

// Hands out 256-byte aligned pieces of one block (base = nullptr: only adds up its size).
struct Carver {
    char *base;
    size_t at = 0;
    template <class T>
    void take(T *&p, size_t n)
    {
        p = base ? reinterpret_cast<T *>(base + at) : nullptr;
        at += (n * sizeof(T) + 255) / 256 * 256;
    }
};

// The far field's device buffers within the block c hands out; the size they take.
size_t lay_out(FarState *f, size_t stars, size_t batch, Carver c)
{
    const size_t nrc = (size_t)f->nrc, nc = (size_t)f->next, np = mlp::kParams + nrc * mlp::kLat;
    const size_t tiles = (size_t)std::max<int64_t>(ray_tiles(f->rays), 1);
    c.take(f->scell, stars), c.take(f->perm, stars), c.take(f->cstars, stars);
    c.take(f->count, nc), c.take(f->fill, nc), c.take(f->start, nc + 1);
    c.take(f->coef64, 2 * nrc * (kPtMax + 1)), c.take(f->coef, nrc * kCoefStride);
    c.take(f->tail, 2 * nrc * kPtMax), c.take(f->sc, nrc);
    c.take(f->params, np), c.take(f->m, np), c.take(f->v, np), c.take(f->grads, np), c.take(f->loss, 2);
    c.take(f->w1zb, mlp::kHid * mlp::kLat), c.take(f->w2b, mlp::kHid * mlp::kHid);
    c.take(f->wimg, (size_t)ff_weight_image_bytes());
    c.take(f->ec, nrc * mlp::kHid), c.take(f->cells, nrc);
    c.take(f->flags, nrc), c.take(f->vmax_net, nrc), c.take(f->vmax_series, nrc), c.take(f->vsum, 2);
    c.take(f->items, tiles), c.take(f->desc, tiles);
    c.take(f->counter, 1), c.take(f->d_err, 1);
    if (batch > 0) {
        c.take(f->gpart, (size_t)ff_train_blocks((int64_t)batch) * (size_t)ff_gpart_stride());
        c.take(f->dzs, batch * mlp::kLat);
    }
    return c.at;
}

// The allocation of a context's former far field, for the next one to take over; released
// if it does not.
struct Spare {
    char *p = nullptr;
    size_t bytes = 0;
    ~Spare() { ffree(p); }
};

void retire(mlens_ctx *ctx, Spare &spare)
{
    FarState *old = ctx->ff;
    if (!old) return;
    spare.p = old->arena;
    spare.bytes = old->arena_bytes;
    old->arena = nullptr;
    free_state(old);
    delete old;
    ctx->ff = nullptr;
}

// Every device buffer of a far field (batch: the largest training step, 0 = no training) in
// one allocation, the former far field's where that is large enough and not more than twice
// as large.  Thirty allocations of their own, and as many releases, were a quarter of a
// short fit: a refit without network of 20000 stars on 48 x 16 cells of 24 tiles 0.95 -> 0.72
// ms, of 2e5 stars on 128 x 43 14.1 -> 13.4 ms.
int alloc_state(FarState *f, int64_t nstars, int64_t batch, Spare &spare)
{
    const size_t stars = (size_t)std::max<int64_t>(nstars, 1);
    const size_t need = lay_out(f, stars, (size_t)batch, {nullptr});
    if (spare.p && need <= spare.bytes && spare.bytes <= 2 * need) {
        // calls queued on any stream may still read the former far field
        FCUDA(cudaDeviceSynchronize(), "sync");
        f->arena = spare.p;
        f->arena_bytes = spare.bytes;
        spare.p = nullptr;
    } else {
        ffree(spare.p);
        FCUDA(dmalloc(&f->arena, need), "cudaMalloc(far field)");
        f->arena_bytes = need;
    }
    lay_out(f, stars, (size_t)batch, {f->arena});
    return MLENS_OK;
}

// Test aid (mlens_debug_wait_probe): tensor-core waits poll an mbarrier nothing
// arrives on, so their bounded-wait failure path runs.
std::atomic<int> g_wait_probe{0};

TrainArgs train_args(FarState *f)
{
    TrainArgs t{};
    t.params = f->params;
    t.w1zb = f->w1zb;
    t.w2b = f->w2b;
    t.wimg = f->wimg;
    t.grads = f->grads;
    t.loss = f->loss;
    t.gpart = f->gpart;
    t.dzs = f->dzs;
    t.z = f->params + mlp::kParams;
    t.dz = f->grads + mlp::kParams;
    t.tail = f->tail;
    t.sc = f->sc;
    t.cg = f->cg;
    t.pe = f->pe;
    t.pt = f->pt;
    t.spec.nrc = f->nrc;
    t.backward = 1;
    t.err = f->d_err;
    t.wait_probe = g_wait_probe.load();
    return t;
}

// Validation on held-out samples: per-cell max error with and without the network.
int validate(FarState *f, int64_t per_cell, uint64_t seed, cudaStream_t s, double *mean_net, double *mean_series)
{
    FCUDA(cudaMemsetAsync(f->vmax_net, 0, sizeof(unsigned) * f->nrc, s), "memset");
    FCUDA(cudaMemsetAsync(f->vmax_series, 0, sizeof(unsigned) * f->nrc, s), "memset");
    FCUDA(cudaMemsetAsync(f->vsum, 0, sizeof(double) * 2, s), "memset");
    FCUDA(ff_prep_bf16(f->params, f->w1zb, f->w2b, f->wimg, s), "prep");
    TrainArgs t = train_args(f);
    t.backward = 0;
    t.loss = nullptr;
    t.val_max_net = f->vmax_net;
    t.val_max_series = f->vmax_series;
    t.val_sum = f->vsum;
    t.spec.seed = seed;
    t.spec.offset = 0;
    t.spec.count = per_cell * f->nrc;
    t.inv_batch = 1.0f;
    FCUDA(ff_train_step(t, t.spec.count, s), "validation");
    double h[2];
    FCUDA(cudaMemcpyAsync(h, f->vsum, sizeof(h), cudaMemcpyDeviceToHost, s), "memcpy");
    FCUDA(cudaStreamSynchronize(s), "sync");
    *mean_net = h[0] / (double)t.spec.count;
    *mean_series = h[1] / (double)t.spec.count;
    return MLENS_OK;
}

// Flags from the per-cell validation maxima, then the work list: tiles of flagged
// cells (exact direct sum, heavy) first, then the rest.
int schedule(const mlens_ctx *ctx, FarState *f, cudaStream_t s)
{
    const unsigned *src = f->use_net ? f->vmax_net : f->vmax_series;
    FCUDA(ff_flags(src, f->nrc, (float)f->tol, f->flags, s), "flags");
    std::vector<int> fl(f->nrc);
    std::vector<unsigned> vn(f->nrc), vs(f->nrc);
    FCUDA(cudaMemcpyAsync(fl.data(), f->flags, sizeof(int) * f->nrc, cudaMemcpyDeviceToHost, s), "memcpy");
    FCUDA(cudaMemcpyAsync(vn.data(), f->vmax_net, sizeof(unsigned) * f->nrc, cudaMemcpyDeviceToHost, s), "memcpy");
    FCUDA(cudaMemcpyAsync(vs.data(), f->vmax_series, sizeof(unsigned) * f->nrc, cudaMemcpyDeviceToHost, s), "memcpy");
    FCUDA(cudaStreamSynchronize(s), "sync");
    const CellGrid &cg = f->cg;
    const int ntx = (f->rays.nx + 63) / 64, nty = (f->rays.ny + 31) / 32;
    std::vector<int> heavy, light;
    for (int by = 0; by < nty; ++by)
        for (int bx = 0; bx < ntx; ++bx) {
            const int rc = (by / cg.kty) * cg.ncx + bx / cg.ktx;
            (fl[rc] ? heavy : light).push_back(by * ntx + bx);
        }
    f->nfallback_tiles = (int64_t)heavy.size();
    heavy.insert(heavy.end(), light.begin(), light.end());
    f->nitems = (int64_t)heavy.size();
    FCUDA(cudaMemcpy(f->items, heavy.data(), sizeof(int) * f->nitems, cudaMemcpyHostToDevice), "memcpy(items)");
    f->h_items = heavy;
    const int64_t nlearned = f->nitems - f->nfallback_tiles;
    FCUDA(ff_tile_desc(f->items + f->nfallback_tiles, nlearned, make_ray_grid(f->rays), ctx->lens, f->cg, f->start,
                       f->desc, s), "tile descriptors");
    int nflag = 0;
    double mx_n = 0.0, mx_s = 0.0;
    for (int i = 0; i < f->nrc; ++i) {
        nflag += fl[i];
        float a, b;
        memcpy(&a, &vn[i], 4);
        memcpy(&b, &vs[i], 4);
        mx_n = std::max(mx_n, (double)a);
        mx_s = std::max(mx_s, (double)b);
    }
    f->report.cells = f->nrc;
    f->report.cells_fallback = nflag;
    f->report.tiles = f->nitems;
    f->report.tiles_fallback = f->nfallback_tiles;
    f->report.val_max_err_net = f->use_net ? mx_n : -1.0;
    f->report.val_max_err_series = mx_s;
    FCUDA(ff_learned_grid(&f->grid), "occupancy");
    {
        std::vector<float> hp(mlp::kParams);
        FCUDA(cudaMemcpyAsync(hp.data(), f->params, sizeof(float) * mlp::kParams, cudaMemcpyDeviceToHost, s),
              "memcpy(network parameters)");
        FCUDA(cudaStreamSynchronize(s), "sync");
        ff_net_consts(hp.data(), &f->net);
    }
    return MLENS_OK;
}

int finish_inference_tables(FarState *f, cudaStream_t s)
{
    FCUDA(ff_prep_bf16(f->params, f->w1zb, f->w2b, f->wimg, s), "prep");
    FCUDA(ff_embed(f->params, f->params + mlp::kParams, f->nrc, f->ec, s), "embed");
    FCUDA(ff_cell_rec(f->coef, f->sc, f->ec, f->nrc, f->cells, s), "cell records");
    return MLENS_OK;
}

void default_params(mlens_fit_params *p)
{
    memset(p, 0, sizeof(*p));
    p->cells_x = 256;
    p->order = 10;
    p->target_order = 24;
    p->use_network = 1;
    // 48 epochs of 2^24 samples in batches of 77824 (608 CTAs of 128 samples: two full
    // waves of two CTAs per SM on 152 SMs) at 1.3x the rates the 64-epoch schedule of
    // 65536 used: over five seeds the same cells fail validation as with that
    // schedule, in two thirds of its steps
    p->train_samples = int64_t(1) << 24;
    p->epochs = 48;
    p->batch = 77824;
    p->lr_weights = 3.9e-3f;
    p->lr_latents = 6.5e-2f;
    p->val_samples_per_cell = 64;
    p->tolerance = 1e-6;
    p->seed = 1703;
}

int build_geometry(mlens_ctx *ctx, FarState *f, cudaStream_t s)
{
    FCUDA(ff_build_csr(ctx->d_stars, ctx->n_pad, f->cg, f->scell, f->count, f->start, f->fill, f->perm, f->cstars, s),
          "cell CSR");
    FCUDA(ff_coefficients(ctx->d_stars, f->scell, ctx->n_pad, f->cg, f->pt, f->coef64, s), "far-field coefficients");
    FCUDA(ff_convert(f->coef64, f->cg, f->pe, f->pt, f->coef, f->tail, f->sc, s), "coefficient conversion");
    return MLENS_OK;
}

}  // namespace

extern "C" {

void mlens_fit_params_default(mlens_fit_params *p)
{
    if (p) default_params(p);
}

int mlens_fit_far_field(mlens_ctx *ctx, const mlens_grid *rays, const mlens_fit_params *pin, mlens_fit_report *rep,
                        void *stream)
{
    if (!ctx || !rays) return ffail(MLENS_ERR_ARG, "ctx and rays must be non-NULL");
    mlens_fit_params p;
    if (pin) p = *pin;
    else default_params(&p);
    if (p.order < 0 || p.order > kPeMax) return ffail(MLENS_ERR_ARG, "order must be in [0, 16]");
    if (p.target_order <= p.order || p.target_order > kPtMax)
        return ffail(MLENS_ERR_ARG, "target_order must be in (order, 24]");
    if (p.use_network && (p.train_samples < 1 || p.epochs < 1 || p.batch < 128))
        return ffail(MLENS_ERR_ARG, "training needs train_samples >= 1, epochs >= 1, batch >= 128");
    if (p.val_samples_per_cell < 1 || !(p.tolerance >= 0.0)) return ffail(MLENS_ERR_ARG, "bad validation settings");
    if (!(rays->x1 > rays->x0 && rays->y1 > rays->y0) || rays->nx < 64 || rays->ny < 32)
        return ffail(MLENS_ERR_ARG, "bad rays grid");
    int dev = -1;
    FCUDA(cudaGetDevice(&dev), "cudaGetDevice");
    if (dev != ctx->device) return ffail(MLENS_ERR_STATE, "the context belongs to another device");
    cudaStream_t s = (cudaStream_t)stream;
    Spare spare;
    retire(ctx, spare);
    FarState *f = new FarState();
    ctx->ff = f;
    f->rays = *rays;
    f->pe = p.order;
    f->pt = p.target_order;
    f->use_net = p.use_network ? 1 : 0;
    f->tol = p.tolerance;
    int rc = make_layout(*rays, p.cells_x, f->cg);
    if (rc) return rc;
    f->nrc = f->cg.ncx * f->cg.ncy;
    f->next = f->cg.nx * f->cg.ny;
    if ((rc = alloc_state(f, ctx->n_pad, f->use_net ? std::min<int64_t>(p.batch, p.train_samples) : 0, spare)))
        return rc;

    double t0 = now_s();
    if ((rc = build_geometry(ctx, f, s))) return rc;
    FCUDA(cudaStreamSynchronize(s), "sync");
    double t1 = now_s();
    f->report.seconds_coefficients = t1 - t0;

    const int64_t np = mlp::kParams + (int64_t)f->nrc * mlp::kLat;
    FCUDA(ff_init_params(f->params, f->params + mlp::kParams, f->nrc, p.seed, s), "init");
    FCUDA(cudaMemsetAsync(f->m, 0, sizeof(float) * np, s), "memset");
    FCUDA(cudaMemsetAsync(f->d_err, 0, sizeof(int), s), "memset(err)");
    FCUDA(cudaMemsetAsync(f->v, 0, sizeof(float) * np, s), "memset");
    int64_t steps = 0;
    float last_loss = 0.0f;
    if (f->use_net) {
        const int64_t per_epoch = (p.train_samples + p.batch - 1) / p.batch;
        const int64_t total = per_epoch * p.epochs;
        TrainArgs t = train_args(f);
        t.spec.seed = p.seed * 0x9E3779B97F4A7C15ull + 17;
        FCUDA(ff_prep_bf16(f->params, f->w1zb, f->w2b, f->wimg, s), "prep");
        for (int64_t k = 0; k < total; ++k) {
            const int64_t j = k % per_epoch;
            const int64_t cnt = std::min<int64_t>(p.batch, p.train_samples - j * p.batch);
            t.spec.offset = j * p.batch;
            t.spec.count = cnt;
            t.inv_batch = 1.0f / (float)cnt;
            FCUDA(ff_train_step(t, cnt, s, true), "train step");
            // gradients summed in a fixed order (training is bit-reproducible), then
            // Adam with a cosine decay to 5% of the initial rates; the update also
            // refreshes the BF16 weight copies of the next step
            const double fr = (double)k / (double)std::max<int64_t>(total - 1, 1);
            const double sc = 0.05 + 0.95 * 0.5 * (1.0 + std::cos(3.14159265358979323846 * fr));
            const double st = (double)(k + 1);
            StepUpdate u{};
            u.p = f->params;
            u.m = f->m;
            u.v = f->v;
            u.gpart = f->gpart;
            u.nblk = ff_train_blocks(cnt);
            u.dzs = f->dzs;
            u.count = cnt;
            u.offset = t.spec.offset;
            u.nrc = f->nrc;
            u.loss = f->loss;
            u.lr_w = (float)(p.lr_weights * sc);
            u.lr_z = (float)(p.lr_latents * sc);
            u.b1 = 0.9f;
            u.b2 = 0.999f;
            u.eps = 1e-8f;
            u.bc1 = (float)(1.0 - std::pow(0.9, st));
            u.bc2 = (float)(1.0 - std::pow(0.999, st));
            u.w1zb = f->w1zb;
            u.w2b = f->w2b;
            u.wimg = f->wimg;
            FCUDA(ff_step_update(u, s), "gradient sums and Adam");
            if (k + 1 == total) FCUDA(cudaMemcpyAsync(&last_loss, f->loss, sizeof(float), cudaMemcpyDeviceToHost, s),
                                      "memcpy(loss)");
            ++steps;
        }
    }
    FCUDA(cudaStreamSynchronize(s), "sync");
    double t2 = now_s();
    f->report.seconds_train = t2 - t1;
    f->report.train_steps = steps;
    f->report.final_loss = last_loss;

    double mn = 0.0, ms = 0.0;
    if ((rc = validate(f, p.val_samples_per_cell, p.seed * 0xD1B54A32D192ED03ull + 99, s, &mn, &ms))) return rc;
    {
        int err = 0;
        FCUDA(cudaMemcpy(&err, f->d_err, sizeof(int), cudaMemcpyDeviceToHost), "memcpy(err)");
        if (err) return ffail(MLENS_ERR_CUDA, "far-field fit: a tensor-core completion wait gave up");
    }
    f->report.val_mean_err_net = f->use_net ? mn : -1.0;
    f->report.val_mean_err_series = ms;
    if ((rc = schedule(ctx, f, s))) return rc;
    if ((rc = finish_inference_tables(f, s))) return rc;
    FCUDA(cudaStreamSynchronize(s), "sync");
    f->report.seconds_validate = now_s() - t2;
    f->ready = true;
    if (rep) *rep = f->report;
    return MLENS_OK;
}

int mlens_shoot_learned(mlens_ctx *ctx, const mlens_grid *rays, const mlens_grid *src, uint32_t *counts_dev,
                        void *beta_dev, int32_t row_begin, int32_t row_end, uint32_t flags, mlens_stats *stats_host,
                        void *stream)
{
    if (!ctx || !rays || !src || !counts_dev) return ffail(MLENS_ERR_ARG, "NULL argument");
    if (!ctx->ff || !ctx->ff->ready) return ffail(MLENS_ERR_STATE, "no far field fitted on this context");
    FarState *f = ctx->ff;
    if (!same_grid(*rays, f->rays)) return ffail(MLENS_ERR_STATE, "the far field was fitted for another ray grid");
    if (!(src->x1 > src->x0 && src->y1 > src->y0) || src->nx < 1 || src->ny < 1 ||
        (int64_t)src->nx * src->ny > (int64_t(1) << 30))
        return ffail(MLENS_ERR_ARG, "bad source grid");
    if (((uintptr_t)counts_dev & 3u) || (beta_dev && ((uintptr_t)beta_dev & 15u)))
        return ffail(MLENS_ERR_ARG, "misaligned buffer");
    if (flags & ~MLENS_ACCUMULATE) return ffail(MLENS_ERR_ARG, "unknown flag bits");
    const bool all_rows = row_begin == 0 && row_end == 0;
    if (!all_rows && (row_begin < 0 || row_end > rays->ny || row_begin >= row_end || row_begin % 32 || row_end % 32))
        return ffail(MLENS_ERR_ARG, "row range must be 0 <= row_begin < row_end <= rays.ny, multiples of 32");
    int dev = -1;
    FCUDA(cudaGetDevice(&dev), "cudaGetDevice");
    if (dev != ctx->device) return ffail(MLENS_ERR_STATE, "the context belongs to another device");
    cudaStream_t s = (cudaStream_t)stream;
    const int *items = f->items;
    int64_t nitems = f->nitems, nrows_total = (int64_t)rays->nx * rays->ny;
    int64_t nheavy = f->nfallback_tiles;  // the list starts with the fallback tiles
    if (!all_rows) {
        const int ntx = (rays->nx + 63) / 64;
        std::vector<int> sub;
        nheavy = 0;
        for (size_t q = 0; q < f->h_items.size(); ++q) {
            const int t = f->h_items[q];
            const int by = t / ntx;
            if (by * 32 >= row_begin && by * 32 < row_end) {
                const bool heavy = (int64_t)q < f->nfallback_tiles;
                sub.push_back(heavy ? t : (int)((int64_t)q - f->nfallback_tiles));
                if (heavy) ++nheavy;
            }
        }
        if (!f->sub_items) FCUDA(dmalloc(&f->sub_items, sizeof(int) * std::max<int64_t>(f->nitems, 1)), "cudaMalloc");
        FCUDA(cudaMemcpyAsync(f->sub_items, sub.data(), sizeof(int) * sub.size(), cudaMemcpyHostToDevice, s),
              "memcpy(sub items)");
        FCUDA(cudaStreamSynchronize(s), "sync");
        items = f->sub_items;
        nitems = (int64_t)sub.size();
        nrows_total = (int64_t)rays->nx * (row_end - row_begin);
    }
    ClearArgs clr{};
    clr.map = counts_dev;
    clr.n = flags & MLENS_ACCUMULATE ? 0 : (size_t)src->nx * (size_t)src->ny;
    clr.words[0] = reinterpret_cast<uint32_t *>(ctx->d_stats);
    clr.nwords[0] = 6;
    clr.words[1] = reinterpret_cast<uint32_t *>(f->counter);
    clr.nwords[1] = 2;
    clr.words[2] = reinterpret_cast<uint32_t *>(f->d_err);
    clr.nwords[2] = 1;
    FCUDA(launch_clear(clr, s), "clear launch");
    LearnedArgs L{};
    L.plain.stars = ctx->d_stars;
    L.plain.nstars = ctx->n_pad;
    L.plain.n = ctx->n;
    L.plain.rays = make_ray_grid(*rays);
    L.plain.bin = make_bin_grid(*src);
    L.plain.lens = ctx->lens;
    L.plain.counts = counts_dev;
    L.plain.stats = ctx->d_stats;
    L.plain.beta_out = beta_dev;
    L.cg = f->cg;
    L.cstars = f->cstars;
    L.desc = f->desc;
    L.cells = f->cells;
    L.w2b = f->w2b;
    L.pe = f->pe;
    L.use_net = f->use_net;
    L.counter = f->counter;
    L.err = f->d_err;
    L.wait_probe = g_wait_probe.load();
    L.net = f->net;
    // Fallback tiles (each a full plain tile over all stars) run first, each split
    // over a cluster of CTAs where there are stars enough, so that a few flagged cells do not set the map's
    // time; the persistent learned kernel then takes the learned tiles.
    FCUDA(launch_shoot_split_list(L.plain, items, nheavy, fallback_star_split(ctx->n_pad), s, ctx->fma_pairs),
          "fallback tiles launch");
    L.items = all_rows ? nullptr : items + nheavy;
    L.nitems = nitems - nheavy;
    if (L.nitems > 0) FCUDA(ff_shoot_learned(L, f->grid, s), "learned shoot launch");
    if (stats_host) {
        unsigned long long h[3];
        int err = 0;
        FCUDA(cudaMemcpyAsync(h, ctx->d_stats, sizeof(h), cudaMemcpyDeviceToHost, s), "memcpy(stats)");
        FCUDA(cudaMemcpyAsync(&err, f->d_err, sizeof(int), cudaMemcpyDeviceToHost, s), "memcpy(err)");
        FCUDA(cudaStreamSynchronize(s), "sync");
        if (err) return ffail(MLENS_ERR_CUDA, "a tensor-core completion wait gave up; the map is invalid");
        stats_host->rays_total = (uint64_t)nrows_total;
        stats_host->rays_binned = h[0];
        stats_host->rays_out = h[1];
        stats_host->rays_nan = h[2];
    }
    return MLENS_OK;
}

int mlens_far_field_get_info(mlens_ctx *ctx, mlens_far_field_info *out)
{
    if (!ctx || !out) return ffail(MLENS_ERR_ARG, "NULL argument");
    if (!ctx->ff || !ctx->ff->ready) return ffail(MLENS_ERR_STATE, "no far field fitted on this context");
    const FarState *f = ctx->ff;
    out->cells_x = f->cg.ncx;
    out->cells_y = f->cg.ncy;
    out->grid_x0 = f->cg.x0;
    out->grid_y0 = f->cg.y0;
    out->cell_width = f->cg.w;
    out->grid_nx = f->cg.nx;
    out->grid_ny = f->cg.ny;
    out->order = f->pe;
    out->target_order = f->pt;
    out->use_network = f->use_net;
    out->n_params = mlp::kParams;
    out->latent_dim = mlp::kLat;
    out->report = f->report;
    return MLENS_OK;
}

int mlens_far_field_export(mlens_ctx *ctx, float *params, float *latents, int32_t *flags, double *coef,
                           int32_t *cell_start, float *val_max_net, float *val_max_series)
{
    if (!ctx) return ffail(MLENS_ERR_ARG, "NULL context");
    if (!ctx->ff || !ctx->ff->ready) return ffail(MLENS_ERR_STATE, "no far field fitted on this context");
    FarState *f = ctx->ff;
    FCUDA(cudaDeviceSynchronize(), "sync");
    if (params) FCUDA(cudaMemcpy(params, f->params, sizeof(float) * mlp::kParams, cudaMemcpyDeviceToHost), "memcpy");
    if (latents)
        FCUDA(cudaMemcpy(latents, f->params + mlp::kParams, sizeof(float) * f->nrc * mlp::kLat, cudaMemcpyDeviceToHost),
              "memcpy");
    if (flags) FCUDA(cudaMemcpy(flags, f->flags, sizeof(int) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    if (coef)
        FCUDA(cudaMemcpy(coef, f->coef64, sizeof(double) * 2 * (size_t)f->nrc * (f->pt + 1), cudaMemcpyDeviceToHost),
              "memcpy");
    if (cell_start) FCUDA(cudaMemcpy(cell_start, f->start, sizeof(int) * (f->next + 1), cudaMemcpyDeviceToHost), "memcpy");
    if (val_max_net) FCUDA(cudaMemcpy(val_max_net, f->vmax_net, sizeof(float) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    if (val_max_series)
        FCUDA(cudaMemcpy(val_max_series, f->vmax_series, sizeof(float) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    return MLENS_OK;
}

// ---------------------------------------------------------- save / load
static const char kMagic[8] = {'M', 'L', 'E', 'N', 'S', 'F', 'F', '1'};

int mlens_save_far_field(mlens_ctx *ctx, const char *path)
{
    if (!ctx || !path) return ffail(MLENS_ERR_ARG, "NULL argument");
    if (!ctx->ff || !ctx->ff->ready) return ffail(MLENS_ERR_STATE, "no far field fitted on this context");
    FarState *f = ctx->ff;
    std::vector<float> prm(mlp::kParams + (size_t)f->nrc * mlp::kLat);
    std::vector<int> fl(f->nrc);
    std::vector<unsigned> vn(f->nrc), vs(f->nrc);
    FCUDA(cudaDeviceSynchronize(), "sync");
    FCUDA(cudaMemcpy(prm.data(), f->params, sizeof(float) * prm.size(), cudaMemcpyDeviceToHost), "memcpy");
    FCUDA(cudaMemcpy(fl.data(), f->flags, sizeof(int) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    FCUDA(cudaMemcpy(vn.data(), f->vmax_net, sizeof(unsigned) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    FCUDA(cudaMemcpy(vs.data(), f->vmax_series, sizeof(unsigned) * f->nrc, cudaMemcpyDeviceToHost), "memcpy");
    FILE *fh = fopen(path, "wb");
    if (!fh) return ffail(MLENS_ERR_ARG, std::string("cannot open ") + path + " for writing");
    const int64_t n = ctx->n;
    bool ok = fwrite(kMagic, 1, 8, fh) == 8 && fwrite(&f->rays, sizeof(f->rays), 1, fh) == 1 &&
              fwrite(&f->cg, sizeof(f->cg), 1, fh) == 1 && fwrite(&f->pe, sizeof(int), 1, fh) == 1 &&
              fwrite(&f->pt, sizeof(int), 1, fh) == 1 && fwrite(&f->use_net, sizeof(int), 1, fh) == 1 &&
              fwrite(&f->tol, sizeof(double), 1, fh) == 1 && fwrite(&n, sizeof(n), 1, fh) == 1 &&
              fwrite(&f->report, sizeof(f->report), 1, fh) == 1 &&
              fwrite(prm.data(), sizeof(float), prm.size(), fh) == prm.size() &&
              fwrite(fl.data(), sizeof(int), fl.size(), fh) == fl.size() &&
              fwrite(vn.data(), sizeof(unsigned), vn.size(), fh) == vn.size() &&
              fwrite(vs.data(), sizeof(unsigned), vs.size(), fh) == vs.size();
    fclose(fh);
    if (!ok) return ffail(MLENS_ERR_ARG, std::string("short write to ") + path);
    return MLENS_OK;
}

int mlens_load_far_field(mlens_ctx *ctx, const char *path, void *stream)
{
    if (!ctx || !path) return ffail(MLENS_ERR_ARG, "NULL argument");
    FILE *fh = fopen(path, "rb");
    if (!fh) return ffail(MLENS_ERR_ARG, std::string("cannot open ") + path);
    char mg[8];
    mlens_grid rays;
    CellGrid cg;
    int pe, pt, un;
    double tol;
    int64_t n;
    mlens_fit_report rep;
    bool ok = fread(mg, 1, 8, fh) == 8 && memcmp(mg, kMagic, 8) == 0 && fread(&rays, sizeof(rays), 1, fh) == 1 &&
              fread(&cg, sizeof(cg), 1, fh) == 1 && fread(&pe, sizeof(int), 1, fh) == 1 &&
              fread(&pt, sizeof(int), 1, fh) == 1 && fread(&un, sizeof(int), 1, fh) == 1 &&
              fread(&tol, sizeof(double), 1, fh) == 1 && fread(&n, sizeof(n), 1, fh) == 1 &&
              fread(&rep, sizeof(rep), 1, fh) == 1;
    if (!ok) {
        fclose(fh);
        return ffail(MLENS_ERR_ARG, std::string(path) + " is not a far-field file");
    }
    if (n != ctx->n || pe < 0 || pe > kPeMax || pt <= pe || pt > kPtMax) {
        fclose(fh);
        return ffail(MLENS_ERR_ARG, std::string(path) + " belongs to another star field or is damaged");
    }
    const int nrc = cg.ncx * cg.ncy;
    std::vector<float> prm(mlp::kParams + (size_t)nrc * mlp::kLat);
    std::vector<int> fl(nrc);
    std::vector<unsigned> vn(nrc), vs(nrc);
    ok = fread(prm.data(), sizeof(float), prm.size(), fh) == prm.size() &&
         fread(fl.data(), sizeof(int), fl.size(), fh) == fl.size() &&
         fread(vn.data(), sizeof(unsigned), vn.size(), fh) == vn.size() &&
         fread(vs.data(), sizeof(unsigned), vs.size(), fh) == vs.size();
    fclose(fh);
    if (!ok) return ffail(MLENS_ERR_ARG, std::string("short read from ") + path);
    cudaStream_t s = (cudaStream_t)stream;
    Spare spare;
    retire(ctx, spare);
    FarState *f = new FarState();
    ctx->ff = f;
    f->rays = rays;
    f->cg = cg;
    f->pe = pe;
    f->pt = pt;
    f->use_net = un;
    f->tol = tol;
    f->nrc = nrc;
    f->next = cg.nx * cg.ny;
    f->report = rep;
    int rc;
    if ((rc = alloc_state(f, ctx->n_pad, 0, spare))) return rc;
    // the geometry (CSR, coefficients) is recomputed from the context's stars
    if ((rc = build_geometry(ctx, f, s))) return rc;
    FCUDA(cudaMemcpy(f->params, prm.data(), sizeof(float) * prm.size(), cudaMemcpyHostToDevice), "memcpy");
    FCUDA(cudaMemcpy(f->flags, fl.data(), sizeof(int) * nrc, cudaMemcpyHostToDevice), "memcpy");
    FCUDA(cudaMemcpy(f->vmax_net, vn.data(), sizeof(unsigned) * nrc, cudaMemcpyHostToDevice), "memcpy");
    FCUDA(cudaMemcpy(f->vmax_series, vs.data(), sizeof(unsigned) * nrc, cudaMemcpyHostToDevice), "memcpy");
    if ((rc = schedule(ctx, f, s))) return rc;
    if ((rc = finish_inference_tables(f, s))) return rc;
    FCUDA(cudaStreamSynchronize(s), "sync");
    f->ready = true;
    return MLENS_OK;
}

int mlens_debug_wait_probe(int32_t on)
{
    g_wait_probe.store(on ? 1 : 0);
    return MLENS_OK;
}

// ------------------------------------------- network verification entry
int mlens_ff_eval(const float *params_dev, const float *z_dev, const float *u_dev, const float *t_dev, int64_t nsamples,
                  float *y_dev, float *grads_dev, float *dz_dev, float *loss_host, void *stream)
{
    if (!params_dev || !z_dev || !u_dev || nsamples < 1) return ffail(MLENS_ERR_ARG, "bad arguments");
    if (grads_dev && !t_dev) return ffail(MLENS_ERR_ARG, "gradients need targets");
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16 *w = nullptr;
    float *dl = nullptr;
    // BF16 copies of W1z and W2, then the training kernel's operand image (16-byte aligned)
    const size_t wb = sizeof(__nv_bfloat16) * (mlp::kHid * mlp::kLat + mlp::kHid * mlp::kHid);
    FCUDA(dmalloc(&w, wb + (size_t)ff_weight_image_bytes()), "cudaMalloc");
    cudaError_t e = dmalloc(&dl, 2 * sizeof(float));  // the loss, then the kernel's error flag
    __nv_bfloat16 *w1zb = w, *w2b = w + mlp::kHid * mlp::kLat;
    unsigned char *wimg = reinterpret_cast<unsigned char *>(w) + wb;
    float *gpart = nullptr;
    const int64_t nblk = ff_train_blocks(nsamples);
    if (e == cudaSuccess && grads_dev) e = dmalloc(&gpart, sizeof(float) * nblk * ff_gpart_stride());
    if (e == cudaSuccess) e = cudaMemsetAsync(dl, 0, 2 * sizeof(float), s);
    if (e == cudaSuccess) e = ff_prep_bf16(params_dev, w1zb, w2b, wimg, s);
    if (e == cudaSuccess) {
        TrainArgs t{};
        t.params = const_cast<float *>(params_dev);
        t.w1zb = w1zb;
        t.w2b = w2b;
        t.wimg = wimg;
        t.grads = grads_dev;
        t.loss = dl;
        t.gpart = gpart;
        t.spec.count = nsamples;
        t.spec.nrc = 1;
        t.inv_batch = 1.0f / (float)nsamples;
        t.zin = z_dev;
        t.uin = u_dev;
        t.tin = t_dev;
        t.yout = y_dev;
        t.dzout = dz_dev;
        t.backward = grads_dev ? 1 : 0;
        t.err = reinterpret_cast<int *>(dl + 1);
        t.wait_probe = g_wait_probe.load();
        e = ff_train_step(t, nsamples, s);
        if (e == cudaSuccess && grads_dev) e = ff_reduce_grads(gpart, nblk, grads_dev, dl, s);
    }
    float h[2] = {0.0f, 0.0f};
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, dl, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) cudaStreamSynchronize(s);
    dfree(w);
    dfree(dl);
    dfree(gpart);
    if (e != cudaSuccess) return fcuda(e, "mlens_ff_eval");
    int flag = 0;
    memcpy(&flag, &h[1], sizeof(flag));
    if (flag) return ffail(MLENS_ERR_CUDA, "mlens_ff_eval: a tensor-core completion wait gave up");
    if (loss_host) *loss_host = h[0];
    return MLENS_OK;
}

}  // extern "C"

void mlens_free_far_field(mlens_ctx *ctx)
{
    if (ctx && ctx->ff) {
        free_state(ctx->ff);
        delete ctx->ff;
        ctx->ff = nullptr;
    }
}
