// Host side of the C ABI declared in include/splatloam.h: the context (workspace owned and
// sized at creation), view registration (FP64 pose inversion, per-tile frame tables), and the
// stream-ordered call sequences.  No call after splat_ctx_create allocates or synchronises,
// except the ones the header marks as synchronous.

#include <cmath>
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <memory>
#include <vector>

#include "splat_internal.cuh"

using splat::PairRec;
using splat::PixFrame;
using splat::TileInfo;
using splat::ViewDesc;

namespace {
thread_local char g_cuda_err[256] = "";
}  // namespace

namespace splat {
int cuda_fail(cudaError_t e, const char *what)
{
    std::snprintf(g_cuda_err, sizeof g_cuda_err, "%s: %s", what, cudaGetErrorString(e));
    return SPLAT_ERR_CUDA;
}
}  // namespace splat

namespace {
using splat::cuda_fail;

#define CK(call)                                          \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

template <typename T>
cudaError_t dalloc(T **p, size_t count)
{
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc(reinterpret_cast<void **>(p), sizeof(T) * count);
}

bool supported_tile(int th, int tw)
{
    return (th == 16 && tw == 16) || (th == 8 && tw == 32) || (th == 32 && tw == 8) ||
           (th == 4 && tw == 64);
}

// T^c_w = inverse of the rigid sensor->world pose; t entries summed as ((a + b) + c)
void inverse_pose(const double *T, double *Rcw, double *tcw)
{
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) Rcw[3 * i + j] = T[4 * j + i];
    for (int i = 0; i < 3; ++i) {
        const double a = T[4 * 0 + i] * T[3];
        const double b = T[4 * 1 + i] * T[7];
        const double c = T[4 * 2 + i] * T[11];
        tcw[i] = -((a + b) + c);
    }
}

void split(double x, float &hi, float &lo)
{
    hi = static_cast<float>(x);
    lo = static_cast<float>(x - static_cast<double>(hi));
}

}  // namespace

constexpr int kCountersBin = 8, kCounters = kCountersBin + splat::kBinWords;
// words of splat_ctx::d_zero: queue f, pairs that touch a tile, record chunks taken, forward
// evaluations (64 bits), rows met (64 bits), then one word per tile
enum { kZeroQueue = 0, kZeroTouching, kZeroChunks, kZeroEvals = 4, kZeroRows = 6, kZeroTiles = 8 };

struct splat_ctx {
    splat_render_config cfg{};
    splat_capacity cap{};
    int device = 0;
    int sms = 0;
    int grid_fwd = 0, grid_bwd = 0;

    // registered views
    int n_views = 0;
    std::vector<ViewDesc> views;
    int64_t n_pixels = 0, n_tiles = 0;
    int bands = 0, max_view_bands = 0, max_band_tiles = 0;   // of the binning (splat::view_bands)
    ViewDesc *d_views = nullptr;
    PixFrame *d_pixframes = nullptr;   // grown by splat_set_views
    int64_t pixframe_cap = 0;
    std::unique_ptr<unsigned char[]> h_tables;   // host copy of the view tables being registered
    size_t h_tables_cap = 0;
    TileInfo *d_tileinfo = nullptr;
    uint32_t *d_tile_order = nullptr;

    // workspace
    uint64_t *d_prect = nullptr;   // pair pixel rectangles with the normal-flip bit
    // touching pairs by view and block of primitives: tile rectangles, range keys, counts
    uint2 *d_touch = nullptr;
    float *d_kappa = nullptr;
    uint32_t *d_touch_count = nullptr;
    uint32_t *d_cta_count = nullptr;
    uint64_t *d_entries = nullptr, *d_entries2 = nullptr;   // tile lists (BinArgs)
    uint8_t *d_blocks = nullptr;
    splat::ListSegment *d_segments = nullptr;
    uint2 *d_ranges = nullptr;
    float *d_tfinal = nullptr;
    int32_t *d_nlast = nullptr;
    float4 *d_wgrad = nullptr;
    float4 *d_prim = nullptr;      // per primitive: the staged axes, normal and opacity
    float *d_pose = nullptr;        // per view (dL/drho, dL/domega) of the last backward
    uint2 *d_rec = nullptr;         // contributor records: chunks of 32 (forward -> backward)
    uint32_t *d_rec_prev = nullptr, *d_rec_head = nullptr, *d_rec_fill = nullptr;
    uint32_t rec_cap = 0;           // chunks in the record pool
    float *d_img = nullptr;     // refine: depth, normal(3), alpha  (5 x max_pixels)
    float *d_gimg = nullptr;    // refine: their gradients
    uint32_t *d_counters = nullptr;   // [0] pairs M, [1] status, [3] queue b, [6] map-growth draws,
                                      // [7] sampling step, [8..] binning (splat::kBin...)
    unsigned long long *d_grow_sums = nullptr;  // map growth: block sums, Q, offset
    unsigned long long *d_bwd_evals = nullptr;
    // what a render starts from zero, in one piece (kZero... words, then the tiles' list lengths)
    uint32_t *d_zero = nullptr;

    // profiling events: [0,1] forward compositing, [2,3] backward compositing, then one event
    // after the stages of the last profiled render / refinement step: [0] before the
    // projection, [1] after it, [2] after layout and emission, [3] after the list sort, [4] after
    // the loss, [5] after the fused Adam
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    static constexpr int kStageEvents = 6;
    cudaEvent_t stage_ev[kStageEvents] = {};
    bool stage_rec[kStageEvents] = {};
    bool profiling = false;
    bool rec_fwd = false, rec_bwd = false;
    int64_t launches = 0;

    // state of the last render
    bool rendered = false;
    bool have_pose = false;         // a backward with pose terms ran since the views were set
    int samp_draws = 0;             // keyframe sampling: draws per step (0 = every view)
    uint64_t samp_seed = 0;
    uint32_t *d_samp_thr = nullptr;   // integer thresholds of the sampling law
    uint8_t *d_active = nullptr;      // per view: sampled for the current step
    bool want_pose = false;         // backward calls also accumulate the pose gradient
    int64_t last_n = 0;
    bool last_sampled = false;      // the last render drew its views
};

namespace {

bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}

int check_gaussians(const splat_ctx *ctx, const splat_gaussians *g)
{
    if (!g || g->n < 0 || g->n > ctx->cap.max_gaussians) return SPLAT_ERR_INVALID_ARG;
    if (g->n > 0 && (!g->pos_logit || !g->quat_wxyz || !g->log_scale)) return SPLAT_ERR_INVALID_ARG;
    auto aligned = [](const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; };
    if (g->n > 0 && (!aligned(g->pos_logit, 16) || !aligned(g->quat_wxyz, 16) ||
                     !aligned(g->log_scale, 8)))
        return SPLAT_ERR_INVALID_ARG;
    return SPLAT_OK;
}

splat::RenderArgs render_args(splat_ctx *ctx, const splat_gaussians *g)
{
    splat::RenderArgs a{};
    a.chain = splat::chained_size(g->n * ctx->n_views);
    a.prim = ctx->d_prim;
    a.n = g->n;
    a.tiles = ctx->d_tileinfo;
    a.pixframes = ctx->d_pixframes;
    a.ranges = ctx->d_ranges;
    a.tile_order = ctx->d_tile_order;
    a.entries = reinterpret_cast<const uint2 *>(ctx->d_entries);
    a.entry_blocks = ctx->d_blocks;
    a.rec = ctx->d_rec;
    a.rec_prev = ctx->d_rec_prev;
    a.rec_alloc = ctx->d_zero + kZeroChunks;
    a.rec_cap = ctx->rec_cap;
    a.rec_head = ctx->d_rec_head;
    a.rec_fill = ctx->d_rec_fill;
    a.status = ctx->d_counters + 1;
    a.n_tiles = ctx->n_tiles;
    a.split = ctx->d_counters + kCountersBin + splat::kBinSplit4;
    a.alpha_min = ctx->cfg.alpha_min;
    a.alpha_max = ctx->cfg.alpha_max;
    a.t_min = ctx->cfg.t_min;
    a.sigma = ctx->cfg.sigma_cut;
    a.n_pixels = ctx->n_pixels;
    a.t_final = ctx->d_tfinal;
    a.n_last = ctx->d_nlast;
    a.wgrad = ctx->d_wgrad;
    return a;
}

// forward pipeline: projection -> list layout -> emission -> list sort -> composite
// refine (nullable): what the refinement step around it starts from, set on the way
int render_core(splat_ctx *ctx, const splat_gaussians *g, float *depth, float *normal,
                float *alpha, cudaStream_t st, const splat::RefineStart *refine = nullptr)
{
    const int64_t n = g->n;
    const int th = ctx->cfg.tile_h, tw = ctx->cfg.tile_w;
    uint32_t *cnt = ctx->d_counters;
    uint32_t *zero = ctx->d_zero;
    CK(cudaMemsetAsync(zero, 0, sizeof(uint32_t) * static_cast<size_t>(kZeroTiles + ctx->n_tiles),
                       st));
    const uint8_t *active = nullptr;
    if (ctx->samp_draws > 0) {
        CK(splat::launch_sample_views(ctx->n_views, ctx->samp_draws, ctx->d_samp_thr,
                                      static_cast<uint32_t>(ctx->samp_seed),
                                      static_cast<uint32_t>(ctx->samp_seed >> 32), cnt + 7,
                                      ctx->d_active, st));
        active = ctx->d_active;
    }
    const bool prof = ctx->profiling && !capturing(st);
    auto stage_mark = [&](int k) -> cudaError_t {
        if (!prof) return cudaSuccess;
        ctx->stage_rec[k] = true;
        return cudaEventRecord(ctx->stage_ev[k], st);
    };
    if (prof)
        for (int k = 0; k < splat_ctx::kStageEvents; ++k) ctx->stage_rec[k] = false;
    CK(stage_mark(0));
    splat::ProjectArgs pa{};
    pa.pos_logit = reinterpret_cast<const float4 *>(g->pos_logit);
    pa.quat = reinterpret_cast<const float4 *>(g->quat_wxyz);
    pa.log_scale = reinterpret_cast<const float2 *>(g->log_scale);
    pa.n = n;
    pa.views = ctx->d_views;
    pa.n_views = ctx->n_views;
    pa.sigma = ctx->cfg.sigma_cut;
    pa.alpha_min = ctx->cfg.alpha_min;
    pa.tile_h = th;
    pa.tile_w = tw;
    pa.flip_normals = ctx->cfg.flip_normals;
    pa.prect = ctx->d_prect;
    pa.touch = ctx->d_touch;
    pa.kappa = ctx->d_kappa;
    pa.touch_count = ctx->d_touch_count;
    pa.prim = ctx->d_prim;
    pa.status = cnt + 1;
    pa.n_valid = zero + kZeroTouching;
    pa.n_rows = reinterpret_cast<unsigned long long *>(zero + kZeroRows);
    pa.wgrad = refine ? ctx->d_wgrad : nullptr;
    pa.active = active;
    CK(splat::launch_project(pa, st));
    CK(stage_mark(1));
    splat::BinArgs ba{};
    ba.views = ctx->d_views;
    ba.n_views = ctx->n_views;
    ba.active = active;
    ba.bands = ba.max_active_bands = ctx->bands;
    if (active)
        ba.max_active_bands =
            std::min(ctx->bands, std::min(ctx->samp_draws, ctx->n_views) * ctx->max_view_bands);
    ba.n = n;
    ba.tile_h = th;
    ba.tile_w = tw;
    ba.n_tiles = ctx->n_tiles;
    ba.tiles = ctx->d_tileinfo;
    ba.prect = ctx->d_prect;
    ba.touch = ctx->d_touch;
    ba.kappa = ctx->d_kappa;
    ba.touch_count = ctx->d_touch_count;
    ba.max_pairs = ctx->cap.max_pairs;
    ba.max_band_tiles = ctx->max_band_tiles;
    ba.tile_count = zero + kZeroTiles;
    ba.cta_count = ctx->d_cta_count;
    ba.ranges = ctx->d_ranges;
    ba.order = ctx->d_tile_order;
    ba.entries = ctx->d_entries;
    ba.entries2 = ctx->d_entries2;
    ba.entry_blocks = ctx->d_blocks;
    ba.segments = ctx->d_segments;
    ba.d_count = cnt;
    ba.status = cnt + 1;
    ba.bin = cnt + kCountersBin;
    ba.sms = ctx->sms;
    ba.warps = static_cast<uint32_t>(ctx->grid_fwd) * (splat::kBlock / 32);
    ba.rec_cap = ctx->rec_cap;
    ba.n_rows = pa.n_rows;
    if (refine) ba.refine = *refine;
    CK(splat::launch_bin_counts(ba, st));
    CK(splat::launch_emit(ba, st));
    CK(stage_mark(2));
    CK(splat::launch_lists(ba, st));
    CK(stage_mark(3));
    splat::RenderArgs a = render_args(ctx, g);
    a.depth = depth;
    a.normal = normal;
    a.alpha = alpha;
    a.queue = zero + kZeroQueue;
    a.evals = reinterpret_cast<unsigned long long *>(zero + kZeroEvals);
    if (prof) CK(cudaEventRecord(ctx->ev[0], st));
    CK(splat::launch_render_fwd(a, th, tw, ctx->grid_fwd, st));
    if (prof) {
        CK(cudaEventRecord(ctx->ev[1], st));
        ctx->rec_fwd = true;
    }
    ctx->launches += 1 + splat::bin_launches(n) + 1;   // projection, binning, compositing
    ctx->last_sampled = active != nullptr;
    ctx->rendered = true;
    ctx->last_n = n;
    return SPLAT_OK;
}

// the counters and accumulators a backward adds to
splat::RefineStart backward_start(splat_ctx *ctx)
{
    splat::RefineStart s{};
    s.queue = ctx->d_counters + 3;
    s.evals = ctx->d_bwd_evals;
    if (ctx->want_pose) {
        s.pose = ctx->d_pose;
        s.n_pose = 6 * ctx->n_views;
    }
    return s;
}

// backward into the per-primitive world-frame accumulators; started: they and the counters are
// already zero
int backward_core(splat_ctx *ctx, const splat_gaussians *g, const float *gD, const float *gN,
                  const float *gO, cudaStream_t st, bool started)
{
    uint32_t *cnt = ctx->d_counters;
    if (!started) {
        CK(splat::launch_backward_start(backward_start(ctx), ctx->d_wgrad, g->n,
                                        splat::chained_size(g->n * ctx->n_views), st));
        ctx->launches += 1;
    }
    splat::RenderArgs a = render_args(ctx, g);
    a.g_depth = gD;
    a.g_normal = gN;
    a.g_alpha = gO;
    a.queue = cnt + 3;
    a.evals = ctx->d_bwd_evals;
    a.pose_grad = ctx->want_pose ? ctx->d_pose : nullptr;
    const bool prof = ctx->profiling && !capturing(st);
    if (prof) CK(cudaEventRecord(ctx->ev[2], st));
    CK(splat::launch_render_bwd(a, ctx->cfg.tile_h, ctx->cfg.tile_w, ctx->grid_bwd, st));
    if (prof) {
        CK(cudaEventRecord(ctx->ev[3], st));
        ctx->rec_bwd = true;
    }
    ctx->launches += 1;
    ctx->have_pose = ctx->want_pose;
    return SPLAT_OK;
}

void free_ctx(splat_ctx *c)
{
    void *ptrs[] = {c->d_views, c->d_prect, c->d_touch, c->d_kappa, c->d_touch_count, c->d_zero,
                    c->d_cta_count, c->d_entries, c->d_entries2, c->d_blocks, c->d_segments,
                    c->d_ranges, c->d_tfinal, c->d_nlast, c->d_wgrad, c->d_prim,
                    c->d_pose, c->d_rec, c->d_rec_prev, c->d_rec_head, c->d_rec_fill,
                    c->d_samp_thr, c->d_active, c->d_grow_sums,
                    c->d_img, c->d_gimg, c->d_counters, c->d_bwd_evals, c->d_pixframes,
                    c->d_tileinfo, c->d_tile_order};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    for (cudaEvent_t e : c->ev)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : c->stage_ev)
        if (e) cudaEventDestroy(e);
    delete c;
}

}  // namespace

extern "C" {

SPLAT_API int splat_version(void) { return 100; }

SPLAT_API const char *splat_error_string(int code)
{
    switch (code) {
    case SPLAT_OK: return "ok";
    case SPLAT_ERR_INVALID_ARG: return "invalid argument";
    case SPLAT_ERR_CUDA: return "CUDA error";
    case SPLAT_ERR_CAPACITY: return "pair capacity exceeded";
    case SPLAT_ERR_TIMEOUT: return "device wait timed out";
    case SPLAT_ERR_NONFINITE: return "non-finite primitive parameter";
    case SPLAT_ERR_STATE: return "call order violated";
    case SPLAT_ERR_UNSUPPORTED: return "unsupported configuration";
    default: return "unknown error";
    }
}

SPLAT_API const char *splat_last_cuda_error(void) { return g_cuda_err; }

SPLAT_API void splat_default_config(splat_render_config *cfg)
{
    if (!cfg) return;
    cfg->alpha_min = 1.0f / 255.0f;
    cfg->alpha_max = 0.99f;
    cfg->t_min = 1e-4f;
    cfg->sigma_cut = 3.0f;
    cfg->tile_h = 16;
    cfg->tile_w = 16;
    cfg->work_cap = 0;
    cfg->flip_normals = 1;
}

SPLAT_API int splat_ctx_create(const splat_render_config *cfg, const splat_capacity *cap,
                               splat_ctx **out)
{
    if (!cfg || !cap || !out) return SPLAT_ERR_INVALID_ARG;
    *out = nullptr;
    if (!supported_tile(cfg->tile_h, cfg->tile_w)) return SPLAT_ERR_UNSUPPORTED;
    if (cfg->work_cap != 0) return SPLAT_ERR_UNSUPPORTED;
    if (!(cfg->alpha_min > 0.0f && cfg->alpha_min < cfg->alpha_max && cfg->alpha_max < 1.0f &&
          cfg->t_min > 0.0f && cfg->t_min < 1.0f && cfg->sigma_cut > 0.0f))
        return SPLAT_ERR_INVALID_ARG;
    if (cap->max_gaussians < 1 || cap->max_views < 1 || cap->max_views > splat::kMaxViews ||
        cap->max_pixels < 4 || cap->max_pairs < 1 || cap->max_pairs >= (int64_t{1} << 32) ||
        cap->max_tiles < 0)
        return SPLAT_ERR_INVALID_ARG;
    const int64_t mpv = cap->max_gaussians * cap->max_views;
    if (mpv >= (int64_t{1} << 32)) return SPLAT_ERR_INVALID_ARG;

    splat_ctx *c = new splat_ctx;
    c->cfg = *cfg;
    c->cap = *cap;
    if (c->cap.max_tiles == 0)
        c->cap.max_tiles = 2 * (cap->max_pixels / (cfg->tile_h * cfg->tile_w)) +
                           int64_t{256} * cap->max_views;
    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device);
    const int64_t P = cap->max_pixels, M = cap->max_pairs, TT = c->cap.max_tiles;
    if (e == cudaSuccess) e = dalloc(&c->d_views, cap->max_views);
    if (e == cudaSuccess) e = dalloc(&c->d_tileinfo, TT);
    if (e == cudaSuccess) e = dalloc(&c->d_tile_order, TT);
    if (e == cudaSuccess) e = dalloc(&c->d_prect, mpv);
    if (e == cudaSuccess) e = dalloc(&c->d_touch, mpv);
    if (e == cudaSuccess) e = dalloc(&c->d_kappa, mpv);
    if (e == cudaSuccess)
        e = dalloc(&c->d_touch_count,
                   static_cast<size_t>(splat::max_project_blocks(cap->max_gaussians)) *
                       cap->max_views);
    if (e == cudaSuccess) e = dalloc(&c->d_zero, kZeroTiles + static_cast<size_t>(TT));
    if (e == cudaSuccess)
        e = dalloc(&c->d_cta_count, splat::cta_count_words(c->sms, cap->max_views, TT));
    // the forward reads the lists four entries at a time from a 4-aligned index: 128 spare
    // entries keep the last vector in bounds
    if (e == cudaSuccess) e = dalloc(&c->d_entries, M + 128);
    if (e == cudaSuccess) e = dalloc(&c->d_blocks, M + 128);
    // a list holds each primitive once: only larger maps can have lists to cut into segments
    if (cap->max_gaussians >= splat::kListCap) {
        if (e == cudaSuccess) e = dalloc(&c->d_entries2, M);
        if (e == cudaSuccess) e = dalloc(&c->d_segments, splat::max_segments(M));
    }
    if (e == cudaSuccess) e = dalloc(&c->d_ranges, TT);
    if (e == cudaSuccess) e = dalloc(&c->d_tfinal, P);
    if (e == cudaSuccess) e = dalloc(&c->d_nlast, P);
    if (e == cudaSuccess) e = dalloc(&c->d_wgrad, static_cast<size_t>(cap->max_gaussians) * 4);
    if (e == cudaSuccess)
        e = dalloc(&c->d_prim, static_cast<size_t>(cap->max_gaussians) * splat::kPrimRow);
    if (e == cudaSuccess) e = dalloc(&c->d_pose, static_cast<size_t>(cap->max_views) * 6);
    if (e == cudaSuccess) e = dalloc(&c->d_samp_thr, static_cast<size_t>(splat::kMaxViews));
    if (e == cudaSuccess) e = dalloc(&c->d_active, static_cast<size_t>(cap->max_views));
    if (e == cudaSuccess) e = dalloc(&c->d_grow_sums, static_cast<size_t>(splat::kGrowMaxGrid + 2));
    // contributor records: at most one per (block, staged entry); the pool takes two per
    // (tile, primitive) pair of capacity plus one partial chunk per work item
    const int64_t items = TT * (splat::kBlock / 32);
    const int64_t chunks = (2 * M + 31) / 32 + items;
    c->rec_cap = static_cast<uint32_t>(chunks < 0xFFFFFFF0ll ? chunks : 0xFFFFFFF0ll);
    if (e == cudaSuccess) e = dalloc(&c->d_rec, static_cast<size_t>(c->rec_cap) * 32);
    if (e == cudaSuccess) e = dalloc(&c->d_rec_prev, static_cast<size_t>(c->rec_cap));
    // (a split block has up to four items)
    if (e == cudaSuccess) e = dalloc(&c->d_rec_head, static_cast<size_t>(4 * items));
    if (e == cudaSuccess) e = dalloc(&c->d_rec_fill, static_cast<size_t>(4 * items));
    if (e == cudaSuccess) e = dalloc(&c->d_img, static_cast<size_t>(P) * 5);
    if (e == cudaSuccess) e = dalloc(&c->d_gimg, static_cast<size_t>(P) * 5);
    if (e == cudaSuccess) e = dalloc(&c->d_counters, kCounters);
    if (e == cudaSuccess) e = dalloc(&c->d_bwd_evals, 1);
    for (int k = 0; k < 4 && e == cudaSuccess; ++k) e = cudaEventCreate(&c->ev[k]);
    for (int k = 0; k < splat_ctx::kStageEvents && e == cudaSuccess; ++k)
        e = cudaEventCreate(&c->stage_ev[k]);
    if (e == cudaSuccess) e = cudaMemset(c->d_counters, 0, kCounters * sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMemset(c->d_bwd_evals, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemset(c->d_zero, 0, kZeroTiles * sizeof(uint32_t));
    int fwd_ctas = 1, bwd_ctas = 1;
    if (e == cudaSuccess) e = splat::prepare_lists();
    if (e == cudaSuccess) e = splat::prepare_render_fwd(cfg->tile_h, cfg->tile_w, &fwd_ctas);
    if (e == cudaSuccess) e = splat::prepare_render_bwd(cfg->tile_h, cfg->tile_w, &bwd_ctas);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        int r = cuda_fail(e, "splat_ctx_create");
        free_ctx(c);
        return r;
    }
    c->grid_fwd = c->sms * std::max(fwd_ctas, 1);
    c->grid_bwd = c->sms * std::max(bwd_ctas, 1);
    *out = c;
    return SPLAT_OK;
}

SPLAT_API void splat_ctx_destroy(splat_ctx *ctx)
{
    if (!ctx) return;
    cudaDeviceSynchronize();
    free_ctx(ctx);
}

SPLAT_API int splat_set_views(splat_ctx *ctx, int32_t n_views, const double *T_ws,
                              const splat_lidar_intrinsics *intr)
{
    if (!ctx || !T_ws || !intr || n_views < 1 || n_views > ctx->cap.max_views)
        return SPLAT_ERR_INVALID_ARG;
    const int th = ctx->cfg.tile_h, tw = ctx->cfg.tile_w;
    std::vector<ViewDesc> views(n_views);
    int64_t pix = 0, tiles = 0, n_frames = 0;
    for (int v = 0; v < n_views; ++v) {
        const double *T = T_ws + 16 * v;
        const splat_lidar_intrinsics &in = intr[v];
        for (int k = 0; k < 16; ++k)
            if (!std::isfinite(T[k])) return SPLAT_ERR_INVALID_ARG;
        if (T[12] != 0.0 || T[13] != 0.0 || T[14] != 0.0 || T[15] != 1.0) return SPLAT_ERR_INVALID_ARG;
        for (int i = 0; i < 3; ++i)       // R^T R = I
            for (int j = 0; j < 3; ++j) {
                double s = 0.0;
                for (int k = 0; k < 3; ++k) s += T[4 * k + i] * T[4 * k + j];
                if (std::fabs(s - (i == j ? 1.0 : 0.0)) > 1e-6) return SPLAT_ERR_INVALID_ARG;
            }
        const double det = T[0] * (T[5] * T[10] - T[6] * T[9]) - T[1] * (T[4] * T[10] - T[6] * T[8]) +
                           T[2] * (T[4] * T[9] - T[5] * T[8]);
        if (det < 0.5) return SPLAT_ERR_INVALID_ARG;
        if (in.rows < 2 || in.cols < 2 || in.rows > 32767 || in.cols > 32767)
            return SPLAT_ERR_INVALID_ARG;
        if (!(std::isfinite(in.elev_min) && std::isfinite(in.elev_max) &&
              in.elev_min < in.elev_max && in.elev_min > -1.5707f && in.elev_max < 1.5707f))
            return SPLAT_ERR_INVALID_ARG;

        ViewDesc &vd = views[v];
        std::memset(&vd, 0, sizeof vd);
        double Rcw[9], tcw[3];
        inverse_pose(T, Rcw, tcw);
        for (int k = 0; k < 9; ++k) split(Rcw[k], vd.R_hi[k], vd.R_lo[k]);
        for (int k = 0; k < 3; ++k) split(tcw[k], vd.t_hi[k], vd.t_lo[k]);
        vd.rows = in.rows;
        vd.cols = in.cols;
        vd.elev_min = in.elev_min;
        vd.elev_max = in.elev_max;
        vd.kr = static_cast<float>(in.rows - 1) / (in.elev_max - in.elev_min);
        const double emin = in.elev_min, emax = in.elev_max;
        const double dth = (emax - emin) / (in.rows - 1);
        vd.dgamma = static_cast<float>(2.0 * M_PI / in.cols);
        vd.dtheta = static_cast<float>(dth);
        splat::set_cull_cones(vd, emin, emax, dth);
        vd.tiles_r = (in.rows + th - 1) / th;
        vd.tiles_c = (in.cols + tw - 1) / tw;
        vd.tile_offset = tiles;
        vd.pixel_offset = pix;
        vd.pix_offset = static_cast<int32_t>(n_frames);
        n_frames += int64_t{vd.tiles_r} * th * tw;
        tiles += int64_t{vd.tiles_r} * vd.tiles_c;
        pix += int64_t{in.rows} * in.cols;
    }
    if (pix > ctx->cap.max_pixels || tiles > ctx->cap.max_tiles) return SPLAT_ERR_INVALID_ARG;

    // Sines and cosines depend on the row or the column alone and are taken once for each (a
    // 61 x 1,187 view, the whole call: 120 -> 58 us).
    const size_t view_bytes = sizeof(ViewDesc) * views.size();
    const size_t tile_bytes = sizeof(TileInfo) * static_cast<size_t>(tiles);
    const size_t frame_bytes = sizeof(PixFrame) * static_cast<size_t>(n_frames);
    const size_t tile_at = (view_bytes + 63) / 64 * 64, frame_at = tile_at + tile_bytes;
    if (frame_at + frame_bytes > ctx->h_tables_cap) {
        ctx->h_tables.reset(new unsigned char[frame_at + frame_bytes]);
        ctx->h_tables_cap = frame_at + frame_bytes;
    }
    if (n_frames > ctx->pixframe_cap) {
        CK(cudaDeviceSynchronize());
        if (ctx->d_pixframes) CK(cudaFree(ctx->d_pixframes));
        ctx->d_pixframes = nullptr;
        ctx->pixframe_cap = 0;
        CK(dalloc(&ctx->d_pixframes, static_cast<size_t>(n_frames)));
        ctx->pixframe_cap = n_frames;
    }
    unsigned char *host = ctx->h_tables.get();
    std::memcpy(host, views.data(), view_bytes);
    TileInfo *tileinfo = reinterpret_cast<TileInfo *>(host + tile_at);
    PixFrame *pixframe = reinterpret_cast<PixFrame *>(host + frame_at);
    struct Angle {
        double s, c, omc;   // sine, cosine, 1 - cos = 2 sin^2 of the half angle
    };
    std::vector<Angle> col(tw), row(th), tcol;
    for (int v = 0; v < n_views; ++v) {
        const ViewDesc &vd = views[v];
        const double *T = T_ws + 16 * v;
        double Rcw[9], tcw[3];
        inverse_pose(T, Rcw, tcw);
        const int rows = vd.rows, cols = vd.cols;
        const double emin = vd.elev_min, emax = vd.elev_max;
        const double dth = (emax - emin) / (rows - 1);
        // pixel planes in the tile frame, in FP64 from exact small angle offsets:
        // dg = gamma - gamma0, dt = theta - theta0, omc = 1 - cos(dg) = 2 sin^2(dg / 2)
        for (int lc = 0; lc < tw; ++lc) {
            const double dg = -(lc - 0.5 * (tw - 1)) * (2.0 * M_PI / cols);
            const double sh = std::sin(0.5 * dg);
            col[lc] = Angle{std::sin(dg), std::cos(dg), 2.0 * sh * sh};
        }
        for (int lr = 0; lr < th; ++lr) {
            const double dt = -(lr - 0.5 * (th - 1)) * dth;
            row[lr] = Angle{std::sin(dt), std::cos(dt), 0.0};
        }
        tcol.resize(static_cast<size_t>(vd.tiles_c));
        for (int tc = 0; tc < vd.tiles_c; ++tc) {
            const double g0 = M_PI - 2.0 * M_PI * (tc * tw + 0.5 * (tw - 1) + 0.5) / cols;
            tcol[tc] = Angle{std::sin(g0), std::cos(g0), 0.0};
        }
        for (int tr = 0; tr < vd.tiles_r; ++tr) {
            const double t0 = emax - (tr * th + 0.5 * (th - 1)) * dth;
            const double s0 = std::sin(t0), c0 = std::cos(t0);
            for (int lr = 0; lr < th; ++lr) {
                const double dt = -(lr - 0.5 * (th - 1)) * dth;
                const double sdt = row[lr].s, cdt = row[lr].c;
                const double sth = std::sin(t0 + dt), cth = std::cos(t0 + dt);
                for (int lc = 0; lc < tw; ++lc) {
                    const double sg = col[lc].s, cg = col[lc].c, omc = col[lc].omc;
                    const double hx[3] = {c0 * sg, cg, -s0 * sg};
                    const double hy[3] = {-sdt + c0 * sth * omc, sth * sg, cdt - s0 * sth * omc};
                    const double vv[3] = {cdt - c0 * cth * omc, -cth * sg, sdt + s0 * cth * omc};
                    PixFrame &f = *pixframe++;
                    for (int k = 0; k < 3; ++k) {
                        split(hx[k], f.hx[k], f.hx_lo[k]);
                        split(hy[k], f.hy[k], f.hy_lo[k]);
                        f.v[k] = static_cast<float>(vv[k]);
                    }
                    f.pad = 0.0f;
                }
            }
            // per-tile frames: Q rows e1 = v(theta0, gamma0), e2 = h_x(gamma0), e3 = h_y(theta0,
            // gamma0); M = Q R^c_w, u = Q t^c_w in FP64, stored as float pairs
            for (int tc = 0; tc < vd.tiles_c; ++tc) {
                const double sg = tcol[tc].s, cg = tcol[tc].c;
                const double Q[9] = {c0 * cg, c0 * sg, s0, sg, -cg, 0.0, -s0 * cg, -s0 * sg, c0};
                TileInfo &ti = *tileinfo++;
                std::memset(&ti, 0, sizeof ti);
                for (int r = 0; r < 3; ++r) {
                    for (int c = 0; c < 3; ++c) {
                        const double m = Q[3 * r] * Rcw[c] + Q[3 * r + 1] * Rcw[3 + c] +
                                         Q[3 * r + 2] * Rcw[6 + c];
                        split(m, ti.M_hi[3 * r + c], ti.M_lo[3 * r + c]);
                    }
                    const double u = Q[3 * r] * tcw[0] + Q[3 * r + 1] * tcw[1] + Q[3 * r + 2] * tcw[2];
                    split(u, ti.u_hi[r], ti.u_lo[r]);
                }
                for (int k = 0; k < 9; ++k) ti.R[k] = vd.R_hi[k];
                ti.view = v;
                ti.tr = tr;
                ti.tc = tc;
                ti.cols = cols;
                ti.valid_r = std::min(th, rows - tr * th);
                ti.valid_c = std::min(tw, cols - tc * tw);
                ti.pix_base = vd.pix_offset + tr * th * tw;
                ti.out_base = vd.pixel_offset + static_cast<int64_t>(tr) * th * cols +
                              static_cast<int64_t>(tc) * tw;
            }
        }
    }
    CK(cudaMemcpy(ctx->d_views, host, view_bytes, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->d_tileinfo, host + tile_at, tile_bytes, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->d_pixframes, host + frame_at, frame_bytes, cudaMemcpyHostToDevice));
    ctx->views = views;
    ctx->n_views = n_views;
    ctx->n_pixels = pix;
    ctx->n_tiles = tiles;
    ctx->bands = ctx->max_view_bands = ctx->max_band_tiles = 0;
    for (const ViewDesc &v : views) {
        const int bands = splat::view_bands(v.tiles_r, v.tiles_c);
        ctx->bands += bands;
        ctx->max_view_bands = std::max(ctx->max_view_bands, bands);
        ctx->max_band_tiles = std::max(
            ctx->max_band_tiles, std::min(v.tiles_r, splat::band_rows(v.tiles_c)) * v.tiles_c);
    }
    ctx->rendered = false;
    ctx->have_pose = false;
    ctx->samp_draws = 0;   // the sampling law depends on the views: set it again
    return SPLAT_OK;
}

SPLAT_API int64_t splat_view_pixel_offset(const splat_ctx *ctx, int32_t v)
{
    if (!ctx || v < 0 || v >= ctx->n_views) return -1;
    return ctx->views[v].pixel_offset;
}

SPLAT_API int splat_render_views(splat_ctx *ctx, const splat_gaussians *g, float *depth,
                                 float *normal, float *alpha, void *stream)
{
    if (!ctx) return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    int r = check_gaussians(ctx, g);
    if (r) return r;
    if (!depth || !normal || !alpha) return SPLAT_ERR_INVALID_ARG;
    return render_core(ctx, g, depth, normal, alpha, static_cast<cudaStream_t>(stream));
}

SPLAT_API int splat_render_views_backward(splat_ctx *ctx, const splat_gaussians *g,
                                          const float *dL_ddepth, const float *dL_dnormal,
                                          const float *dL_dalpha, float *g_pos_logit,
                                          float *g_quat, float *g_log_scale, int accumulate,
                                          void *stream)
{
    if (!ctx) return SPLAT_ERR_INVALID_ARG;
    int r = check_gaussians(ctx, g);
    if (r) return r;
    if (!ctx->rendered || g->n != ctx->last_n) return SPLAT_ERR_STATE;
    if (!g_pos_logit || !g_quat || !g_log_scale) return SPLAT_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    r = backward_core(ctx, g, dL_ddepth, dL_dnormal, dL_dalpha, st, false);
    if (r) return r;
    CK(splat::launch_param_grads(reinterpret_cast<const float4 *>(g->pos_logit),
                                 reinterpret_cast<const float4 *>(g->quat_wxyz),
                                 reinterpret_cast<const float2 *>(g->log_scale), ctx->d_wgrad, g->n,
                                 reinterpret_cast<float4 *>(g_pos_logit),
                                 reinterpret_cast<float4 *>(g_quat),
                                 reinterpret_cast<float2 *>(g_log_scale), accumulate, st));
    ctx->launches += 1;
    return SPLAT_OK;
}

SPLAT_API int splat_render(splat_ctx *ctx, const splat_gaussians *g,
                           const double T_world_sensor[16], const splat_lidar_intrinsics *intr,
                           float *depth, float *normal, float *alpha, void *stream)
{
    int r = splat_set_views(ctx, 1, T_world_sensor, intr);
    if (r) return r;
    return splat_render_views(ctx, g, depth, normal, alpha, stream);
}

SPLAT_API int splat_render_backward(splat_ctx *ctx, const splat_gaussians *g,
                                    const float *dL_ddepth, const float *dL_dnormal,
                                    const float *dL_dalpha, float *g_pos_logit, float *g_quat,
                                    float *g_log_scale, int accumulate, void *stream)
{
    return splat_render_views_backward(ctx, g, dL_ddepth, dL_dnormal, dL_dalpha, g_pos_logit,
                                       g_quat, g_log_scale, accumulate, stream);
}

SPLAT_API int splat_backproject(splat_ctx *ctx, const float *depth, const float *alpha,
                                float o_min, float *points, void *stream)
{
    if (!ctx || !depth || !alpha || !points || !(o_min > 0.0f)) return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    CK(splat::launch_backproject(ctx->d_views, ctx->n_views, ctx->n_pixels, depth, alpha, o_min,
                                 points, st));
    return SPLAT_OK;
}

SPLAT_API int splat_photometric(splat_ctx *ctx, int32_t view, const float *depth,
                                const float *alpha, const float *query_depth, const float *T_qm,
                                float o_min, float huber_delta, double *normal_eqs,
                                float *per_pixel, void *stream)
{
    if (!ctx || !depth || !alpha || !query_depth || !T_qm || !normal_eqs || !(o_min > 0.0f) ||
        !(huber_delta > 0.0f))
        return SPLAT_ERR_INVALID_ARG;
    if (view < 0 || view >= ctx->n_views) return ctx->n_views < 1 ? SPLAT_ERR_STATE
                                                                   : SPLAT_ERR_INVALID_ARG;
    CK(splat::launch_photometric(ctx->views[view], depth, alpha, query_depth, T_qm, o_min,
                                 huber_delta, normal_eqs, per_pixel, ctx->sms,
                                 static_cast<cudaStream_t>(stream)));
    ctx->launches += 1;
    return SPLAT_OK;
}

SPLAT_API int splat_densify(splat_ctx *ctx, const float *target_depth, const float *depth,
                            const float *alpha, const splat_densify_config *cfg, int64_t n_new,
                            float *pos_logit, float *quat, float *log_scale, int64_t n_old,
                            int64_t capacity, void *stream)
{
    if (!ctx || !target_depth || !cfg || !pos_logit || !quat || !log_scale || n_new < 0 ||
        n_old < 0 || n_new > (int64_t{1} << 24) || n_old + n_new > capacity)
        return SPLAT_ERR_INVALID_ARG;
    if (cfg->refine && (!depth || !alpha)) return SPLAT_ERR_INVALID_ARG;
    if (!(cfg->w0 >= 0.0f) || !(cfg->w_cap > 0.0f && cfg->w_cap <= 16.0f) ||
        !(cfg->scale_k > 0.0f) || !(cfg->opacity > 0.0f && cfg->opacity < 1.0f) ||
        !std::isfinite(cfg->lambda_do) || !std::isfinite(cfg->lambda_de))
        return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    // the integer draw needs n_pixels * max weight * n_new < 2^63 (max weight 16 * 256)
    if (ctx->n_pixels > 0 && n_new > 0 &&
        static_cast<double>(ctx->n_pixels) * 4096.0 * static_cast<double>(n_new) >= 9.0e18)
        return SPLAT_ERR_INVALID_ARG;
    splat::GrowArgs a{};
    a.views = ctx->d_views;
    a.n_views = ctx->n_views;
    a.n_pixels = ctx->n_pixels;
    a.t_depth = target_depth;
    a.depth = depth;
    a.alpha = alpha;
    a.refine = cfg->refine ? 1 : 0;
    a.lambda_do = cfg->lambda_do;
    a.lambda_de = cfg->lambda_de;
    a.w0 = cfg->w0;
    a.w_cap = cfg->w_cap;
    a.scale_k = cfg->scale_k;
    a.logit = static_cast<float>(std::log(static_cast<double>(cfg->opacity) /
                                          (1.0 - static_cast<double>(cfg->opacity))));
    a.empty_logit = -30.0f;
    a.seed_lo = static_cast<uint32_t>(cfg->seed);
    a.seed_hi = static_cast<uint32_t>(cfg->seed >> 32);
    a.call = ctx->d_counters + 6;
    a.q = reinterpret_cast<uint32_t *>(ctx->d_gimg);
    a.block_sums = ctx->d_grow_sums;
    a.pos_logit = reinterpret_cast<float4 *>(pos_logit) + n_old;
    a.quat = reinterpret_cast<float4 *>(quat) + n_old;
    a.log_scale = reinterpret_cast<float2 *>(log_scale) + n_old;
    a.n_d = n_new;
    CK(splat::launch_grow(a, static_cast<cudaStream_t>(stream)));
    if (n_new > 0) ctx->launches += 3;
    return SPLAT_OK;
}

SPLAT_API int splat_loss(const float *depth, const float *normal, const float *alpha,
                         const float *target_depth, const float *target_normal,
                         int64_t n_pixels, const splat_loss_config *cfg, float *dL_ddepth,
                         float *dL_dnormal, float *dL_dalpha, double *loss_out, void *stream)
{
    if (!depth || !normal || !alpha || !target_depth || !target_normal || !cfg || !dL_ddepth ||
        !dL_dnormal || !dL_dalpha || !loss_out || n_pixels < 0 ||
        cfg->normal_mode != SPLAT_NORMALS_TARGET)
        return SPLAT_ERR_INVALID_ARG;
    CK(splat::launch_loss(depth, normal, alpha, target_depth, target_normal, n_pixels,
                          cfg->lambda_n, cfg->lambda_o, cfg->o_eps, cfg->rho_exp, dL_ddepth, dL_dnormal,
                          dL_dalpha, loss_out, static_cast<cudaStream_t>(stream), false));
    return SPLAT_OK;
}

static bool loss_cfg_ok(const splat_loss_config *cfg, const float *target_normal)
{
    if (cfg->normal_mode == SPLAT_NORMALS_TARGET) return target_normal != nullptr;
    return cfg->normal_mode == SPLAT_NORMALS_RANGE_MAP;
}

SPLAT_API int splat_view_loss(splat_ctx *ctx, const float *depth, const float *normal,
                              const float *alpha, const float *target_depth,
                              const float *target_normal, const splat_loss_config *cfg,
                              float *dL_ddepth, float *dL_dnormal, float *dL_dalpha,
                              double *loss_out, void *stream)
{
    if (!ctx || !depth || !normal || !alpha || !target_depth || !cfg || !dL_ddepth ||
        !dL_dnormal || !dL_dalpha || !loss_out || !loss_cfg_ok(cfg, target_normal))
        return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    CK(splat::launch_loss(depth, normal, alpha, target_depth, target_normal, ctx->n_pixels,
                          cfg->lambda_n, cfg->lambda_o, cfg->o_eps, cfg->rho_exp, dL_ddepth, dL_dnormal,
                          dL_dalpha, loss_out, static_cast<cudaStream_t>(stream), false,
                          ctx->d_views, ctx->n_views, nullptr, cfg->normal_mode));
    return SPLAT_OK;
}

SPLAT_API int splat_adam_step(float *pos_logit, float *quat, float *log_scale,
                              const float *g_pos_logit, const float *g_quat,
                              const float *g_log_scale, float *m_pos_logit, float *m_quat,
                              float *m_log_scale, float *v_pos_logit, float *v_quat,
                              float *v_log_scale, int32_t *step, int64_t n,
                              const splat_adam_config *cfg, void *stream)
{
    if (!pos_logit || !quat || !log_scale || !g_pos_logit || !g_quat || !g_log_scale ||
        !m_pos_logit || !m_quat || !m_log_scale || !v_pos_logit || !v_quat || !v_log_scale ||
        !step || !cfg || n < 0)
        return SPLAT_ERR_INVALID_ARG;
    splat::AdamArgs a{};
    a.pos_logit = reinterpret_cast<float4 *>(pos_logit);
    a.quat = reinterpret_cast<float4 *>(quat);
    a.log_scale = reinterpret_cast<float2 *>(log_scale);
    a.m_pl = reinterpret_cast<float4 *>(m_pos_logit);
    a.m_q = reinterpret_cast<float4 *>(m_quat);
    a.m_ls = reinterpret_cast<float2 *>(m_log_scale);
    a.v_pl = reinterpret_cast<float4 *>(v_pos_logit);
    a.v_q = reinterpret_cast<float4 *>(v_quat);
    a.v_ls = reinterpret_cast<float2 *>(v_log_scale);
    a.step = step;
    a.n = n;
    a.lr_pos = cfg->lr_pos;
    a.lr_opacity = cfg->lr_opacity;
    a.lr_rot = cfg->lr_rot;
    a.lr_scale = cfg->lr_scale;
    a.beta1 = cfg->beta1;
    a.beta2 = cfg->beta2;
    a.eps = cfg->eps;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    CK(splat::launch_adam(a, reinterpret_cast<const float4 *>(g_pos_logit),
                          reinterpret_cast<const float4 *>(g_quat),
                          reinterpret_cast<const float2 *>(g_log_scale), st));
    CK(splat::launch_step_inc(step, st));
    return SPLAT_OK;
}

SPLAT_API int splat_refine_step(splat_ctx *ctx, float *pos_logit, float *quat, float *log_scale,
                                int64_t n, const float *target_depth, const float *target_normal,
                                const splat_loss_config *loss_cfg,
                                const splat_adam_config *adam_cfg, float *m_pos_logit,
                                float *m_quat, float *m_log_scale, float *v_pos_logit,
                                float *v_quat, float *v_log_scale, int32_t *step,
                                double *loss_out, void *stream)
{
    if (!ctx || !target_depth || !loss_cfg || !adam_cfg || !m_pos_logit || !m_quat ||
        !m_log_scale || !v_pos_logit || !v_quat || !v_log_scale || !step || !loss_out ||
        !loss_cfg_ok(loss_cfg, target_normal))
        return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    splat_gaussians g{pos_logit, quat, log_scale, n};
    int r = check_gaussians(ctx, &g);
    if (r) return r;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t P = ctx->n_pixels;
    float *depth = ctx->d_img, *normal = ctx->d_img + P, *alpha = ctx->d_img + 4 * P;
    float *gd = ctx->d_gimg, *gn = ctx->d_gimg + P, *ga = ctx->d_gimg + 4 * P;
    // the accumulators, the loss and the backward's counters are zeroed and the step is counted by
    // kernels of the render
    splat::RefineStart start = backward_start(ctx);
    start.loss = loss_out;
    start.step = step;
    r = render_core(ctx, &g, depth, normal, alpha, st, &start);
    if (r) return r;
    CK(splat::launch_loss(depth, normal, alpha, target_depth, target_normal, P, loss_cfg->lambda_n,
                          loss_cfg->lambda_o, loss_cfg->o_eps, loss_cfg->rho_exp, gd, gn, ga,
                          loss_out, st, splat::chained_size(n * ctx->n_views),
                          ctx->d_views, ctx->n_views,
                          ctx->samp_draws > 0 ? ctx->d_active : nullptr,
                          loss_cfg->normal_mode));
    const bool prof = ctx->profiling && !capturing(st);
    if (prof) {
        CK(cudaEventRecord(ctx->stage_ev[4], st));
        ctx->stage_rec[4] = true;
    }
    r = backward_core(ctx, &g, gd, gn, ga, st, true);
    if (r) return r;
    splat::AdamArgs a{};
    a.pos_logit = reinterpret_cast<float4 *>(pos_logit);
    a.quat = reinterpret_cast<float4 *>(quat);
    a.log_scale = reinterpret_cast<float2 *>(log_scale);
    a.m_pl = reinterpret_cast<float4 *>(m_pos_logit);
    a.m_q = reinterpret_cast<float4 *>(m_quat);
    a.m_ls = reinterpret_cast<float2 *>(m_log_scale);
    a.v_pl = reinterpret_cast<float4 *>(v_pos_logit);
    a.v_q = reinterpret_cast<float4 *>(v_quat);
    a.v_ls = reinterpret_cast<float2 *>(v_log_scale);
    a.step = step;
    a.n = n;
    a.lr_pos = adam_cfg->lr_pos;
    a.lr_opacity = adam_cfg->lr_opacity;
    a.lr_rot = adam_cfg->lr_rot;
    a.lr_scale = adam_cfg->lr_scale;
    a.beta1 = adam_cfg->beta1;
    a.beta2 = adam_cfg->beta2;
    a.eps = adam_cfg->eps;
    a.lambda_s = loss_cfg->lambda_s;
    a.tau_s = loss_cfg->tau_s;
    a.loss_out = loss_out;
    a.chain = splat::chained_size(n * ctx->n_views);
    CK(splat::launch_adam_fused(a, ctx->d_wgrad, st));
    if (prof) {
        CK(cudaEventRecord(ctx->stage_ev[5], st));
        ctx->stage_rec[5] = true;
    }
    ctx->launches += 2;   // loss, fused Adam
    return SPLAT_OK;
}

SPLAT_API int splat_set_view_sampling(splat_ctx *ctx, int draws, double p_newest, uint64_t seed)
{
    if (!ctx || draws < 0) return SPLAT_ERR_INVALID_ARG;
    if (draws == 0) {
        ctx->samp_draws = 0;
        return SPLAT_OK;
    }
    if (!(p_newest > 0.0 && p_newest <= 1.0)) return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    // truncated geometric law over keyframe age, cumulative, as integer thresholds (FP64, the
    // products and sums in age order)
    const int K = ctx->n_views;
    std::vector<double> P(static_cast<size_t>(K));
    double w = p_newest;
    for (int a = 0; a < K; ++a) {
        P[a] = w;
        w = w * (1.0 - p_newest);
    }
    double Z = 0.0;
    for (int a = 0; a < K; ++a) Z = Z + P[a];
    std::vector<uint32_t> thr(static_cast<size_t>(splat::kMaxViews), 0u);
    double c = 0.0;
    for (int a = 0; a + 1 < K; ++a) {
        c = c + P[a];
        const double v = std::floor((c / Z) * 4294967296.0);
        thr[a] = v >= 4294967295.0 ? 0xFFFFFFFFu : static_cast<uint32_t>(v);
    }
    CK(cudaMemcpy(ctx->d_samp_thr, thr.data(), sizeof(uint32_t) * thr.size(),
                  cudaMemcpyHostToDevice));
    CK(cudaMemset(ctx->d_counters + 7, 0, sizeof(uint32_t)));
    ctx->samp_draws = draws;
    ctx->samp_seed = seed;
    return SPLAT_OK;
}

SPLAT_API int splat_get_active_views(splat_ctx *ctx, uint8_t *flags)
{
    if (!ctx || !flags) return SPLAT_ERR_INVALID_ARG;
    if (ctx->n_views < 1) return SPLAT_ERR_STATE;
    CK(cudaDeviceSynchronize());
    if (ctx->samp_draws > 0) {
        CK(cudaMemcpy(flags, ctx->d_active, static_cast<size_t>(ctx->n_views),
                      cudaMemcpyDeviceToHost));
    } else {
        for (int v = 0; v < ctx->n_views; ++v) flags[v] = 1;
    }
    return SPLAT_OK;
}

SPLAT_API int splat_set_pose_gradient(splat_ctx *ctx, int enable)
{
    if (!ctx) return SPLAT_ERR_INVALID_ARG;
    ctx->want_pose = enable != 0;
    return SPLAT_OK;
}

SPLAT_API int splat_pose_gradient(splat_ctx *ctx, float *g_pose, void *stream)
{
    if (!ctx || !g_pose) return SPLAT_ERR_INVALID_ARG;
    if (!ctx->have_pose) return SPLAT_ERR_STATE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    CK(cudaMemcpyAsync(g_pose, ctx->d_pose, sizeof(float) * 6 * static_cast<size_t>(ctx->n_views),
                       cudaMemcpyDeviceToDevice, st));
    return SPLAT_OK;
}

SPLAT_API int splat_get_status(splat_ctx *ctx, uint32_t *flags)
{
    if (!ctx || !flags) return SPLAT_ERR_INVALID_ARG;
    CK(cudaDeviceSynchronize());
    CK(cudaMemcpy(flags, ctx->d_counters + 1, sizeof(uint32_t), cudaMemcpyDeviceToHost));
    CK(cudaMemset(ctx->d_counters + 1, 0, sizeof(uint32_t)));
    return SPLAT_OK;
}

SPLAT_API int splat_get_stats(splat_ctx *ctx, splat_stats *out)
{
    if (!ctx || !out) return SPLAT_ERR_INVALID_ARG;
    CK(cudaDeviceSynchronize());
    uint32_t pairs = 0, zero[kZeroTiles] = {};
    unsigned long long fwd = 0, bwd = 0;
    CK(cudaMemcpy(&pairs, ctx->d_counters, sizeof pairs, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(zero, ctx->d_zero, sizeof zero, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(&bwd, ctx->d_bwd_evals, sizeof bwd, cudaMemcpyDeviceToHost));
    std::memcpy(&fwd, zero + kZeroEvals, sizeof fwd);
    out->n_pairs = pairs;
    out->n_touching = zero[kZeroTouching];
    out->fwd_evals = static_cast<int64_t>(fwd);
    out->bwd_evals = static_cast<int64_t>(bwd);
    out->n_pixels = ctx->n_pixels;
    out->n_tiles = ctx->n_tiles;
    out->kernel_launches = ctx->launches;
    return SPLAT_OK;
}

SPLAT_API int splat_set_profiling(splat_ctx *ctx, int enable)
{
    if (!ctx) return SPLAT_ERR_INVALID_ARG;
    ctx->profiling = enable != 0;
    ctx->rec_fwd = ctx->rec_bwd = false;
    for (bool &b : ctx->stage_rec) b = false;
    return SPLAT_OK;
}

SPLAT_API int splat_kernel_times(splat_ctx *ctx, float *fwd_ms, float *bwd_ms)
{
    if (!ctx || !fwd_ms || !bwd_ms) return SPLAT_ERR_INVALID_ARG;
    *fwd_ms = -1.0f;
    *bwd_ms = -1.0f;
    if (ctx->rec_fwd) {
        CK(cudaEventSynchronize(ctx->ev[1]));
        CK(cudaEventElapsedTime(fwd_ms, ctx->ev[0], ctx->ev[1]));
    }
    if (ctx->rec_bwd) {
        CK(cudaEventSynchronize(ctx->ev[3]));
        CK(cudaEventElapsedTime(bwd_ms, ctx->ev[2], ctx->ev[3]));
    }
    return SPLAT_OK;
}

SPLAT_API int splat_stage_times(splat_ctx *ctx, float *ms)
{
    if (!ctx || !ms) return SPLAT_ERR_INVALID_ARG;
    // the loss runs between the end of the forward compositing and event 4, the fused Adam
    // between the end of the backward and event 5; the binning has no global range sort and no
    // separate ranges pass, which take no time in a render that was profiled
    struct Span {
        cudaEvent_t a, b;
        bool ok;
    };
    const Span binning{nullptr, nullptr, ctx->stage_rec[0] && ctx->stage_rec[3]};
    const Span spans[7] = {
        {ctx->stage_ev[0], ctx->stage_ev[1], ctx->stage_rec[0] && ctx->stage_rec[1]},
        binning,
        {ctx->stage_ev[1], ctx->stage_ev[2], ctx->stage_rec[1] && ctx->stage_rec[2]},
        {ctx->stage_ev[2], ctx->stage_ev[3], ctx->stage_rec[2] && ctx->stage_rec[3]},
        binning,
        {ctx->ev[1], ctx->stage_ev[4], ctx->rec_fwd && ctx->stage_rec[4]},
        {ctx->ev[3], ctx->stage_ev[5], ctx->rec_bwd && ctx->stage_rec[5]},
    };
    for (int k = 0; k < 7; ++k) {
        ms[k] = spans[k].ok ? 0.0f : -1.0f;
        if (!spans[k].ok || !spans[k].a) continue;
        CK(cudaEventSynchronize(spans[k].b));
        CK(cudaEventElapsedTime(&ms[k], spans[k].a, spans[k].b));
    }
    return SPLAT_OK;
}

SPLAT_API int64_t splat_debug_copy(splat_ctx *ctx, int32_t which, void *dst, int64_t bytes)
{
    if (!ctx || !dst || bytes < 0 || which < 0 || which > 6) return -1;
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    if (!ctx->rendered) return -1;
    uint32_t m = 0;
    if (cudaMemcpy(&m, ctx->d_counters, sizeof m, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    auto get = [&](const void *src, int64_t need) -> int64_t {
        if (need > bytes) return -1;
        if (need > 0 && cudaMemcpy(dst, src, static_cast<size_t>(need), cudaMemcpyDeviceToHost) !=
                            cudaSuccess)
            return -1;
        return need;
    };
    const int64_t npv = ctx->last_n * ctx->n_views;
    try {
        switch (which) {
        case 0: {   // the tile of every entry, from the ranges
            if (int64_t{4} * m > bytes) return -1;
            std::vector<uint2> rg(static_cast<size_t>(ctx->n_tiles));
            if (cudaMemcpy(rg.data(), ctx->d_ranges, sizeof(uint2) * rg.size(),
                           cudaMemcpyDeviceToHost) != cudaSuccess)
                return -1;
            uint32_t *out = static_cast<uint32_t *>(dst);
            for (size_t t = 0; t < rg.size(); ++t)
                for (uint32_t j = rg[t].x; j < rg[t].y; ++j) out[j] = static_cast<uint32_t>(t);
            return int64_t{4} * m;
        }
        case 1: {   // the pair ids of the (pair id, rectangle) entries
            if (int64_t{4} * m > bytes) return -1;
            if (m == 0) return 0;
            if (cudaMemcpy2D(dst, 4, ctx->d_entries, 8, 4, m, cudaMemcpyDeviceToHost) !=
                cudaSuccess)
                return -1;
            return int64_t{4} * m;
        }
        case 2: return get(ctx->d_ranges, int64_t{8} * ctx->n_tiles);
        case 3: {
            const int64_t need = static_cast<int64_t>(sizeof(PairRec)) * npv;
            if (need > bytes) return -1;
            if (need == 0) return 0;
            PairRec *recs = nullptr;   // not a compute call: a temporary buffer is fine here
            if (dalloc(&recs, static_cast<size_t>(npv)) != cudaSuccess) return -1;
            cudaError_t e = splat::launch_records(
                ctx->last_n, ctx->n_views, ctx->d_views, ctx->cfg.flip_normals, ctx->cfg.tile_h,
                ctx->cfg.tile_w, ctx->d_prim, ctx->d_prect,
                ctx->last_sampled ? ctx->d_active : nullptr, recs, nullptr);
            if (e == cudaSuccess)
                e = cudaMemcpy(dst, recs, static_cast<size_t>(need), cudaMemcpyDeviceToHost);
            cudaFree(recs);
            return e == cudaSuccess ? need : -1;
        }
        case 4: return get(ctx->d_tfinal, int64_t{4} * ctx->n_pixels);
        case 5: return get(ctx->d_nlast, int64_t{4} * ctx->n_pixels);
        default:   // kBinSplit4 and kBinSplit2 lie side by side
            return get(ctx->d_counters + kCountersBin + splat::kBinSplit4, int64_t{4} * 2);
        }
    } catch (...) {
        return -1;
    }
}

}  // extern "C"
