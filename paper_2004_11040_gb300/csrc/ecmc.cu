// ecmc.cu -- the C ABI of libecmc: multithreaded event-chain Monte Carlo for
// hard disks on one GPU (sm_103a), after Li, Todo, Maggs & Krauth,
// "Multithreaded event-chain Monte Carlo with local times" (arXiv:2004.11040).
//
// Contexts, batches, read-backs, the device memory cache and the leg that
// allocates nothing. The legs themselves run in graph.cu, for both kinds of
// context: with ECMC_GRAPH the conflict flag is on the disks a chain reads,
// otherwise on the cells its scans cover.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "devmem.h"
#include "ecmc.h"
#include "graph.h"

namespace {

// Coordinates in [0, L) (counted in *bad_xy; not checked with x == null) and
// distinct active ids in [0, n) (*bad_id), checked on the device where the
// inputs already are. seen[] must be zero.
__global__ void k_check_inputs(const double *x, const double *y, const int32_t *active,
                               int64_t n, int k, double L, uint32_t *seen,
                               unsigned long long *bad_xy, unsigned long long *bad_id) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t q = t0; x && q < n; q += stride)
        if (!(x[q] >= 0.0 && x[q] < L && y[q] >= 0.0 && y[q] < L)) atomicAdd(bad_xy, 1ull);
    for (int64_t c = t0; c < k; c += stride) {
        const int32_t a = active[c];
        if (a < 0 || (int64_t)a >= n || atomicExch(seen + a, 1u) != 0u) atomicAdd(bad_id, 1ull);
    }
}

}  // namespace

void graph_check_inputs(const double *x, const double *y, const int32_t *active, int64_t n, int k,
                        double L, uint32_t *seen, unsigned long long *bad_xy,
                        unsigned long long *bad_id, cudaStream_t st) {
    const int64_t work = x ? std::max<int64_t>(n, k) : (int64_t)k;
    const unsigned blocks = (unsigned)std::min<int64_t>((work + 255) / 256, 4096);
    k_check_inputs<<<blocks, 256, 0, st>>>(x, y, active, n, k, L, seen, bad_xy, bad_id);
}

// ------------------------------------------------ device memory cache

namespace {
struct CudaBackend {
    int alloc(void **p, size_t bytes) {
        const cudaError_t e = cudaMalloc(p, bytes);
        if (e != cudaSuccess) (void)cudaGetLastError();
        return (int)e;
    }
    void free(void *p) { cudaFree(p); }
};
constexpr int DM_MAX_DEVICES = 64;
constexpr size_t DM_DEFAULT_LIMIT = (size_t)4 << 30;  // cached bytes per device
std::mutex g_dm_mu;
BlockCache<CudaBackend> *g_dm[DM_MAX_DEVICES];
size_t g_dm_limit = DM_DEFAULT_LIMIT;

// The cache of device dev (created on first use, never destroyed: its blocks
// would outlive the CUDA runtime at process exit).
BlockCache<CudaBackend> *dm_cache(int dev) {
    if (dev < 0 || dev >= DM_MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lock(g_dm_mu);
    if (!g_dm[dev]) g_dm[dev] = new BlockCache<CudaBackend>(g_dm_limit);
    return g_dm[dev];
}
}  // namespace

int dm_alloc(void **p, size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    BlockCache<CudaBackend> *c = dm_cache(dev);
    if (!c) return CudaBackend().alloc(p, bytes);
    return c->acquire(p, bytes);
}

void dm_free(void *p) {
    if (!p) return;
    // the block goes back to the cache of the device that holds it
    cudaPointerAttributes a;
    int dev = -1;
    if (cudaPointerGetAttributes(&a, p) == cudaSuccess)
        dev = a.device;
    else
        (void)cudaGetLastError();
    BlockCache<CudaBackend> *c = dm_cache(dev);
    if (c)
        c->release(p);
    else
        cudaFree(p);
}

extern "C" int ecmc_set_cache_limit(int64_t bytes) {
    if (bytes < 0) return ECMC_EINVAL;
    std::lock_guard<std::mutex> lock(g_dm_mu);
    g_dm_limit = (size_t)bytes;
    for (auto *c : g_dm)
        if (c) c->set_limit(g_dm_limit);
    return ECMC_OK;
}

extern "C" int ecmc_cache_info(int64_t *cached_bytes, int64_t *in_use_bytes, int64_t *hits,
                               int64_t *misses) {
    DevCacheInfo t = {0, 0, 0, 0};
    {
        std::lock_guard<std::mutex> lock(g_dm_mu);
        for (auto *c : g_dm) {
            if (!c) continue;
            const DevCacheInfo i = c->info();
            t.cached_bytes += i.cached_bytes;
            t.in_use_bytes += i.in_use_bytes;
            t.hits += i.hits;
            t.misses += i.misses;
        }
    }
    if (cached_bytes) *cached_bytes = t.cached_bytes;
    if (in_use_bytes) *in_use_bytes = t.in_use_bytes;
    if (hits) *hits = t.hits;
    if (misses) *misses = t.misses;
    return ECMC_OK;
}

struct ecmc_ctx {
    ecmc_params p;
    GraphCtx *graph = nullptr;  // the system (graph.cu)
    bool cells = false;         // the flag is on cells (no ECMC_GRAPH)
    int C = 4;                  // slots per cell
    cudaStream_t stream = nullptr;
    std::string err;
    int64_t lifts_total = 0;
    int64_t legs_total = 0;
    int64_t conflict_legs = 0;
    int64_t repaired = 0;
    int64_t continued = 0;
    int64_t restarts = 0;
    int64_t row_windows = 0;
    int64_t blocked = 0;
    int64_t cwindows = 0;
    int64_t horizon = 0;
    int64_t order_err = 0;
    unsigned long long wait_ns = BARRIER_TIMEOUT_NS;  // bound on device waits
    double device_ms = 0.0;
    ecmc_profile_t prof = {};
    int32_t direction = 0;  // 0: +x; 1: +y (the context is stored transposed)
    // scratch of ecmc_positions, one block
    char *exp = nullptr;
    int64_t exp_bytes = 0;
    double *exp_x = nullptr, *exp_t = nullptr;
};

static std::string g_create_err;

static int fail(ecmc_ctx *ctx, int code, const std::string &msg) {
    if (ctx)
        ctx->err = msg;
    else
        g_create_err = msg;
    return code;
}

#define CU(call)                                                                        \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return fail(ctx, ECMC_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

static int pick_cells(const ecmc_params *p, int *nc_out, int *C_out) {
    const double d = p->d, L = p->box;
    int nc = p->cells_per_side;
    if (nc == 0) {
        nc = (int)(L / (d * (1.0 + std::ldexp(1.0, -20))));
        while (nc > 3 && !(L / nc >= d * (1.0 + std::ldexp(1.0, -20)))) --nc;
    }
    if (nc < 3) return -1;
    const double a = L / nc;
    if (!(a >= d * (1.0 + std::ldexp(1.0, -20)))) return -1;
    // At most 4 centres at mutual distance >= d fit in a cell with a < sqrt(2) d
    // (one per quadrant); at most 6 for a < 1.664 d (a 3 x 2 split).
    int C;
    if (a < std::sqrt(2.0) * d * (1.0 - 1e-9))
        C = 4;
    else if (a < 1.664 * d)
        C = 8;
    else
        return -1;
    *nc_out = nc;
    *C_out = C;
    return 0;
}

// Parts of the scratch of ecmc_positions (x and t, each on a 256-byte boundary).
static int64_t export_layout(int64_t n, ecmc_ctx *ctx) {
    const int64_t n8 = (n * 8 + 255) & ~(int64_t)255;
    if (ctx) {
        ctx->exp_x = (double *)ctx->exp;
        ctx->exp_t = (double *)(ctx->exp + n8);
    }
    return 2 * n8;
}

// The system of a new context; host inputs are uploaded first.
static int create_graph(ecmc_ctx *ctx, int nc, const double *x, const double *y,
                        const int32_t *active) {
    const ecmc_params *p = &ctx->p;
    const size_t n = (size_t)p->n, k = (size_t)p->n_chains;
    int rc = 0;
    char *scratch = nullptr;
    if (!(p->flags & ECMC_INPUT_DEVICE)) {
        if (dm_alloc_t(&scratch, 2 * n * 8 + k * 4) != 0) {
            g_create_err = "cudaMalloc failed (inputs)";
            return ECMC_ENOMEM;
        }
        double *dx = (double *)scratch, *dy = dx + n;
        int32_t *da = (int32_t *)(dy + n);
        cudaError_t e = cudaMemcpyAsync(dx, x, n * 8, cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(dy, y, n * 8, cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(da, active, k * 4, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            g_create_err = "input upload";
            rc = ECMC_ECUDA;
        }
        x = dx;
        y = dy;
        active = da;
    }
    if (!rc) {
        std::string err;
        rc = graph_create(p, nc, x, y, active, ctx->stream, &ctx->graph, err);
        if (rc) g_create_err = err;
    }
    // (copies, the check or the build may still read the inputs)
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        (void)cudaGetLastError();
        if (!rc) {
            g_create_err = "graph build";
            rc = ECMC_ECUDA;
        }
    }
    dm_free(scratch);
    return rc;
}

extern "C" int ecmc_context_bytes(const ecmc_params *p, int64_t *bytes) {
    if (!p || !bytes) return ECMC_EINVAL;
    if (p->n < 3 || p->n > (int64_t)0x3FFFFFFF || p->n_chains < 1 || p->n_chains > p->n)
        return ECMC_EINVAL;
    if (p->undo_cap < 0 || p->undo_cap >= (1 << 24) || !(p->box > 0.0) || !(p->d > 0.0) ||
        !(p->ell > 0.0))
        return ECMC_EINVAL;
    int nc = 0, C = 4;
    if (pick_cells(p, &nc, &C)) return ECMC_EINVAL;
    const int64_t graph_bytes = graph_plan_bytes(p, nc);
    if (graph_bytes < 0) return ECMC_EINVAL;
    // (with the scratch of ecmc_positions, allocated by its first call)
    *bytes = graph_bytes + export_layout(p->n, nullptr);
    return ECMC_OK;
}

extern "C" int ecmc_create(const ecmc_params *p, const double *x, const double *y,
                           const int32_t *active, void *stream, ecmc_ctx **out) {
    ecmc_ctx *ctx = nullptr;
    if (!p || !x || !y || !active || !out) return fail(nullptr, ECMC_EINVAL, "null argument");
    *out = nullptr;
    if (p->n < 3 || p->n > (int64_t)0x3FFFFFFF) return fail(nullptr, ECMC_EINVAL, "n out of range");
    if (p->n_chains < 1 || p->n_chains > p->n) return fail(nullptr, ECMC_EINVAL, "n_chains out of range");
    if (p->windows < 0 || p->windows > 4096) return fail(nullptr, ECMC_EINVAL, "windows out of range");
    if (p->undo_cap < 0 || p->undo_cap >= (1 << 24))
        return fail(nullptr, ECMC_EINVAL, "undo_cap out of range (0 .. 2^24 - 1)");
    if (!(p->d > 0.0) || !(p->ell > 0.0) || !(p->box > 0.0) || !std::isfinite(p->box) ||
        !std::isfinite(p->ell))
        return fail(nullptr, ECMC_EINVAL, "d, ell and box must be positive and finite");
    int nc = 0, C = 4;
    if (pick_cells(p, &nc, &C))
        return fail(nullptr, ECMC_EINVAL, "cell geometry: need nc >= 3 and d < L/nc < 1.664 d");
    if ((int64_t)nc * nc * C > (int64_t)0xFFFFFFF0)
        return fail(nullptr, ECMC_EINVAL, "too many cells");

    ctx = new (std::nothrow) ecmc_ctx();
    if (!ctx) return fail(nullptr, ECMC_ENOMEM, "host allocation");
    ctx->p = *p;
    ctx->stream = (cudaStream_t)stream;
    ctx->C = C;
    if ((p->flags & ECMC_RESTART) && (!(p->flags & ECMC_GRAPH) || p->windows > 1)) {
        delete ctx;
        return fail(nullptr, ECMC_EINVAL, "ECMC_RESTART needs ECMC_GRAPH and one claim window");
    }
    ctx->cells = (p->flags & ECMC_GRAPH) == 0;
    const int rc = create_graph(ctx, nc, x, y, active);
    if (rc) {
        ecmc_destroy(ctx);
        return rc;
    }
    *out = ctx;
    return ECMC_OK;
}

static void fold_graph_totals(ecmc_ctx *c, const GraphTotals &t, bool alone) {
    c->legs_total += t.legs;
    c->lifts_total += t.lifts;
    c->conflict_legs += t.conflict_legs;
    c->repaired += t.repaired;
    c->continued += t.continued;
    c->restarts += t.restarts;
    c->blocked += t.blocked;
    c->cwindows += t.cwindows;
    c->row_windows += t.row_windows;
    c->horizon += t.horizon;
    c->order_err += t.order_err;
    c->prof.pass1_launches += t.legs;
    c->prof.other_launches += t.legs;
    c->prof.repair_launches += t.conflict_legs;
    c->prof.pass1_liftings += t.p1_lifts;
    c->prof.repair_liftings += t.repair_lifts;
    if (alone) {
        c->device_ms += t.ms;
        c->prof.pass1_ms += t.pass1_ms;
        c->prof.repair_ms += t.repair_ms;
        c->prof.other_ms += t.other_ms;
    }
}

// Legs a launch may be asked for (its member tags count 2^24 claim windows). A
// call on cell-scan contexts for more runs in several launches.
static int32_t launch_legs(int windows) { return std::max(1, ((1 << 24) - 1) / windows); }

static int windows_of(const ecmc_ctx *c) { return c->p.windows > 0 ? c->p.windows : 1; }

// Up to max_legs legs of every context of a batch on `st`, in one persistent
// launch (cell-scan contexts: in several beyond launch_legs); per-context totals
// are folded into each context's host counters.
static int batch_run(GBatchScratch **scratch, cudaStream_t st, ecmc_ctx *const *ctxs, int R,
                     int32_t max_legs, const uint64_t *budgets, int64_t *lifts_out,
                     int32_t *legs_out, std::string &err, double *ms_out) {
    if (R < 1 || max_legs < 0) {
        err = "bad batch size or leg count";
        return ECMC_EINVAL;
    }
    for (int r = 0; r < R; ++r)
        if (!ctxs[r] || ctxs[r]->cells != ctxs[0]->cells) {
            err = "a batch holds either constraint-graph contexts or cell-scan contexts";
            return ECMC_EINVAL;
        }
    const bool cells = ctxs[0]->cells;
    for (int r = 0; r < R; ++r) {
        if (cells && (ctxs[r]->C != ctxs[0]->C || windows_of(ctxs[r]) != windows_of(ctxs[0]))) {
            err = "all contexts of a batch need the same cell slots (cell size) and windows";
            return ECMC_EINVAL;
        }
        for (int q = 0; q < r; ++q)
            if (ctxs[q] == ctxs[r]) {
                err = "a context appears twice in a batch";
                return ECMC_EINVAL;
            }
    }
    unsigned long long wait_ns = BARRIER_TIMEOUT_NS;
    for (int r = 0; r < R; ++r) {
        if (lifts_out) lifts_out[r] = 0;
        if (legs_out) legs_out[r] = 0;
        if (cells) wait_ns = std::min(wait_ns, ctxs[r]->wait_ns);
    }
    const int32_t chunk = cells ? launch_legs(windows_of(ctxs[0])) : max_legs;
    std::vector<int64_t> lifts(R, 0);
    std::vector<int> live(R);
    for (int r = 0; r < R; ++r) live[r] = r;
    int32_t done = 0;
    do {
        const int32_t now = std::min(max_legs - done, chunk);
        std::vector<GraphCtx *> gs;
        std::vector<uint64_t> left;
        for (int r : live) {
            gs.push_back(ctxs[r]->graph);
            left.push_back(budgets && budgets[r] ? budgets[r] - (uint64_t)lifts[r] : 0);
        }
        std::vector<GraphTotals> tots(live.size());
        std::vector<int32_t> got(live.size(), 0);
        double ms = 0.0;
        const int rc = graph_batch_run(scratch, gs.data(), (int)live.size(), now, left.data(), st,
                                       tots.data(), got.data(), &ms, err, wait_ns);
        if (ms_out) *ms_out += ms;
        std::vector<int> next;
        for (size_t q = 0; q < live.size(); ++q) {
            const int r = live[q];
            fold_graph_totals(ctxs[r], tots[q], R == 1);
            lifts[r] += tots[q].lifts;
            if (lifts_out) lifts_out[r] = lifts[r];
            if (legs_out) legs_out[r] += got[q];
            if (got[q] == now && !(budgets && budgets[r] && (uint64_t)lifts[r] >= budgets[r]))
                next.push_back(r);
        }
        if (rc) return rc;
        live = next;
        done += now;
    } while (done < max_legs && !live.empty());
    return 0;
}

extern "C" int ecmc_run_to_breakpoint(ecmc_ctx *ctx, int32_t n_legs, uint64_t event_budget,
                                      uint8_t *leg_flags_out, int32_t *legs_done) {
    if (!ctx) return ECMC_EINVAL;
    if (n_legs < 0) return fail(ctx, ECMC_EINVAL, "n_legs < 0");
    if (legs_done) *legs_done = 0;
    if (n_legs == 0) return ECMC_OK;
    const unsigned long long wait_ns = ctx->cells ? ctx->wait_ns : BARRIER_TIMEOUT_NS;
    const int32_t chunk = ctx->cells ? launch_legs(windows_of(ctx)) : n_legs;
    std::string err;
    int rc = 0;
    int32_t done = 0;
    uint64_t lifts = 0;
    while (!rc && done < n_legs) {
        const int32_t now = std::min(n_legs - done, chunk);
        GraphTotals t;
        int32_t legs = 0;
        rc = graph_run(ctx->graph, now, event_budget ? event_budget - lifts : 0,
                       leg_flags_out ? leg_flags_out + done : nullptr, &legs, &t, err, wait_ns);
        fold_graph_totals(ctx, t, true);
        done += legs;
        lifts += (uint64_t)t.lifts;
        if (legs < now || (event_budget && lifts >= event_budget)) break;
    }
    if (legs_done) *legs_done = done;
    return rc ? fail(ctx, rc, err) : ECMC_OK;
}

struct ecmc_batch {
    GBatchScratch *scratch = nullptr;
    cudaStream_t stream = nullptr;
    std::string err;
    double device_ms = 0.0;
};

extern "C" int ecmc_batch_create(void *stream, ecmc_batch **out) {
    if (!out) return ECMC_EINVAL;
    ecmc_batch *b = new (std::nothrow) ecmc_batch();
    if (!b) return ECMC_ENOMEM;
    b->stream = (cudaStream_t)stream;
    *out = b;
    return ECMC_OK;
}

extern "C" int ecmc_batch_run(ecmc_batch *b, ecmc_ctx *const *ctxs, int32_t n_ctx,
                              int32_t max_legs, const uint64_t *budgets, int64_t *liftings_out,
                              int32_t *legs_out, double *device_ms_out) {
    if (!b || !ctxs || n_ctx < 1) return ECMC_EINVAL;
    double ms = 0.0;
    const int rc = batch_run(&b->scratch, b->stream, ctxs, n_ctx, max_legs, budgets, liftings_out,
                             legs_out, b->err, &ms);
    b->device_ms += ms;
    if (device_ms_out) *device_ms_out = ms;
    return rc;
}

extern "C" const char *ecmc_batch_last_error(const ecmc_batch *b) {
    return b ? b->err.c_str() : "";
}

extern "C" void ecmc_batch_destroy(ecmc_batch *b) {
    if (!b) return;
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) (void)cudaGetLastError();
    graph_batch_free(b->scratch);
    delete b;
}

extern "C" int ecmc_positions(ecmc_ctx *ctx, double *x, double *y, double *t, int32_t *active) {
    if (!ctx) return ECMC_EINVAL;
    cudaStream_t st = ctx->stream;
    const size_t n = (size_t)ctx->p.n, k = (size_t)ctx->p.n_chains;
    if (!ctx->exp) {  // device scratch, allocated at the first call and kept
        const int64_t total = export_layout(ctx->p.n, nullptr);
        const int e = dm_alloc_t(&ctx->exp, (size_t)total);
        if (e != 0) {
            ctx->exp = nullptr;
            return fail(ctx, ECMC_ENOMEM,
                        std::string("cudaMalloc: ") + cudaGetErrorString((cudaError_t)e));
        }
        ctx->exp_bytes = export_layout(ctx->p.n, ctx);
    }
    // (in a transposed context the stored x is the caller's y)
    double *const ox = ctx->direction ? y : x, *const oy = ctx->direction ? x : y;
    const double *sy = nullptr;
    const int32_t *sa = nullptr;
    if (graph_export(ctx->graph, ox ? ctx->exp_x : nullptr, t ? ctx->exp_t : nullptr, &sy, &sa) != 0)
        return fail(ctx, ECMC_ECUDA, "positions (graph)");
    cudaError_t e = cudaSuccess;
    if (ox) e = cudaMemcpyAsync(ox, ctx->exp_x, n * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && oy) e = cudaMemcpyAsync(oy, sy, n * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && t) e = cudaMemcpyAsync(t, ctx->exp_t, n * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && active)
        e = cudaMemcpyAsync(active, sa, k * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess)
        return fail(ctx, ECMC_ECUDA, std::string("positions: ") + cudaGetErrorString(e));
    return ECMC_OK;
}

extern "C" int ecmc_set_direction(ecmc_ctx *ctx, int32_t direction) {
    if (!ctx) return ECMC_EINVAL;
    if (direction != 0 && direction != 1)
        return fail(ctx, ECMC_EINVAL, "direction must be 0 (+x) or 1 (+y)");
    if (direction == ctx->direction) return ECMC_OK;
    std::string err;
    const int rc = graph_transpose(ctx->graph, err);
    if (rc) return fail(ctx, rc, "set_direction: " + err);
    ctx->direction = direction;
    return ECMC_OK;
}

extern "C" int ecmc_set_wait_limit(ecmc_ctx *ctx, uint64_t ns) {
    if (!ctx) return ECMC_EINVAL;
    if (ns == 0 || ns > BARRIER_TIMEOUT_NS) return fail(ctx, ECMC_EINVAL, "wait limit out of range");
    ctx->wait_ns = ns;
    return ECMC_OK;
}

extern "C" int ecmc_stats(ecmc_ctx *ctx, ecmc_stats_t *out) {
    if (!ctx || !out) return ECMC_EINVAL;
    out->liftings = ctx->lifts_total;
    out->legs = ctx->legs_total;
    out->conflict_legs = ctx->conflict_legs;
    out->repaired_chains = ctx->repaired;
    out->continued_chains = ctx->continued;
    out->restarts = ctx->restarts;
    out->row_windows = ctx->row_windows;
    out->blocked_chains = ctx->blocked;
    out->conflict_windows = ctx->cwindows;
    out->device_bytes = graph_device_bytes(ctx->graph) + ctx->exp_bytes;
    out->horizon_asserts = ctx->horizon;
    out->order_errors = ctx->order_err;
    out->device_ms = ctx->device_ms;
    return ECMC_OK;
}

extern "C" int ecmc_profile(ecmc_ctx *ctx, ecmc_profile_t *out) {
    if (!ctx || !out) return ECMC_EINVAL;
    *out = ctx->prof;
    return ECMC_OK;
}

extern "C" int ecmc_graph_arrows(ecmc_ctx *ctx, int32_t *a, double *b) {
    if (!ctx) return ECMC_EINVAL;
    if (ctx->cells) return fail(ctx, ECMC_EINVAL, "not a constraint-graph context");
    std::string err;
    const int rc = graph_arrows(ctx->graph, a, b, err);
    return rc ? fail(ctx, rc, err) : ECMC_OK;
}

extern "C" int ecmc_liftings(ecmc_ctx *ctx, ecmc_lift_t *buf, int64_t cap, int64_t *n_out) {
    if (!ctx || !n_out) return ECMC_EINVAL;
    std::string err;
    const int rc = graph_liftings(ctx->graph, buf, cap, n_out, err);
    return rc ? fail(ctx, rc, err) : ECMC_OK;
}

extern "C" void ecmc_destroy(ecmc_ctx *ctx) {
    if (!ctx) return;
    // (every call on the context has synchronised its stream before
    // returning; this one makes sure before its blocks go to the cache)
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) (void)cudaGetLastError();
    graph_destroy(ctx->graph);
    dm_free(ctx->exp);
    delete ctx;
}

extern "C" const char *ecmc_last_error(const ecmc_ctx *ctx) {
    return ctx ? ctx->err.c_str() : g_create_err.c_str();
}

// ------------------------------------------ one leg without any allocation
//
// For callers that cannot allocate device memory: code that runs while a
// framework owns the whole device heap through its own caching allocator
// (a cudaMalloc would fail or fragment that pool), real-time loops that must
// not pay allocation latency, and plug-ins that are only handed pointers.
// All working memory of the leg comes from one file-scope device array of
// fixed size; the caller passes only inputs and outputs.

namespace {

// The sizes a call takes: those whose arrays, counted as below (33 bytes a cell
// slot, 24.7 KB a chain), are at most ECMC_NOALLOC_SCRATCH_MIB. What a leg needs
// here is more a disk and less a slot; over all sizes of that count whose disks
// do not overlap it is at most 48.6 MiB.
constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)52 << 20;
constexpr int NOALLOC_CAP = ECMC_NOALLOC_RECORDS;  // event records per chain per leg
constexpr int NOALLOC_MAX_DEVICES = 64;

size_t noalloc_count(size_t nslot, size_t ncell, size_t n, size_t k) {
    size_t off = 0;
    auto take = [&](size_t bytes) { off = ((off + 255) & ~(size_t)255) + bytes; };
    for (int q = 0; q < 3; ++q) take(nslot * 8);
    for (int q = 0; q < 2; ++q) take(nslot * 4);
    take(ncell * 4);
    take(n * 4);
    for (int q = 0; q < 8; ++q) take(k * 8);
    for (int q = 0; q < 22; ++q) take(k * 4);
    take((k + 1) * 4);
    for (int q = 0; q < 3; ++q) take(152);
    take(k * (size_t)NOALLOC_CAP * 96);
    return off;
}

// Shared by every call on a device and kept until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

static std::mutex g_noalloc_mu;
static void *g_noalloc_ptr[NOALLOC_MAX_DEVICES];

// Device address of the scratch array for the current device, looked up once.
static int noalloc_scratch(unsigned char **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return ECMC_ECUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return ECMC_ECUDA;
        }
        g_noalloc_ptr[dev] = p;
    }
    *out = (unsigned char *)g_noalloc_ptr[dev];
    return ECMC_OK;
}

}  // namespace

extern "C" int ecmc_leg_noalloc(int64_t n, double box, double d, double ell, int32_t n_chains,
                                int32_t cells_per_side, double *x, const double *y,
                                int32_t *active, double *t_out, void *stream, uint8_t *flag_out,
                                int64_t *lifts_out) {
    if (!x || !y || !active) return ECMC_EINVAL;
    if (n < 3 || n > (int64_t)0x3FFFFFFF || n_chains < 1 || n_chains > n) return ECMC_EINVAL;
    if (!(d > 0.0) || !(ell > 0.0) || !(box > 0.0) || !std::isfinite(box) || !std::isfinite(ell))
        return ECMC_EINVAL;
    ecmc_params p;
    memset(&p, 0, sizeof p);
    p.n = n;
    p.box = box;
    p.d = d;
    p.ell = ell;
    p.n_chains = n_chains;
    p.cells_per_side = cells_per_side;
    p.undo_cap = NOALLOC_CAP;
    int nc = 0, C = 4;
    if (pick_cells(&p, &nc, &C)) return ECMC_EINVAL;
    const size_t ncell = (size_t)nc * nc, nslot = ncell * C;
    // sizes beyond the count are rejected before any device work
    if (noalloc_count(nslot, ncell, (size_t)n, (size_t)n_chains) >
        ((size_t)ECMC_NOALLOC_SCRATCH_MIB << 20))
        return ECMC_EINVAL;
    unsigned char *base = nullptr;
    const int rc = noalloc_scratch(&base);
    if (rc) return rc;
    std::string err;
    if (graph_leg_bytes(&p, nc) > NOALLOC_SCRATCH_BYTES) {
        // more disks than the cells can hold apart: the inputs' own faults, or
        // an overfull cell
        cudaStream_t st = (cudaStream_t)stream;
        unsigned long long bad[2] = {0ull, 0ull};
        unsigned long long *const d_bad = (unsigned long long *)base;
        if (cudaMemsetAsync(base, 0, 256 + (size_t)n * 4, st) != cudaSuccess) {
            (void)cudaGetLastError();
            return ECMC_ECUDA;
        }
        graph_check_inputs(x, y, active, n, n_chains, box, (uint32_t *)(base + 256), d_bad,
                           d_bad + 1, st);
        if (cudaMemcpyAsync(bad, d_bad, sizeof bad, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            (void)cudaGetLastError();
            return ECMC_ECUDA;
        }
        return bad[0] || bad[1] ? ECMC_EINVAL : ECMC_ECAPACITY;
    }
    return graph_leg(&p, nc, base, x, y, active, t_out, (cudaStream_t)stream, flag_out, lifts_out,
                     err);
}
