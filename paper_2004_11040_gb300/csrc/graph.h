// graph.h -- internal interface between the C ABI (ecmc.cu) and the
// engine of the legs (graph.cu). Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "ecmc.h"

struct GraphCtx;

// Totals of one graph_run call.
struct GraphTotals {
    int64_t legs, lifts, conflict_legs, repaired, continued, horizon, order_err, p1_lifts,
        repair_lifts, restarts, blocked, cwindows, row_windows;
    double ms, pass1_ms, repair_ms, other_ms;
};

// A context on device inputs x, y (n each) and active (k), which are checked here
// and which the work it queues on the stream reads; nc cells per side. With
// ECMC_GRAPH the conflict flag is on the disks read, otherwise on the cells
// scanned.
int graph_create(const ecmc_params *p, int nc, const double *x, const double *y,
                 const int32_t *active, cudaStream_t st, GraphCtx **out, std::string &err);
int graph_run(GraphCtx *g, int32_t n_legs, uint64_t budget, uint8_t *flags_host,
              int32_t *legs_done, GraphTotals *tot, std::string &err,
              unsigned long long wait_ns);
// x and t (device, each may be null) filled on the context's stream; *y and
// *active point to the context's own arrays.
int graph_export(GraphCtx *g, double *x, double *t, const double **y, const int32_t **active);
// Exchanges x and y of every disk (the next legs move along the other axis),
// clears the local times and rebuilds the graph.
int graph_transpose(GraphCtx *g, std::string &err);
// Host copies of the arrows (3 per disk, -1: none) and their b_ij.
int graph_arrows(GraphCtx *g, int32_t *a, double *b, std::string &err);
int graph_liftings(GraphCtx *g, ecmc_lift_t *buf, int64_t cap, int64_t *n_out,
                   std::string &err);
void graph_destroy(GraphCtx *g);
// Batches of graph contexts: one persistent launch advances n contexts (same
// claim windows, no restart mode), each to max_legs legs or its liftings
// budget (budgets may be null; 0: none), exactly as graph_run would. The
// scratch (launch tables) is kept by the caller between calls and freed with
// graph_batch_free. tots[r] and legs_out[r] (may be null) receive each
// context's totals; *ms_out the launch's device time. wait_ns bounds every
// device wait of the launch.
struct GBatchScratch;
int graph_batch_run(GBatchScratch **scratch, GraphCtx *const *gs, int32_t n, int32_t max_legs,
                    const uint64_t *budgets, cudaStream_t st, GraphTotals *tots,
                    int32_t *legs_out, double *ms_out, std::string &err,
                    unsigned long long wait_ns);
void graph_batch_free(GBatchScratch *scratch);
// Device memory held by the context (bytes).
int64_t graph_device_bytes(const GraphCtx *g);
// What graph_create(p, nc, ...) would hold, without allocating (-1: error).
int64_t graph_plan_bytes(const ecmc_params *p, int nc);
// One leg of a cell-scan system in given device memory (graph_leg_bytes of it,
// 256-byte aligned), nothing allocated; inputs as in ecmc_leg_noalloc.
size_t graph_leg_bytes(const ecmc_params *p, int nc);
int graph_leg(const ecmc_params *p, int nc, unsigned char *base, double *x, const double *y,
              int32_t *active, double *t_out, cudaStream_t st, uint8_t *flag, int64_t *lifts,
              std::string &err);
// Counts coordinates outside [0, L) in *bad_xy (not with x null) and active ids that repeat or
// lie outside [0, n) in *bad_id (seen: n words of zero).
void graph_check_inputs(const double *x, const double *y, const int32_t *active, int64_t n, int k,
                        double L, uint32_t *seen, unsigned long long *bad_xy,
                        unsigned long long *bad_id, cudaStream_t st);
