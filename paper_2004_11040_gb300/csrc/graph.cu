// graph.cu -- the legs of libecmc. The liftings of a chain are found through the
// arrows of the constraint graph G(3) of Sec. 3.1; contexts differ in the
// conflict flag, which is on the disks a chain reads (ECMC_GRAPH) or on the
// cells that the scans of a cell search would cover.
//
// For v = (1, 0) the arrows of disk i are, in each of three corridors of
// dy = y_j - y_i (minimum image) -- centre |dy| < d/2, upper d/2 <= dy < d,
// lower -d < dy <= -d/2 -- the disk of least time of flight (tau, j), if any.
// Disks closer than d in y cannot pass one another while v holds, so the
// arrows stay valid across breakpoints (Sec. 3.1) and a step reads at most
// three target disks; b_ij = sqrt(d^2 - dy^2) is fixed with the arrow and
// stored beside it, so the step does no square root.
//
// Layout: one 64-byte record per disk (x, local time, owner word, three arrows
// and their b, claim word); y in an array of its own (it never changes along
// +x).
//
// Conflicts. Every chain first runs alone from the window's start state, which
// nothing changes meanwhile (g_spec_chain); a chain then publishes its events
// up to the first one on a disk that another chain's run reaches earlier
// (g_resolve_chain). The leg's flag is 1 iff the disks that two chains read,
// each run alone, overlap. Chains that were cut are continued one after
// another where Eq. 2 allows it, else rolled back to the earliest time one of
// them stopped and replayed in global event-time order (Alg. 2), one warp per
// conflict component.
//
// A frame whose cell rows are out of reach of each other (a lattice start on
// cells aligned with it) is a set of rings, on which runs and continuations
// are stretches of consecutive disks (frames of rings, below).
//
// All FP64 arithmetic uses explicit round-to-nearest intrinsics (the file is
// compiled with -fmad=false) so that results are reproducible bit for bit.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "devmem.h"
#include "graph.h"

namespace {

// chains are numbered by the owner word's 30 bits
constexpr int MAX_CHAINS = (int)OWN_CHAIN;

struct __align__(64) GDisk {
    double x, t;               // position along the motion; local time (leg-relative)
    uint32_t own;              // owner word: active / stalled + chain, or static + the leg
                               // (stamp) in which t was written (t is 0 in any other leg)
    uint32_t a[3];             // arrows: centre, upper, lower corridor (NONE: empty)
    unsigned long long claim;  // pass epoch << 32 | chain + 1 holding the disk in that pass
    double b[3];               // b_ij = sqrt(d^2 - dy^2) of each arrow
};
static_assert(sizeof(GDisk) == 64, "one disk record is one 64-byte line");

// One event of a chain: enough to undo it exactly, and the lifting (Eq. 1).
struct __align__(16) GEv {
    uint32_t i, j, seq, pad;  // moved disk, target (NONE: stall), application order
    double x_old;             // x of i before the move
    double ti_old, tj_old;    // local times of i and j before the event
    double t, tau, xi, xj;    // event time (= new t_j), time of flight, x_i at contact, x_j
    double d_after;           // remaining chain length after the event
};
static_assert(sizeof(GEv) == 80, "a record is written as five 16-byte words");

// What a chain's run alone in the parallel pass left.
struct __align__(16) GSpec {
    int32_t n, touch;     // events; disks touched
    int32_t end, partner; // SP_*; the chain met
    double tc, D;
    uint32_t ci;
    int32_t cut;          // events that may be published (strict: a disk in reach)
    int32_t pad[2];
};

struct GDev {
    int64_t n;
    int k, cap, windows, nc;
    double L, d, ell;
    GDisk *g;   // [n]
    double *y;  // [n]
    // parallel pass: per disk the least touch key (time << 32 | chain) of the
    // chains whose run alone touches it, ~0 untouched; per chain the touched
    // disks of its run (entry e of chain c at e * k + c). With claim windows there
    // are two sets of keys, [2n], used in turn (keys: the first; key: the
    // window's, in the warp's copy in shared memory)
    unsigned long long *key, *keys;
    uint32_t *path;        // [(cap + 2) * k]
    unsigned long long *fl;  // flag words, epoch << 32 | chain + 1: per disk read, or
                             // per cell scanned
    // a cell-scan context (cells != 0: its flag is on cells): the stop rule of
    // the scan, and per entry of path what its step's scan needs -- the active
    // disk's x and the least of D and its best time of flight, and its cell
    int cells;
    uint32_t epoch0;       // epoch of the launch's first pass, less one
    double inv_a;
    StopK sk;
    double2 *pxt;         // [(cap + 2) * k]
    uint32_t *pcell;      // [(cap + 2) * k]
    // a frame of rings (ring != 0): the disks ring after ring, each in the order
    // of x; every disk's place there, its ring's first place and length, its row
    int open;  // a launch with open arrows
    int ring;
    uint32_t *rid;  // [n]
    uint4 *pos;     // [n]
    GSpec *sp;             // [k] the run alone of each chain, for the resolve
    uint32_t stamp0;       // stamp of the launch's first leg, less one
    uint32_t stamp;        // stamp of the leg (the warp's copy in shared memory)
    // per chain
    uint32_t *ci, *ci0;  // active disk now / at the leg start
    double *D, *tc;
    int32_t *status, *partner, *nrec, *nlift;
    GEv *rec;  // [k * cap]
    // pending events of the replay, and the arrows they were computed from
    double *ev_T, *ev_tau, *ev_xj, *ev_tj;
    uint32_t *ev_j, *ev_a;  // ev_a: [4k]
    int32_t *ev_lift;
    // conflict components (names as the union-find of common.cuh expects)
    double *vt;
    int32_t *uf, *fin, *comp_of, *abort_to, *comp_cnt, *comp_off, *comp_root, *comp_mem, *ctl;
    // the trees of the union-find while the pass builds them: a root's last
    // hooked child, the child hooked before it, and the pass that took the root
    int32_t *child, *sib, *taken;
    uint64_t *memb;   // (pass of the launch, round) << 32 | root of the component listing the chain
    int restart;      // conflicts by restart strategy 2 (Sec. 3.4) instead of local repair
    int strict;       // the pass claims every disk a step reads, not only those it touches
    double *tstar;    // [1] restart mode: the earliest stop time of a pass
    unsigned long long *lc;      // [2 LC_N], by leg parity
    unsigned long long *tc_cnt;  // [TC_N]
    ecmc_lift_t *log;
    int64_t log_cap;
    int log_on;
    double *dbg;  // [16] first failed internal check
};
// (a warp copies its system's description in rounds of 128 bytes, one after another;
// a fifth cost batches 2%)
static_assert(sizeof(GDev) <= 512, "four rounds");

// Record e of chain c, stored by event index, then chain (the first events of
// a leg of all chains lie in one dense block).
__device__ __forceinline__ GEv *grec_at(const GDev &s, int c, int e) {
    return s.rec + (size_t)e * (size_t)s.k + (size_t)c;
}

__device__ __forceinline__ uint32_t *gpath_at(const GDev &s, int c, int e) {
    return s.path + (size_t)e * (size_t)s.k + (size_t)c;
}

__device__ void gdiag(const GDev &s, int kind, double a, double b, double c, double d,
                      double e, double f) {
    if (!s.dbg) return;
    if (atomicCAS((unsigned long long *)s.dbg, 0ull,
                  (unsigned long long)__double_as_longlong((double)kind)) != 0ull)
        return;
    s.dbg[1] = a;
    s.dbg[2] = b;
    s.dbg[3] = c;
    s.dbg[4] = d;
    s.dbg[5] = e;
    s.dbg[6] = f;
}

// A coordinate as given, -0.0 taken as 0: the build ranks coordinates by their
// bits, where -0.0 lies above every other number. (On the integer pipe; the
// frames' own x and y never are -0.0 again.)
__device__ __forceinline__ double coord(double v) {
    return dbits(v) == 0x8000000000000000ull ? 0.0 : v;
}

__device__ __forceinline__ int cell_coord(double v, double inv_a, int nc) {
    int c = __double2int_rz(__dmul_rn(v, inv_a));
    if (c >= nc) c = nc - 1;
    if (c < 0) c = 0;
    return c;
}

// A disk's cell, as the cell scan keeps it.
__device__ __forceinline__ uint32_t cell_of(const GDev &s, double x, double y) {
    return (uint32_t)cell_coord(y, s.inv_a, s.nc) * (uint32_t)s.nc +
           (uint32_t)cell_coord(x, s.inv_a, s.nc);
}

__device__ __forceinline__ double wrap_add(double x, double dx, double L) {
    double r = __dadd_rn(x, dx);
    if (dbits(r) >= dbits(L)) r = __dsub_rn(r, L);  // r >= 0
    return r;
}

// The owner word says static; the local time of a static disk in this leg.
__device__ __forceinline__ bool g_static(uint32_t own) { return own < OWN_ACTIVE; }
__device__ __forceinline__ double g_time(uint32_t own, double t, uint32_t stamp) {
    return own >= OWN_ACTIVE || own == stamp ? t : 0.0;
}

// b of an arrow not searched to its end (a: NONE): minus the place before which
// there is none (the sign bit also of 0).
constexpr unsigned long long SIGN = 1ull << 63;
__device__ __forceinline__ bool g_open(uint32_t a, double b) {
    return a == NONE && (dbits(b) & SIGN) != 0ull;
}
__device__ __forceinline__ double g_unsigned(double b) {
    return __longlong_as_double((long long)(dbits(b) & ~SIGN));
}

__device__ __forceinline__ double shfl_f64(double v, int src) {
    return __shfl_sync(FULL, v, src);
}

// ------------------------------------------------------------ graph build

// What a build finds: disks without a slot in their cell, rows that are no rings
// (or none asked), disks left to k_gb_far, and of unchecked inputs coordinates
// outside [0, L) and bad ids.
struct BuildCounts {
    unsigned long long full, mixed, listed, bad_xy, bad_id;
    unsigned long long open;  // disks whose record has an open arrow
};

// Inputs and scratch of a build: a cell list of the disks (in any of a cell's
// slots), their FP32 coordinates per slot relative to the cell's corner (an
// error of 1e-7 d whatever the box), and one bit per y bin of width d/128 that
// holds a disk.
struct GBuild {
    int64_t n;
    int nc, nb;
    double L, d, d2, a, inv_a;
    float Lf, df, half_f, af, wf, inv_wf;
    float del;           // a 2^-20: bound on the FP32 error of a difference of
                         // coordinates of neighbouring cells
    const double *x, *y;
    int check;                   // count coordinates outside [0, L)
    double *start;               // [n] x of every disk, kept (arrows may stay open), or null
    uint32_t *scid;        // [nc*nc*C] disk per slot, EMPTY
    float2 *cxy;           // [nc*nc*C] FP32 coordinates within the cell, NaN in an empty slot
    uint32_t *far;         // [2n] slots of the disks left to k_gb_far, and from [n] on
                           // of those with open arrows
    int nblk;              // blocks of FAR_COLS columns in a row
    float4 *ylim;          // [nc*nblk] least and largest y (within the cell row) per block
                           // in the row's lower half, and in its upper one
    uint32_t *bits;        // [nb / 32 + 1]
    GDisk *g;
    double *yout;             // [n] or null: each disk's y
    BuildCounts *count;
};

// A monotone map of y to its bin, the same wherever bins are set or asked for.
__device__ __forceinline__ int y_bin(const GBuild &b, float y) {
    const int q = __float2int_rz(__fmul_rn(y, b.inv_wf));
    return min(max(q, 0), b.nb - 1);
}

__device__ __forceinline__ void set_bin(const GBuild &b, float y) {
    const int q = y_bin(b, y);
    const uint32_t m = 1u << (q & 31);
    // (most bins are set already: an atomic per disk on a lattice's few bins
    // took 70 of the 400 us of creation at 2^20 disks)
    if (!(*(volatile uint32_t *)(b.bits + (q >> 5)) & m)) atomicOr(b.bits + (q >> 5), m);
}

// Coordinates relative to the corner of cell (row, col); an FP32 x of -0 or a
// little less (x on the edge) counts as 0, so that only an empty slot is NaN.
__device__ __forceinline__ float2 in_cell(const GBuild &b, double x, double y, int row, int col) {
    return make_float2(fmaxf(d2f_trunc(__dsub_rn(x, __dmul_rn((double)col, b.a))), 0.f),
                       d2f_trunc(__dsub_rn(y, __dmul_rn((double)row, b.a))));
}

template <int C>
__global__ void k_gb_cells(GBuild b) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= b.n) return;
    const double x = coord(b.x[q]), y = coord(b.y[q]);
    if (b.check && !(x >= 0.0 && x < b.L && y >= 0.0 && y < b.L))
        atomicAdd(&b.count->bad_xy, 1ull);
    const int row = cell_coord(y, b.inv_a, b.nc), col = cell_coord(x, b.inv_a, b.nc);
    const uint32_t cell = (uint32_t)row * (uint32_t)b.nc + (uint32_t)col;
    const float2 v = in_cell(b, x, y, row, col);
    set_bin(b, d2f_trunc(y));
    for (int sl = 0; sl < C; ++sl) {
        const uint32_t loc = cell * C + sl;
        if (atomicCAS(b.scid + loc, EMPTY, (uint32_t)q) == EMPTY) {
            b.cxy[loc] = v;
            return;
        }
    }
    atomicAdd(&b.count->full, 1ull);
}

// Does a bin that meets [lo, hi) (periodic, hi - lo < L) hold a disk? The
// callers' one-bin margin (d/128) is far above the FP32 rounding of y, lo, hi.
__device__ bool band_any(const GBuild &b, float lo, float hi) {
    if (lo < 0.f) {
        lo = __fadd_rn(lo, b.Lf);
        hi = __fadd_rn(hi, b.Lf);
    } else if (lo >= b.Lf) {
        lo = __fsub_rn(lo, b.Lf);
        hi = __fsub_rn(hi, b.Lf);
    }
    auto any = [&](int q0, int q1) {
        uint32_t r = 0u;
        for (int w = q0 >> 5; w <= q1 >> 5; ++w) {
            uint32_t m = ~0u;
            if (w == q0 >> 5) m &= ~0u << (q0 & 31);
            if (w == q1 >> 5) m &= ~0u >> (31 - (q1 & 31));
            r |= b.bits[w] & m;
        }
        return r != 0u;
    };
    const int q0 = y_bin(b, lo);
    if (hi <= b.Lf) return any(q0, y_bin(b, hi));
    return any(q0, b.nb - 1) || any(0, y_bin(b, __fsub_rn(hi, b.Lf)));
}

// One corridor's best so far: the slot, and bounds of its time of flight.
struct GBest {
    float lo, hi;
    uint32_t loc;
};

// (approximate to 2^-22; the slop below is far above that)
__device__ __forceinline__ float sqrt_f(float v) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// The corridor of the disk at v (in its cell, rr rows and m columns on) seen
// from xi, yi (-1: none; EDGE: FP32 cannot tell which, or whether none; NEXT: nor
// whether it is ahead or a lap away) and, but for NEXT, bounds of its time of
// flight.
enum { EDGE = 3, NEXT = 4 };
__device__ __forceinline__ int corridor_f(const GBuild &b, float xi, float yi, int rr, int m,
                                          float2 v, float &lo, float &hi) {
    const float dy = (float)rr * b.af + (v.y - yi);
    const float ay = fabsf(dy);
    if (ay > b.df + b.del) return -1;
    float dx = (float)m * b.af + (v.x - xi);
    float del = b.del + (float)m * (0.25f * b.del);
    if (fabsf(dx) < del) return NEXT;
    if (dx < 0.f) {  // behind in its own column: nearly a lap ahead
        dx += b.Lf;
        del += b.Lf * 0x1p-21f;
    }
    const float d2 = b.df * b.df, an = fmaxf(ay - b.del, 0.f), af = ay + b.del;
    // (2^-19 d covers the roundings of these lines)
    const float slop = b.df * 0x1p-19f + del;
    hi = dx - sqrt_f(fmaxf(d2 - af * af - d2 * 0x1p-21f, 0.f)) + slop;
    lo = dx - sqrt_f(fmaxf(d2 - an * an, 0.f) + d2 * 0x1p-21f) - slop;
    if (ay > b.df - b.del || fabsf(ay - b.half_f) < b.del) return EDGE;
    return ay < b.half_f ? 0 : dy > 0.f ? 1 : 2;
}

// The corridor (-1: none) and the time of flight by their definition, in FP64.
struct GFlight {
    int kc;
    double tau;
};
__device__ __noinline__ GFlight flight_exact(double L, double d, double d2, double xi, double yi,
                                             double xj, double yj) {
    GFlight f = {-1, 0.0};
    const double dy = __dsub_rn(yj, yi);
    double ay = fabs(dy);
    const double la = __dsub_rn(L, ay);
    const bool flip = dbits(la) < dbits(ay);
    if (flip) ay = la;
    if (dbits(ay) >= dbits(d)) return f;
    f.kc = 0;
    if (dbits(ay) >= dbits(__dmul_rn(0.5, d))) {
        bool up = !dneg(dy) && dbits(dy) != 0ull;
        if (flip) up = !up;
        f.kc = up ? 1 : 2;
    }
    double dx = __dsub_rn(xj, xi);
    if (dneg(dx)) dx = __dadd_rn(dx, L);
    f.tau = __dsub_rn(dx, __dsqrt_rn(__dsub_rn(d2, __dmul_rn(ay, ay))));
    if (dneg(f.tau)) f.tau = 0.0;
    return f;
}

// The candidate of a corridor takes the place of the best or not; true where
// the bounds cannot tell.
__device__ __forceinline__ bool take_best(GBest &best, float lo, float hi, uint32_t loc) {
    if (lo > best.hi) return false;
    const bool doubt = best.loc != NONE && !(hi < best.lo);
    if (hi < best.hi) {
        best.hi = hi;
        best.loc = loc;
    }
    best.lo = doubt ? fminf(best.lo, lo) : lo;
    return doubt;
}

__device__ __forceinline__ double gb_x(const GBuild &b, uint32_t loc, uint32_t id) {
    return coord(b.x[id]);
}
__device__ __forceinline__ double gb_y(const GBuild &b, uint32_t loc, uint32_t id) {
    return coord(b.y[id]);
}

// The FP32 coordinates of a cell's slots, all loads at once.
template <int C>
struct GCell {
    float2 v[C];
};
template <int C>
__device__ __forceinline__ GCell<C> load_cell(const GBuild &b, uint32_t c0) {
    GCell<C> r;
    const float4 *p = reinterpret_cast<const float4 *>(b.cxy + c0);
#pragma unroll
    for (int q = 0; q < C / 2; ++q) {
        const float4 u = p[q];
        r.v[2 * q] = make_float2(u.x, u.y);
        r.v[2 * q + 1] = make_float2(u.z, u.w);
    }
    return r;
}

// The arrow in corridor q of a disk (slot loc, FP32 place vi) by its definition,
// where the FP32 bounds of the nearest candidates overlap: the warp looks at the
// columns that hold disks with times of flight from lo to hi (take_best: the
// least lower bound of those that may come first, and the least upper one), and
// at the disk's own column, where one behind lies a lap ahead. The arrow's slot.
template <int C>
__device__ __noinline__ uint32_t arrow_exact(const GBuild &b, int q, uint32_t loc, float2 vi,
                                             double xi, double yi, int cxi, int cyi, float lo,
                                             float hi) {
    const int nc = b.nc, lane = threadIdx.x & 31;
    unsigned long long bt = INF_BITS;
    uint32_t bj = NONE, bl = NONE;
    // (a candidate in column m lies (m - 1) a to (m + 1) a ahead, b <= d beyond tau)
    const int m1 = min(nc - 1, (int)((hi + b.df) / b.af) + 3);
    for (int m0 = max(0, (int)(lo / b.af) - 3); m0 <= m1; m0 += 31) {
        const int m = lane == 31 ? 0 : m0 + lane;
        int col = cxi + m;
        if (col >= nc) col -= nc;
#pragma unroll 1
        for (int z = 0; z < 3; ++z) {
            int row = cyi + z - 1;
            if (row < 0) row += nc;
            if (row >= nc) row -= nc;
#pragma unroll 1
            for (int sl = 0; sl < C; ++sl) {
                const uint32_t slot =
                    m < nc ? ((uint32_t)row * (uint32_t)nc + (uint32_t)col) * C + sl : loc;
                const float2 v = b.cxy[slot];
                if (slot == loc || !(v.x >= 0.f)) continue;
                float l, h;
                const int kc = corridor_f(b, vi.x, vi.y, z - 1, m, v, l, h);
                if (!(kc >= EDGE || (kc == q && l <= hi))) continue;
                const uint32_t id = b.scid[slot];
                const GFlight f =
                    flight_exact(b.L, b.d, b.d2, xi, yi, gb_x(b, slot, id), gb_y(b, slot, id));
                const unsigned long long kt = dbits(f.tau);
                if (f.kc == q && (kt < bt || (kt == bt && id < bj))) {
                    bt = kt;
                    bj = id;
                    bl = slot;
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t2 = shfl_xor_u64(bt, o);
        const uint32_t j2 = __shfl_xor_sync(FULL, bj, o);
        const uint32_t l2 = __shfl_xor_sync(FULL, bl, o);
        if (t2 < bt || (t2 == bt && j2 < bj)) {
            bt = t2;
            bj = j2;
            bl = l2;
        }
    }
    return bl;
}

constexpr int FAR_COLS = 8, FAR_LANES = 8;
static_assert(FAR_LANES >= FAR_COLS, "a lane per column of a block");

// Least and largest y, relative to the corner of the cell row, of every block of
// FAR_COLS columns in either half of the row (a lane per cell; empty: +inf,
// -inf). Limits of a whole row would span a corridor that no disk of the row is
// in wherever two rows of disks share a row of cells.
template <int C>
__global__ void k_gb_blocks(GBuild b, const unsigned long long *searched) {
    if (*searched == 0ull) return;
    static_assert(FAR_COLS == 8, "a block is a quarter of a warp's lanes");
    const int64_t end = (int64_t)b.nc * b.nblk * FAR_COLS;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; __any_sync(FULL, q < end);
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t blk = q / FAR_COLS, row = blk / b.nblk;
        const int col = (int)(blk - row * b.nblk) * FAR_COLS + (int)(q % FAR_COLS);
        float lo[2] = {INFINITY, INFINITY}, hi[2] = {-INFINITY, -INFINITY};
        if (q < end && col < b.nc) {
            const GCell<C> cell =
                load_cell<C>(b, ((uint32_t)row * (uint32_t)b.nc + (uint32_t)col) * C);
#pragma unroll
            for (int sl = 0; sl < C; ++sl) {
                const float y = cell.v[sl].y;
                if (!(cell.v[sl].x >= 0.f)) break;
                const bool up = y > 0.5f * b.af;
                lo[0] = up ? lo[0] : fminf(lo[0], y);
                hi[0] = up ? hi[0] : fmaxf(hi[0], y);
                lo[1] = up ? fminf(lo[1], y) : lo[1];
                hi[1] = up ? fmaxf(hi[1], y) : hi[1];
            }
        }
#pragma unroll
        for (int o = FAR_COLS / 2; o > 0; o >>= 1)
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                lo[z] = fminf(lo[z], __shfl_xor_sync(FULL, lo[z], o));
                hi[z] = fmaxf(hi[z], __shfl_xor_sync(FULL, hi[z], o));
            }
        if (q < end && q % FAR_COLS == 0) b.ylim[blk] = make_float4(lo[0], hi[0], lo[1], hi[1]);
    }
}

// Arrows of G(3), and the whole record of every disk (static, time 0): one
// thread per disk. A block takes BUILD_CELLS cells of consecutive numbers and
// packs their occupied slots first, so that warps are full and neighbours read
// the same cells. The search runs in FP32: per corridor, bounds of the time of
// flight of the best candidate. FP64 is left with one b = sqrt(d^2 - dy^2) per
// arrow, all lanes at once (an FP64 instruction costs the same whatever its lane
// mask). Corridors and rows that the y bins show empty are not searched.
//
// Disks that NEAR_COLS columns do not settle, and those with candidates whose
// bounds overlap (a few in 10^5), go on a list for k_gb_far: half of them on a
// triangular lattice at eta 0.60, a tenth at 0.70, one in 500 along the other
// axis. (With the far search in this kernel it took 92 registers: 129 us on 10^6
// square-lattice disks, 108 so at 64. After 4 columns 175 + 190 us with k_gb_far
// on 10^6 triangular disks at 0.70, after 8 198 + 75.)
constexpr int BUILD_CELLS = 224;
constexpr int NEAR_COLS = 8;

// The search of one disk: its place, what may hold its arrows, the best so far.
template <int C>
struct GSearch {
    const GBuild &b;
    uint32_t loc, i;
    float2 vi;
    double xi, yi;
    int cyi, cxi, rdn, rup;
    bool play[3], row_up, row_dn;
    unsigned doubt = 0u;   // corridors with candidates whose bounds overlap
    GBest best[3];

    __device__ __forceinline__ GSearch(const GBuild &build, uint32_t slot)
        : b(build), loc(slot), i(build.scid[slot]), vi(build.cxy[slot]) {
        const int nc = b.nc;
        xi = gb_x(b, loc, i);
        yi = gb_y(b, loc, i);
        cyi = (int)((loc / C) / (uint32_t)nc);
        cxi = (int)((loc / C) % (uint32_t)nc);
        rdn = cyi == 0 ? nc - 1 : cyi - 1;
        rup = cyi == nc - 1 ? 0 : cyi + 1;
    }

    // by the y bins, nothing found yet
    __device__ __forceinline__ void begin() {
        const float yf = d2f_trunc(yi);
        // corridors that may hold a disk (one bin of margin on each side; the
        // centre one holds the disk itself)
        play[0] = true;
        play[1] = band_any(b, yf + b.half_f - b.wf, yf + b.df + b.wf);
        play[2] = band_any(b, yf - b.df - b.wf, yf - b.half_f + b.wf);
        // the rows beside that hold a disk within d (by the bins): on a lattice
        // neither does
        const float y0 = d2f_trunc(__dmul_rn((double)cyi, b.a));
        row_up = band_any(b, y0 + b.af - b.wf, yf + b.df + b.wf);
        row_dn = band_any(b, yf - b.df - b.wf, y0 + b.wf);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            best[q].lo = best[q].hi = INFINITY;
            best[q].loc = NONE;
        }
    }

    // the corridors that column m may still improve: thr(m) within the best
    __device__ __forceinline__ unsigned open_at(int m) const {
        const float thr = (float)m * b.af - vi.x - b.df - (float)(m + 4) * b.del;
        unsigned o = 0u;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (play[q] && !(thr > best[q].hi)) o |= 1u << q;
        return o;
    }

    // the disks of a cell (its first slot c0), rr rows and m columns on
    __device__ __forceinline__ void disks(const GCell<C> &cl, uint32_t c0, int rr, int m,
                                          GBest (&to)[3]) {
#pragma unroll
        for (int sl = 0; sl < C; ++sl) {
            const float2 v = cl.v[sl];
            if (!(v.x >= 0.f)) break;  // (a cell's slots fill in order)
            if (c0 + sl == loc) continue;
            float lo, hi;
            int kc = corridor_f(b, vi.x, vi.y, rr, m, v, lo, hi);
            if (kc < 0) continue;
            if (kc >= EDGE) {
                const uint32_t id = b.scid[c0 + sl];
                const GFlight f =
                    flight_exact(b.L, b.d, b.d2, xi, yi, gb_x(b, c0 + sl, id), gb_y(b, c0 + sl, id));
                if (f.kc < 0) continue;
                kc = f.kc;
                lo = d2f_trunc(f.tau);
                hi = lo + lo * 0x1p-22f + 0x1p-126f;
                lo -= lo * 0x1p-22f;
            }
            // (selects, not indexing, keep the corridors in registers)
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (q == kc && take_best(to[q], lo, hi, c0 + sl)) doubt |= 1u << q;
        }
    }
    __device__ __forceinline__ void cell(int row, int col, int rr, int m) {
        const uint32_t c0 = ((uint32_t)row * (uint32_t)b.nc + (uint32_t)col) * C;
        disks(load_cell<C>(b, c0), c0, rr, m, best);
    }

    // A disk left to k_gb_far keeps what was found in its record until then.
    __device__ __forceinline__ void keep(bool far, unsigned open) const {
        uint4 *const r = reinterpret_cast<uint4 *>(b.g + i);
#pragma unroll
        for (int q = 0; q < 3; ++q)
            r[q] = make_uint4(__float_as_uint(best[q].lo), __float_as_uint(best[q].hi),
                              best[q].loc,
                              doubt | (far ? 8u : 0u) | (play[1] ? 16u : 0u) |
                                  (play[2] ? 32u : 0u) | (row_up ? 64u : 0u) |
                                  (row_dn ? 128u : 0u) | (open << 8));
    }
    // (true: to be searched beyond the near columns; open: arrows that stay open)
    __device__ __forceinline__ bool take_up(unsigned &open) {
        const uint4 *const r = reinterpret_cast<const uint4 *>(b.g + i);
        unsigned f = 0u;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const uint4 u = r[q];
            best[q].lo = __uint_as_float(u.x);
            best[q].hi = __uint_as_float(u.y);
            best[q].loc = u.z;
            f = u.w;
        }
        open = f >> 8;
        doubt = f & 7u & ~open;
        play[0] = true;
        play[1] = (f & 16u) != 0u;
        play[2] = (f & 32u) != 0u;
        row_up = (f & 64u) != 0u;
        row_dn = (f & 128u) != 0u;
        return (f & 8u) != 0u;
    }

    // the columns up to NEAR_COLS; the number searched
    __device__ __forceinline__ int near() {
        int m = 0;
        for (; m < min(NEAR_COLS, b.nc); ++m) {
            const unsigned open = open_at(m);
            if (!open) break;
            int col = cxi + m;
            if (col >= b.nc) col -= b.nc;
            if (row_dn && (open & 5u)) cell(rdn, col, -1, m);
            cell(cyi, col, 0, m);
            if (row_up && (open & 3u)) cell(rup, col, 1, m);
        }
        return m;
    }

    // The columns from `from` on (FAR_LANES lanes per disk): the next FAR_LANES blocks of
    // columns at once, and of the first one of which a row reaches a corridor
    // that is still open a column per lane. (The first block ends with its
    // columns before that one.)
    __device__ __forceinline__ void beyond(bool far, int from) {
        const int lane = threadIdx.x & 31, sub = lane % FAR_LANES, base = lane - sub;
        const int nc = b.nc, end = cxi + from < nc ? cxi + from : cxi + from - nc;
        const int first = end / FAR_COLS;
        // the corridors as limits of y in the rows (e covers corridor_f's doubts
        // and the roundings of these sums)
        const float e = 4.f * b.del, up0 = (b.half_f - e) + vi.y, up1 = (b.df + e) + vi.y;
        const float dn0 = vi.y - (b.df + e), dn1 = vi.y - (b.half_f - e);
        auto in = [](const float4 &l, float lo, float hi) {
            return (l.x < hi && l.y > lo) || (l.z < hi && l.w > lo);
        };
        for (int k = 0; __any_sync(FULL, far);) {
            int blk = first + k + sub;
            if (blk >= b.nblk) blk -= b.nblk;
            if (blk >= b.nblk) blk -= b.nblk;
            int c0 = k + sub == 0 ? end : blk * FAR_COLS, m = c0 - cxi;
            if (m < 0) m += nc;
            const unsigned open = far && k + sub <= b.nblk ? open_at(max(m, from)) : 0u;
            unsigned rows = 0u;
            if (open) {
                const float4 *const lim = b.ylim + blk;
                const float4 l0 = lim[rdn * b.nblk], l1 = lim[cyi * b.nblk], l2 = lim[rup * b.nblk];
                const bool c = (open & 1u) != 0u, u = (open & 2u) != 0u, d = (open & 4u) != 0u;
                if (row_dn && ((d && in(l0, dn0 + b.af, dn1 + b.af)) ||
                               (c && in(l0, dn1 + b.af, up0 + b.af))))
                    rows |= 1u;
                if ((u && in(l1, up0, up1)) || (d && in(l1, dn0, dn1)) || (c && in(l1, dn1, up0)))
                    rows |= 2u;
                if (row_up && ((u && in(l2, up0 - b.af, up1 - b.af)) ||
                               (c && in(l2, dn1 - b.af, up0 - b.af))))
                    rows |= 4u;
            }
            const unsigned hit = (__ballot_sync(FULL, rows != 0u) >> base) & ((1u << FAR_LANES) - 1u);
            const unsigned any = (__ballot_sync(FULL, open != 0u) >> base) & ((1u << FAR_LANES) - 1u);
            const int f = hit ? __ffs(hit) - 1 : 0, at = base + f;
            rows = __shfl_sync(FULL, rows, at);
            c0 = __shfl_sync(FULL, c0, at);
            blk = __shfl_sync(FULL, blk, at);
            const int c1 = k + f == b.nblk ? end : min(nc, blk * FAR_COLS + FAR_COLS);
            k += hit ? f + 1 : FAR_LANES;
            far = any != 0u;
            if (!__any_sync(FULL, hit != 0u)) continue;
            GBest l[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                l[q].lo = l[q].hi = INFINITY;
                l[q].loc = NONE;
            }
            const int col = c0 + sub;
            m = col - cxi;
            if (m < 0) m += nc;
            if (hit && col < c1 && m >= from) {
#pragma unroll 1
                for (int z = 0; z < 3; ++z) {
                    if (!((rows >> z) & 1u)) continue;
                    const int row = z == 0 ? rdn : z == 1 ? cyi : rup;
                    const uint32_t s0 = ((uint32_t)row * (uint32_t)nc + (uint32_t)col) * C;
                    disks(load_cell<C>(b, s0), s0, z - 1, m, l);
                }
            }
            // the lanes' candidates, then the best so far
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (!__any_sync(FULL, l[q].loc != NONE)) continue;
#pragma unroll
                for (int o = FAR_LANES / 2; o > 0; o >>= 1) {
                    const float lo = __shfl_xor_sync(FULL, l[q].lo, o);
                    const float hi = __shfl_xor_sync(FULL, l[q].hi, o);
                    const uint32_t loc2 = __shfl_xor_sync(FULL, l[q].loc, o);
                    if (loc2 != NONE && take_best(l[q], lo, hi, loc2)) doubt |= 1u << q;
                }
                if (l[q].loc != NONE && take_best(best[q], l[q].lo, l[q].hi, l[q].loc))
                    doubt |= 1u << q;
            }
        }
    }

    // What an open arrow says: nothing lies in its corridor before this place.
    __device__ __forceinline__ double open_until() const {
        const float thr = (float)NEAR_COLS * b.af - vi.x - b.df - (float)(NEAR_COLS + 4) * b.del;
        const double h = __dadd_rn(xi, (double)thr);
        return __longlong_as_double((long long)(dbits(h < b.L ? h : __dsub_rn(h, b.L)) | SIGN));
    }

    // The open arrows of the disk's record, to be searched again from its own
    // column on.
    __device__ __forceinline__ unsigned take_open() {
        const GDisk &r = b.g[i];
        unsigned o = 0u;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            play[q] = r.a[q] == NONE && (dbits(r.b[q]) & SIGN) != 0ull;
            if (play[q]) o |= 1u << q;
            best[q].lo = best[q].hi = INFINITY;
            best[q].loc = NONE;
        }
        row_up = row_dn = true;
        return o;
    }

    // the disk in slot l (NONE: none) and b towards it (the warp)
    __device__ __forceinline__ uint32_t arrow(uint32_t l, double &bv) const {
        bv = 0.0;
        if (!__any_sync(FULL, l != NONE)) return NONE;
        const uint32_t at = l != NONE ? l : loc, j = b.scid[at];
        double ay = fabs(__dsub_rn(gb_y(b, at, j), yi));
        if (__any_sync(FULL, cyi == 0 || cyi == b.nc - 1 || b.nc <= 4)) {
            const double la = __dsub_rn(b.L, ay);
            if (dbits(la) < dbits(ay)) ay = la;
        }
        const double v = __dsqrt_rn(__dsub_rn(b.d2, __dmul_rn(ay, ay)));
        if (l != NONE) bv = v;
        return l != NONE ? j : NONE;
    }

    // 16 bytes (part 0 .. 3) of the disk's record
    __device__ __forceinline__ void store(int part, const uint32_t (&id)[3],
                                          const double (&bv)[3]) const {
        ulonglong2 u;
        if (part == 0) u = make_ulonglong2(dbits(xi), 0ull);
        if (part == 1)
            u = make_ulonglong2((unsigned long long)OWN_STATIC | ((unsigned long long)id[0] << 32),
                                (unsigned long long)id[1] | ((unsigned long long)id[2] << 32));
        if (part == 2) u = make_ulonglong2(0ull, dbits(bv[0]));
        if (part == 3) u = make_ulonglong2(dbits(bv[1]), dbits(bv[2]));
        reinterpret_cast<ulonglong2 *>(b.g + i)[part] = u;
    }
};

template <int C>
__global__ void __launch_bounds__(256, 4) k_gb_arrows(GBuild b) {
    __shared__ uint32_t list[BUILD_CELLS * C];
    __shared__ int count;
    const int lane = threadIdx.x & 31;
    const uint32_t ncell = (uint32_t)b.nc * (uint32_t)b.nc;
    const uint32_t cell0 = blockIdx.x * BUILD_CELLS;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    static_assert(BUILD_CELLS * C % 32 == 0, "whole warps pack the slots");
    for (uint32_t q = threadIdx.x; q < BUILD_CELLS * C; q += blockDim.x) {
        const bool occ = cell0 + q / C < ncell && b.scid[cell0 * C + q] != EMPTY;
        const unsigned om = __ballot_sync(FULL, occ);
        int at = 0;
        if (lane == 0 && om) at = atomicAdd(&count, __popc(om));
        at = __shfl_sync(FULL, at, 0) + __popc(om & ((1u << lane) - 1u));
        if (occ) list[at] = cell0 * C + q;
    }
    __syncthreads();
    const int total = count;
    for (int e0 = 0; e0 < total; e0 += blockDim.x) {
        const int e = e0 + (int)threadIdx.x;
        GSearch<C> r(b, list[e < total ? e : 0]);
        r.begin();
        const int m = r.near();
        const unsigned open = m == NEAR_COLS && m < b.nc ? r.open_at(m) : 0u;
        const bool far = open != 0u && !b.start;
        const bool later = (b.start ? r.doubt & ~open : r.doubt) != 0u || far;
        const unsigned fm = __ballot_sync(FULL, e < total && later);
        if (fm) {
            unsigned at = 0u;
            if (lane == 0) at = (unsigned)atomicAdd(&b.count->listed, (unsigned long long)__popc(fm));
            at = __shfl_sync(FULL, at, 0) + __popc(fm & ((1u << lane) - 1u));
            if (e < total && later) {
                b.far[at] = r.loc;
                r.keep(far, b.start ? open : 0u);
            }
        }
        uint32_t id[3];
        double bv[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const bool op = b.start && ((open >> q) & 1u);
            id[q] = r.arrow(later || op ? NONE : r.best[q].loc, bv[q]);
            if (op) bv[q] = r.open_until();
        }
        if (b.start && __any_sync(FULL, e < total && open != 0u)) {
            const unsigned om = __ballot_sync(FULL, e < total && open != 0u);
            unsigned at = 0u;
            if (lane == 0)
                at = (unsigned)atomicAdd(&b.count->open, (unsigned long long)__popc(om));
            at = __shfl_sync(FULL, at, 0) + __popc(om & ((1u << lane) - 1u));
            if (e < total && open != 0u) b.far[b.n + at] = r.loc;
        }
        if (e < total && b.start) b.start[r.i] = r.xi;
        if (e < total && !later) {
            if (b.yout) b.yout[r.i] = r.yi;
#pragma unroll
            for (int part = 0; part < 4; ++part) r.store(part, id, bv);
        }
    }
}

// The disks that k_gb_arrows has listed, FAR_LANES lanes each. Along rows of
// disks little less than d apart most disks have no arrow to the rows beside or
// one far along: the blocks of columns that hold no disk in a corridor still
// open are passed over (k_gb_blocks).
// Bound by its instructions at eight blocks of 64 registers a multiprocessor
// (360000 disks, eta 0.60, half of them listed: 168 us; 217 at 92 registers).
// One disk per lane took 284 us there and 25 for a list of 40 disks (14 so), the
// whole warp per disk over all columns, inside k_gb_arrows and in FP64 where a
// corridor's edge was in doubt, 1360.
constexpr int FAR_THREADS = 128, FAR_BLOCKS = 1216;

//
// OPEN: the disks with open arrows instead, which are completed; nothing else of
// their records changes.
template <int C, bool OPEN>
__global__ void __launch_bounds__(FAR_THREADS, 8) k_gb_far(GBuild b) {
    constexpr int PER = 32 / FAR_LANES;  // disks a warp
    const int lane = threadIdx.x & 31, sub = lane % FAR_LANES, base = lane - sub;
    const unsigned total = (unsigned)(OPEN ? b.count->open : b.count->listed),
                   step = gridDim.x * (FAR_THREADS / FAR_LANES);
    for (unsigned e0 = (blockIdx.x * FAR_THREADS + threadIdx.x) / 32u * PER; e0 < total;
         e0 += step) {
        const bool has = e0 + base / FAR_LANES < total;
        const unsigned e = has ? e0 + base / FAR_LANES : e0;
        GSearch<C> r(b, b.far[OPEN ? b.n + e : e]);
        unsigned open = 0u;  // arrows: that stay open; OPEN: that are completed
        bool far = true;
        if (OPEN)
            open = r.take_open();
        else
            far = r.take_up(open);
        r.beyond(has && far, OPEN ? 0 : NEAR_COLS);
        uint32_t aj[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            aj[q] = !OPEN && ((open >> q) & 1u) ? NONE : r.best[q].loc;
            unsigned odd = __ballot_sync(FULL, has && ((r.doubt >> q) & 1u));
            while (odd) {
                const int src = __ffs(odd) - 1, g = src / FAR_LANES;
                odd &= ~(((1u << FAR_LANES) - 1u) << (g * FAR_LANES));
                const uint32_t ex = arrow_exact<C>(
                    b, q, __shfl_sync(FULL, r.loc, src),
                    make_float2(__shfl_sync(FULL, r.vi.x, src), __shfl_sync(FULL, r.vi.y, src)),
                    __shfl_sync(FULL, r.xi, src), __shfl_sync(FULL, r.yi, src),
                    __shfl_sync(FULL, r.cxi, src), __shfl_sync(FULL, r.cyi, src),
                    __shfl_sync(FULL, r.best[q].lo, src), __shfl_sync(FULL, r.best[q].hi, src));
                if (lane / FAR_LANES == g) aj[q] = ex;
            }
        }
        // a lane per arrow, then a lane per part of the record
        double v;
        const uint32_t j = r.arrow(sub == 0 ? aj[0] : sub == 1 ? aj[1] : sub == 2 ? aj[2] : NONE, v);
        if (OPEN) {
            if (has && sub < 3 && ((open >> sub) & 1u)) {
                b.g[r.i].b[sub] = v;
                b.g[r.i].a[sub] = j;
            }
            continue;
        }
        if (sub < 3 && ((open >> sub) & 1u)) v = r.open_until();
        uint32_t id[3];
        double bv[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            id[q] = __shfl_sync(FULL, j, base + q);
            bv[q] = shfl_f64(v, base + q);
        }
        if (has && sub < 4) r.store(sub, id, bv);
        if (has && sub == 4 && b.yout) b.yout[r.i] = r.yi;
    }
}

// ---------------------------------------------------------- frames of rings
//
// A cell row whose disks lie within RING_SPREAD d of each other in y, d or
// more from every disk of the rows beside, is a ring: a chain there never
// leaves it, its disks keep their cyclic order in x (all pairs are within d in
// y), and a disk's target is always the next one (every b lies in 0.51 d .. d,
// so the disk after the next is reached 0.02 d later at least). In a frame
// whose rows all are rings -- a lattice start on cells aligned with it -- a
// chain's run is a stretch of consecutive places (g_leap_chain) instead of a
// walk from record to record. The cells' row bands decide (k_ring_rows).

constexpr double RING_SPREAD = 0.86;
constexpr int RING_CHUNK = 256;  // columns of a row per block of the kernels below

struct GRing {
    uint32_t *off;                 // [nc * chunks + 1] disks per chunk, then first places
    unsigned long long *ylo, *yhi; // [nc] least and largest y (bits) per row (all ones, 0)
};

static int ring_chunks(int nc) { return (nc + RING_CHUNK - 1) / RING_CHUNK; }

// Disks per chunk, and the rows' bands (least: all ones; largest: 0 before).
template <int C>
__global__ void __launch_bounds__(RING_CHUNK) k_ring_count(GBuild b, GRing r) {
    __shared__ unsigned long long wlo[RING_CHUNK / 32], whi[RING_CHUNK / 32];
    __shared__ int wn[RING_CHUNK / 32];
    const uint32_t nc = (uint32_t)b.nc, row = blockIdx.y;
    const uint32_t col = blockIdx.x * RING_CHUNK + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long lo = INF_BITS, hi = 0ull;
    int n = 0;
    if (col < nc) {
        uint32_t id[C];
        const uint4 *q = reinterpret_cast<const uint4 *>(b.scid + ((size_t)row * nc + col) * C);
#pragma unroll
        for (int z = 0; z < C / 4; ++z) {
            const uint4 v = q[z];
            id[4 * z] = v.x;
            id[4 * z + 1] = v.y;
            id[4 * z + 2] = v.z;
            id[4 * z + 3] = v.w;
        }
#pragma unroll
        for (int z = 0; z < C; ++z) {
            if (id[z] == EMPTY) continue;
            const unsigned long long y = dbits(coord(b.y[id[z]]));  // ordered by bits
            lo = y < lo ? y : lo;
            hi = y > hi ? y : hi;
            ++n;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l2 = shfl_xor_u64(lo, o), h2 = shfl_xor_u64(hi, o);
        lo = l2 < lo ? l2 : lo;
        hi = h2 > hi ? h2 : hi;
        n += __shfl_xor_sync(FULL, n, o);
    }
    if (lane == 0) {
        wlo[w] = lo;
        whi[w] = hi;
        wn[w] = n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < RING_CHUNK / 32; ++q) {
            lo = wlo[q] < lo ? wlo[q] : lo;
            hi = whi[q] > hi ? whi[q] : hi;
            n += wn[q];
        }
        if (n) {
            atomicMin(r.ylo + row, lo);
            atomicMax(r.yhi + row, hi);
        }
        r.off[row * gridDim.x + blockIdx.x] = (uint32_t)n;
    }
}

// Whether some row is no ring (count->mixed), and the chunks' first places
// (one block). Two neighbour rows lie d apart when RN(ylo(above) - yhi(below))
// >= d: rounding is monotone, so |RN(dy)| >= d for every pair; across the box
// edge RN(L - RN(yhi(nc - 1) - ylo(0))) bounds every pair's periodic image.
__global__ void k_ring_rows(GBuild b, GRing r, int chunks) {
    __shared__ int warp_tot[32];
    __shared__ int tot[2];
    const int nc = b.nc;
    bool no = nc < 5;
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
        const unsigned long long l = r.ylo[q];
        if (l == ~0ull) continue;
        const double yl = __longlong_as_double((long long)l),
                     yh = __longlong_as_double((long long)r.yhi[q]);
        no = no || !(__dsub_rn(yh, yl) < __dmul_rn(RING_SPREAD, b.d));
        const int up = q == nc - 1 ? 0 : q + 1;
        const unsigned long long u = r.ylo[up];
        if (u != ~0ull) {
            const double yu = __longlong_as_double((long long)u);
            no = no || !((up ? __dsub_rn(yu, yh) : __dsub_rn(b.L, __dsub_rn(yh, yu))) >= b.d);
        }
    }
    const int any = __syncthreads_or(no);
    const int n = nc * chunks, per = (n + (int)blockDim.x - 1) / (int)blockDim.x;
    const int lo = min(n, (int)threadIdx.x * per), hi = min(n, lo + per);
    int sum = 0;
    for (int q = lo; q < hi; ++q) sum += (int)r.off[q];
    int off = block_exscan(sum, warp_tot, tot);
    for (int q = lo; q < hi; ++q) {
        const int c = (int)r.off[q];
        r.off[q] = (uint32_t)off;
        off += c;
    }
    if (threadIdx.x == 0) {
        r.off[n] = (uint32_t)tot[0];
        if (any) b.count->mixed = 1ull;
    }
}

// Places: a cell's disks, in the order of x, follow those of the cells before.
template <int C>
__global__ void __launch_bounds__(RING_CHUNK) k_ring_place(GBuild b, GRing r, GDev s) {
    __shared__ int warp_tot[32];
    __shared__ int tot[2];
    const uint32_t nc = (uint32_t)b.nc, row = blockIdx.y, ch = gridDim.x;
    const uint32_t col = blockIdx.x * RING_CHUNK + threadIdx.x;
    const uint32_t first = r.off[row * ch], len = r.off[(row + 1) * ch] - first;
    uint32_t id[C];
    double x[C];
    int n = 0;
    if (col < nc) {
#pragma unroll
        for (int q = 0; q < C; ++q) id[q] = b.scid[((size_t)row * nc + col) * C + q];
#pragma unroll
        for (int q = 0; q < C; ++q) {
            x[q] = id[q] != EMPTY ? coord(b.x[id[q]]) : INFINITY;
            n += id[q] != EMPTY;
        }
    }
    const uint32_t at = r.off[row * ch + blockIdx.x] + (uint32_t)block_exscan(n, warp_tot, tot);
    if (n == 0) return;
#pragma unroll
    for (int q = 0; q < C; ++q) {
        if (id[q] == EMPTY) continue;
        int rank = 0;  // ordered by bits
#pragma unroll
        for (int z = 0; z < C; ++z)
            rank += dbits(x[z]) < dbits(x[q]) || (z < q && dbits(x[z]) == dbits(x[q]));
        s.rid[at + rank] = id[q];
        s.pos[id[q]] = make_uint4(at + (uint32_t)rank, first, len, row);
    }
}

// The records of a frame of rings, each disk's successor its only arrow (a
// cell-scan context; one with graph arrows has them from k_gb_arrows). Bound
// by the 64 bytes a record takes: a thread per disk finds its fields, then four
// lanes write a record, so that a store covers eight whole ones. 2^20 disks:
// 59 us with a thread per record, 28 so.
__global__ void __launch_bounds__(256) k_ring_records(GBuild b, GDev s) {
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i0 = i - lane;
    unsigned long long xb = 0ull, vb = 0ull;
    uint32_t a0 = NONE;
    if (i < s.n) {
        const uint4 at = s.pos[i];
        const double yi = coord(b.y[i]);
        xb = dbits(coord(b.x[i]));
        s.y[i] = yi;
        if (at.z > 1u) {
            a0 = s.rid[at.x + 1u < at.y + at.z ? at.x + 1u : at.y];
            const double ay = fabs(__dsub_rn(coord(b.y[a0]), yi));
            vb = dbits(__dsqrt_rn(__dsub_rn(b.d2, __dmul_rn(ay, ay))));
        }
    }
#pragma unroll
    for (int z = 0; z < 4; ++z) {
        const int src = 8 * z + (lane >> 2), part = lane & 3;
        const unsigned long long x2 = shfl_u64(xb, src), v2 = shfl_u64(vb, src);
        const uint32_t a2 = __shfl_sync(FULL, a0, src);
        ulonglong2 w = make_ulonglong2(0ull, 0ull);
        if (part == 0) w.x = x2;
        if (part == 1)
            w = make_ulonglong2((unsigned long long)OWN_STATIC | ((unsigned long long)a2 << 32),
                                ~0ull);
        if (part == 2) w.y = v2;
        if (i0 + src < s.n) reinterpret_cast<ulonglong2 *>(s.g + i0 + src)[part] = w;
    }
}

// The chains' start disks active (after a build); copied to kept (or null).
__global__ void k_g_init_chains(GDev s, const int32_t *active, int32_t *kept) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.k) return;
    const uint32_t a = active ? (uint32_t)active[c] : s.ci[c];
    if (kept) kept[c] = (int32_t)a;
    s.ci[c] = a;
    s.ci0[c] = a;
    s.g[a].own = OWN_ACTIVE | (uint32_t)c;
    s.nrec[c] = 0;
    s.status[c] = ST_STALLED;
}

// --------------------------------------------------------- parallel pass

// How a chain's run alone ended (sp_end; SP_LAP: it may have come round the
// box, so that a disk can be in its records more than once).
enum { SP_STALL = 0, SP_PAUSE = 1, SP_NONSTATIC = 2, SP_LIMIT = 3, SP_END = 3, SP_LAP = 4 };

// Two levels of disk records per warp in shared memory: the records that the
// targets of the active disk's targets may be next (record 3p + q: arrow q of
// target p), and the level before. They are copied in asynchronously
// (cp.async): a load into registers shares one of the warp's few scoreboards
// with the step's arithmetic and shuffles, which then waited for it (~600 of
// 1400 cycles an event).
struct GLevels {
    GDisk r[2][9];
};
__device__ __forceinline__ GLevels &g_levels() {
    __shared__ GLevels lv[8];  // one per warp of the block
    return lv[threadIdx.x >> 5];
}

__device__ __forceinline__ void g_copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void g_copy_wait() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
}

// 16 bytes (part 0 .. 3) of disk id's record into dst; nothing for NONE.
// (A record that stands for no disk in global memory, read by every warp at
// every step, made its L2 line a hot spot: 3000 cycles an event.)
__device__ __forceinline__ void g_fetch_part(const GDisk *g, uint32_t id, GDisk *dst, int part) {
    if (id != NONE)
        g_copy16(reinterpret_cast<ulonglong2 *>(dst) + part,
                 reinterpret_cast<const ulonglong2 *>(g + id) + part);
}

// Requests the records of the nine arrows of targets from[0 .. 2] into to;
// none: the targets that are no disk (bit p), whose records are not there.
__device__ __forceinline__ void g_fetch(const GDisk *g, const GDisk *from, unsigned none,
                                        GDisk *to) {
    const int lane = threadIdx.x & 31, z = lane >> 2;
    const int zp = z / 3, zq = z - 3 * zp;
    g_fetch_part(g, (none >> zp) & 1u ? NONE : from[zp].a[zq], to + z, lane & 3);
    if (lane < 4) g_fetch_part(g, (none >> 2) & 1u ? NONE : from[2].a[2], to + 8, lane);
}

// Requests the records of the active disk i's three targets into to[0 .. 2].
__device__ __forceinline__ void g_fetch_first(const GDisk *g, uint32_t i, GDisk *to) {
    const int lane = threadIdx.x & 31;
    if (lane < 12) g_fetch_part(g, g[i].a[lane >> 2], to + (lane >> 2), lane & 3);
}

// The targets (tid on lanes 0 .. 2) that are no disk, bit p.
__device__ __forceinline__ unsigned g_none(uint32_t tid) {
    return __ballot_sync(FULL, tid == NONE) & 7u;
}

// A step whose target an open arrow may hide: nothing of the launch will stand
// (the error word ends it after the leg; the host looks for LC_OPEN first).
__device__ __noinline__ void g_undecided(const GDev &s) {
    atomicAdd(s.lc + LC_OPEN, 1ull);
    atomicAdd(s.lc + LC_ERR_REC, 1ull);
}

// Open arrows among the targets (first: the record of target 0) become targets at
// their place, static and never moved; b, on the lanes of such a target (0 .. 2,
// repeated), is 0 from then on.
__device__ __noinline__ void g_open_targets(uint32_t tid, double tb, GDisk *first) {
    const int lane = threadIdx.x & 31;
    if (lane < 3 && g_open(tid, tb)) {
        first[lane].x = g_unsigned(tb);
        first[lane].t = 0.0;
        first[lane].own = OWN_STATIC;
    }
    __syncwarp();
}

// FP64 fix-ups of the uncommon case, out of line: the compiler then never
// evaluates them on the common path (an FP64 instruction occupies its unit
// ~64 cycles on this chip).
__device__ __noinline__ double g_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __noinline__ double g_sub(double a, double b) { return __dsub_rn(a, b); }

// The lane (0 .. 2) with the least (tau, j) (tk: tau bits, INF where the lane
// has no candidate). The high words decide unless two lanes share theirs (or
// none has a candidate: some lane with INF then).
__device__ __forceinline__ int g_winner(unsigned long long tk, uint32_t id) {
    const unsigned hi = (unsigned)(tk >> 32);
    const unsigned mh = __reduce_min_sync(FULL, hi);
    const unsigned eq = __ballot_sync(FULL, hi == mh);
    const int first = __ffs(eq) - 1;
    if ((eq & (eq - 1u)) == 0u) return first;
    const unsigned lo = hi == mh ? (unsigned)tk : ~0u;
    const unsigned ml = __reduce_min_sync(FULL, lo);
    const bool tie = hi == mh && lo == ml;
    const unsigned mj = __reduce_min_sync(FULL, tie ? id : ~0u);
    return (__ffs(__ballot_sync(FULL, tie && id == mj)) - 1) % 3;
}

// Up to 32 events of a chain, event e on lane e mod 32, as the steps found
// them: moved disk, its place, time and remaining length before, tau and the
// target's local time. What else a record holds is the next event's (its
// disk is this one's target) or one addition for all lanes.
struct GEvs {
    uint32_t i;
    double x, t, D, tau, tj;
};

// Writes records n0 .. n - 1 of chain c (n - n0 <= 32 events on the lanes;
// record index nr0 + e, order key seq0 + e). i, xi, ti, D: the state after
// event n - 1 (lift: that event is a lifting). Returns this lane's event: the
// moved disk's new place, its event time and target.
struct GFlush {
    bool has;
    double xn, t;
    uint32_t j;
};
__device__ __forceinline__ GFlush g_flush(const GDev &s, int c, int32_t nr0, uint32_t seq0, int n0,
                                          int n, const GEvs &E, uint32_t i, double xi, double ti,
                                          double D, bool lift) {
    const int lane = threadIdx.x & 31;
    const int e = n0 + ((lane - n0) & 31);  // this lane's event
    const bool last = e == n - 1;
    const int nx = (lane + 1) & 31;
    const uint32_t inx = __shfl_sync(FULL, E.i, nx);
    const double xnx = shfl_f64(E.x, nx), tnx = shfl_f64(E.t, nx), dnx = shfl_f64(E.D, nx);
    GFlush f;
    f.has = e < n;
    f.j = last ? (lift ? i : NONE) : inx;
    f.t = last ? ti : tnx;
    const double xj = last ? (lift ? xi : 0.0) : xnx;
    const double da = last ? (lift ? D : 0.0) : dnx;
    f.xn = __dadd_rn(E.x, E.tau);
    const bool wrap = f.has && dbits(f.xn) >= dbits(s.L);
    if (__any_sync(FULL, wrap) && wrap) f.xn = g_sub(f.xn, s.L);
    if (f.has) {
        ulonglong2 *u = reinterpret_cast<ulonglong2 *>(grec_at(s, c, nr0 + e));
        u[0] = make_ulonglong2((unsigned long long)E.i | ((unsigned long long)f.j << 32),
                               (unsigned long long)(seq0 + (uint32_t)e));
        u[1] = make_ulonglong2(dbits(E.x), dbits(E.t));
        u[2] = make_ulonglong2(dbits(E.tj), dbits(f.t));
        u[3] = make_ulonglong2(dbits(E.tau), dbits(f.xn));
        u[4] = make_ulonglong2(dbits(xj), dbits(da));
    }
    return f;
}

__device__ __forceinline__ unsigned long long g_key(double t, int c) {
    return ((unsigned long long)(unsigned)__float_as_int(d2f_trunc(t)) << 32) | (unsigned)c;
}

// Liftings after which a chain's run may come round the box to a disk it
// moved: n liftings advance by at most n d + (the time gone), and a target
// behind lies L less that ahead, out of reach while it exceeds what is left
// of ell.
__device__ __forceinline__ int g_lap(const GDev &s) {
    const float f = __fsub_rn(__fdiv_rn(d2f_trunc(__dsub_rn(s.L, s.ell)), d2f_trunc(s.d)), 4.f);
    return f > 1e9f ? 1000000000 : (int)f;
}

// Chain c at the start of a leg, on its stalled disk i with D = ell (one warp).
__device__ __forceinline__ void g_begin_state(const GDev &s, int c, uint32_t i, int lane) {
    if (lane != 0) return;
    s.g[i].t = 0.0;
    s.g[i].own = OWN_ACTIVE | (uint32_t)c;
    s.ci0[c] = i;
    s.D[c] = s.ell;
    s.tc[c] = 0.0;
    s.status[c] = ST_RUNNING;
    s.partner[c] = -1;
    s.nrec[c] = 0;
    s.nlift[c] = 0;
}

// Parallel pass of a claim window [tw, tend): one warp runs chain c alone from
// the window-start state -- the isolated run of the conflict flag -- and
// writes no disk, so a step waits for one round of loads and for nothing
// else. While lanes 0 .. 2 compute the times of flight to the active disk's
// three targets, the records of those targets' nine arrows are already on
// their way: whichever target wins, the next step's records are there. Events
// stay on the lanes until 32 are there or the run ends. (One thread per chain
// with an atomicCAS per disk read took ~4000 cycles an event; a warp that
// handed records on by shuffles and wrote each event at once 3300; records
// in registers 1400.)
//
// What the run posts, without waiting: its events as records, and the disks
// it touches (its active disks) in path with a touch key in s.key
// (g_resolve_chain). The flag's words follow later (g_flag_chain).
//
// Another chain's active or stalled disk among the targets ends the run
// there if it lies in reach nearer than the winner (Remark 10). With claim
// windows or restarts a chain's disk lies behind its true place at the
// window's start (lazy frame), so the pass is strict there: such a disk in
// reach at all, or failing Eq. 2, ends the run, and the read disks are
// claimed like the touched ones.
//
// A step is bound by its instructions (one warp runs alone on its
// sub-partition, ~10 cycles an instruction), so the loop holds what every
// step needs; everything else waits for the flush or stands behind any_odd.
//
// OPEN: in a launch with open arrows (a few instructions more a step: 0.13 us).
template <bool OPEN>
__device__ __noinline__ void g_spec_chain(const GDev &s, int c, double tw, double tend,
                                          bool begin) {
    const int lane = threadIdx.x & 31;
    // (loads of one round trip: the chain's state, used or not)
    uint32_t i = s.ci[c];
    double ti = s.tc[c], D = s.D[c];
    int32_t nr0 = s.nrec[c];
    const int32_t st0 = s.status[c];
    if (begin) {
        ti = 0.0;
        D = s.ell;
        nr0 = 0;
        g_begin_state(s, c, i, lane);
    } else if (st0 != ST_RUNNING) {
        if (lane == 0) s.sp[c].touch = 0;
        return;
    }
    const int l3 = lane % 3;
    const double L = s.L;
    const bool strict = s.strict != 0;
    unsigned long long *const key = s.key;
    const GDisk *const g = s.g;
    const uint32_t stamp = s.stamp;
    const bool bounded = dbits(tend) != INF_BITS;
    const int room = s.cap - nr0, n_lap = g_lap(s);
    double xi = g[i].x;
    const uint32_t own0 = g[i].own;
    GLevels &lv = g_levels();
    int cb = 0, sl = 0;  // the active disk's targets: lv.r[cb][sl .. sl + 2]
    g_fetch_first(g, i, lv.r[0]);
    uint32_t tid = g[i].a[l3];
    double tb = g[i].b[l3];
    unsigned none = g_none(tid);
    g_copy_wait();
    // (an arrow not searched to its end: the step that would need it is no step)
    bool op = OPEN && g_open(tid, tb);
    if (OPEN && none) {
        g_open_targets(tid, tb, lv.r[0]);
        if (op) tb = 0.0;
    }
    if (lane == 0 && (g_static(own0) || (own0 & OWN_CHAIN) != (uint32_t)c))
        gdiag(s, 6, tw, c, i, own0, 0, 0);
    if (lane == 31) {
        *gpath_at(s, c, 0) = i;
        red_min_u64(key + i, g_key(ti, c));
    }
    GEvs E;
    E.i = NONE;
    E.x = E.t = E.D = E.tau = E.tj = 0.0;
    double cur = 0.0;  // the last step, evaluated but not taken: its scan's limit
    int n = 0, nf = 0, end = SP_PAUSE;  // nf: events written out
    int cut = 0x7FFFFFFF;
    uint32_t partner = NONE;
    // events nf .. n - 1 to memory, with the touched disks and their keys
    auto flush = [&](bool lift) {
        if (n == nf) return;
        const GFlush f = g_flush(s, c, nr0, (uint32_t)nr0, nf, n, E, i, xi, ti, D, lift);
        if (f.has) {
            const int e = nf + ((lane - nf) & 31);
            if (f.j != NONE) {
                *gpath_at(s, c, e + 1) = f.j;
                red_min_u64(key + f.j, g_key(f.t, c));
            }
            if (s.cells) {
                const size_t at = (size_t)e * (size_t)s.k + (size_t)c;
                s.pxt[at] = make_double2(E.x, E.tau);
                s.pcell[at] = cell_of(s, E.x, s.y[E.i]);
            }
            if (strict) {
#pragma unroll
                for (int z = 0; z < 3; ++z)
                    if (g[E.i].a[z] != NONE) red_min_u64(key + g[E.i].a[z], g_key(E.t, c));
            }
            if (dbits(f.t) < dbits(tw)) {
                // a window's events start at its start time (repairs roll back to it)
                atomicAdd(s.lc + LC_ORDER, 1ull);
                gdiag(s, 9, tw, c, E.i, f.j, E.t, E.tau);
            }
        }
        E.tj = 0.0;
        nf = n;
    };
    // the next event index at which the loop has to do more than a step
    int n_stop = min(min(room, 32), max(n_lap + 1, 0));
    for (;;) {
        const GDisk *const R = &lv.r[cb][sl];
        // the records beyond the targets
        g_fetch(g, R, none, lv.r[cb ^ 1]);
        const bool ev = lane < 3 && (tid != NONE || (OPEN && op));
        double rx = R[l3].x, rt = R[l3].t;
        uint32_t own = R[l3].own;
        if (n >= n_stop) {
            if (n - nf == 32) flush(true);
            if (n > n_lap) {
                // a target the run itself has moved: its place and time from
                // the run's latest record of it
                flush(true);
                __syncwarp();
                for (int z = 0; z < 3; ++z) {
                    const uint32_t id = __shfl_sync(FULL, tid, z);
                    int best = -1;
                    for (int e = lane; id != NONE && e < n; e += 32)
                        if (grec_at(s, c, nr0 + e)->i == id) best = e;
                    best = __reduce_max_sync(FULL, best);
                    if (best >= 0 && l3 == z) {
                        const GEv &u = *grec_at(s, c, nr0 + best);
                        rx = u.xi;
                        rt = u.t;
                        own = stamp;
                    }
                }
                n_stop = n + 1;
            } else {
                n_stop = min(nf + 32, n_lap + 1);
            }
            n_stop = min(n_stop, max(room, n + (n < room ? 1 : 0)));
        }
        // time of flight to each target (Sec. 2.2): forward image in x, b_ij
        // fixed with the arrow, clamped at 0
        double dx = __dsub_rn(rx, xi);
        double tau = __dsub_rn(dx, tb);
        // (anything but a static disk ahead, not moved in this leg)
        const bool odd = ev && (own >= OWN_ACTIVE || own == stamp ||
                                __double_as_longlong(dx) < 0);
        const bool any_odd = __any_sync(FULL, odd);
        bool nsc = false, hv = false, lap = false;
        if (any_odd) {
            if (odd && __double_as_longlong(dx) < 0) tau = g_sub(g_add(dx, L), tb);
            if (__double_as_longlong(tau) < 0) tau = 0.0;
            nsc = ev && own >= OWN_ACTIVE;
            rt = g_time(own, rt, stamp);
            if (ev && dbits(rt) != 0ull) {
                const double sum = g_add(ti, tau);
                // a target with t_i + tau < t_j became static after the
                // chain's disk had passed it and is one lap away (lazy
                // per-chain frame)
                lap = !nsc && dbits(sum) < dbits(rt);
                if (lap) tau = g_add(tau, L);
                // (in the chain's own window only it has moved disks, each at
                // its own time then: an assertion)
                if (lap && dbits(rt) >= dbits(tw)) atomicAdd(s.lc + LC_HORIZON, 1ull);
                hv = nsc && !(dbits(sum) > dbits(rt));
            }
        }
        if (__double_as_longlong(tau) < 0) tau = 0.0;
        const unsigned long long tk = ev && !nsc ? dbits(tau) : INF_BITS;
        const int wl = g_winner(tk, tid);
        const unsigned long long bt = shfl_u64(tk, wl);
        const uint32_t bj = __shfl_sync(FULL, tid, wl);
        const double xj = shfl_f64(rx, wl);
        if (any_odd) {
            // another chain's disk among the targets
            const bool stop = nsc && (strict ? hv || dbits(tau) < dbits(D)
                                             : dbits(tau) <= bt && dbits(tau) < dbits(D));
            const unsigned sb = __ballot_sync(FULL, stop);
            if (sb && cut == 0x7FFFFFFF) {
                partner = __shfl_sync(FULL, own, __ffs(sb) - 1) & OWN_CHAIN;
                // (with the flag on cells a run cut by a disk beyond its winner
                // goes on for its cells, unpublished from here)
                cut = n;
                const bool near = stop && dbits(tau) <= bt && dbits(tau) < dbits(D);
                if (!s.cells || __any_sync(FULL, near)) {
                    end = SP_NONSTATIC;
                    cur = bt < dbits(D) ? __longlong_as_double((long long)bt) : D;
                    break;
                }
            } else if (sb && __any_sync(FULL, stop && dbits(tau) <= bt && dbits(tau) < dbits(D))) {
                end = SP_NONSTATIC;
                cur = bt < dbits(D) ? __longlong_as_double((long long)bt) : D;
                break;
            }
            const double tj = shfl_f64(rt, wl);
            if (lane == (n & 31)) E.tj = bt < dbits(D) ? tj : 0.0;
        }
        bool lift = bt < dbits(D);
        if (OPEN && lift && bj == NONE) {
            if (lane == 0) g_undecided(s);
            lift = false;
        }
        const double ts = lift ? __longlong_as_double((long long)bt) : D;
        const double T = __dadd_rn(ti, ts);
        if (n >= room) {  // out of records: the repair goes on from here, or reports it
            end = SP_LIMIT;
            cur = ts;
            break;
        }
        if (bounded && !(dbits(T) < dbits(tend))) {  // pauses at the window end
            cur = ts;
            break;
        }
        if (lane == (n & 31)) {
            E.i = i;
            E.x = xi;
            E.t = ti;
            E.D = D;
            E.tau = ts;
        }
        ++n;
        ti = T;
        if (!lift) {
            end = SP_STALL;
            D = 0.0;
            break;
        }
        D = __dsub_rn(D, ts);
        xi = xj;
        i = bj;
        tid = R[wl].a[l3];
        tb = R[wl].b[l3];
        none = g_none(tid);
        g_copy_wait();
        cb ^= 1;
        sl = 3 * wl;
        if (OPEN) {
            op = g_open(tid, tb);
            if (none) g_open_targets(tid, tb, &lv.r[cb][sl]);
            if (op) tb = 0.0;
        }
    }
    g_copy_wait();
    // (the reads of a step that was evaluated but not taken)
    if (strict && end != SP_STALL && lane < 3 && tid != NONE) red_min_u64(key + tid, g_key(ti, c));
    flush(end != SP_STALL);
    if (s.cells && end != SP_STALL && lane == 1) {
        const size_t at = (size_t)n * (size_t)s.k + (size_t)c;
        s.pxt[at] = make_double2(xi, cur);
        s.pcell[at] = cell_of(s, xi, s.y[i]);
    }
    if (lane == 0) {
        GSpec r;
        r.n = n;
        r.touch = end == SP_STALL ? n : n + 1;
        r.end = end | (n > n_lap ? SP_LAP : 0);
        if (s.ring && strict && n > 0 && (uint32_t)n >= s.pos[i].z)
            atomicAdd(s.lc + LC_RINGLAP, 1ull);
        r.partner = partner < (uint32_t)s.k ? (int32_t)partner : -1;
        r.tc = ti;
        r.D = D;
        r.ci = i;
        r.cut = cut;
        r.pad[0] = r.pad[1] = 0;
        s.sp[c] = r;
    }
    __syncwarp();
}

// The sums of a stretch of events, tau of event e on lane e: t and D before
// event 0 (the same on every lane) become those before this lane's event, each
// addition rounded as the steps round it, for the events up to `bound` as long
// as D is not negative. Time is summed on the lower lanes and remaining length
// on the upper, in one FP64 instruction an event; before event e they go to
// lane e of each half (e < 16), or to a second register of lane e - 16.
__device__ __forceinline__ void g_sums(double tau, int bound, double &t, double &D) {
    const int lane = threadIdx.x & 31, half = lane & 15;
    const unsigned long long flip = lane < 16 ? 0ull : 1ull << 63;
    double v = lane < 16 ? t : D, v0 = v, v1 = v;
    for (int e0 = 0; e0 <= bound; e0 += 8) {
#pragma unroll
        for (int z = 0; z < 8; ++z) {
            const int e = e0 + z;
            if (half == (e & 15)) {
                if (e0 < 16)
                    v0 = v;
                else
                    v1 = v;
            }
            v = __dadd_rn(v, __longlong_as_double((long long)(shfl_u64(dbits(tau), e) ^ flip)));
        }
        if (__any_sync(FULL, lane >= 16 && __double_as_longlong(v) < 0)) break;
    }
    const double ta = shfl_f64(v0, half), tb = shfl_f64(v1, half);
    const double da = shfl_f64(v0, half + 16), db = shfl_f64(v1, half + 16);
    t = lane < 16 ? ta : tb;
    D = lane < 16 ? da : db;
}

// A disk of a ring as a stretch needs it: the record in three loads, four where
// it has more than one arrow.
struct GRingDisk {
    double x, t;
    uint32_t own, a0, a1, a2;
    unsigned long long claim;
    double b0, b1, b2;
    __device__ __forceinline__ explicit GRingDisk(const GDisk *g) {
        const ulonglong2 *const r = reinterpret_cast<const ulonglong2 *>(g);
        const ulonglong2 r0 = __ldcg(r), r1 = __ldcg(r + 1), r2 = __ldcg(r + 2), r3 = __ldcg(r + 3);
        x = __longlong_as_double((long long)r0.x);
        t = __longlong_as_double((long long)r0.y);
        own = (uint32_t)r1.x;
        a0 = (uint32_t)(r1.x >> 32);
        a1 = (uint32_t)r1.y;
        a2 = (uint32_t)(r1.y >> 32);
        claim = r2.x;
        b0 = __longlong_as_double((long long)r2.y);
        b1 = __longlong_as_double((long long)r3.x);
        b2 = __longlong_as_double((long long)r3.y);
    }
    // b towards disk j; false if no arrow leads there
    __device__ __forceinline__ bool towards(uint32_t j, double &b) const {
        b = a0 == j ? b0 : a1 == j ? b1 : b2;
        return a0 == j || a1 == j || a2 == j;
    }
};

// The same pass in a frame of rings, of a leg from its start (not strict): the
// run's disks are consecutive places, so lane e holds the e-th from the active
// disk on and finds its gap to the next; only the sums of Eq. 1 -- the time and
// the remaining length before each event -- are a chain of additions, each
// rounded as the steps round it (g_sums). A stretch covers 31 events; most legs end within the first.
// What the run leaves is g_spec_chain's, word by word. A run that comes round
// its ring, or out of records, is left to g_spec_chain (false).
//
// Bound by that chain (~100 cycles an event against ~1000 of a step) and the
// four dependent loads before it. 1024 chains on 2^20 disks: the pass 5 us, a
// step per event 12; a leg 82 us with the scan of row bands this replaced, 65
// with it at first, 32 now (16384 chains: 890, 605, 200).
__device__ __noinline__ bool g_leap_chain(const GDev &s, int c) {
    const int lane = threadIdx.x & 31;
    const uint32_t i0 = s.ci[c];
    g_begin_state(s, c, i0, lane);
    const GDisk *const g = s.g;
    const double L = s.L;
    const uint4 at0 = s.pos[i0];
    const uint32_t p0 = at0.x, first = at0.y, len = at0.z, row = at0.w;
    uint32_t id = 0u;
    double t = 0.0, D = s.ell;  // before the event on lane 0
    int n0 = 0, end = SP_STALL, n = 0;
    uint32_t partner = NONE, iend = i0;
    if (lane == 31) {
        *gpath_at(s, c, 0) = i0;
        red_min_u64(s.key + i0, g_key(0.0, c));
    }
    for (;; n0 += 31) {
        uint32_t q = p0 - first + (uint32_t)(n0 + lane);
        if (q >= len) q %= len;
        id = s.rid[first + q];
        const GRingDisk k(g + id);
        const double x = k.x;
        const uint32_t own = k.own;
        const double xn = shfl_f64(x, (lane + 1) & 31);
        const uint32_t idn = __shfl_sync(FULL, id, (lane + 1) & 31);
        const uint32_t ownn = __shfl_sync(FULL, own, (lane + 1) & 31);
        double bb;
        // targets: the last but one of the ring is the last the run has not moved
        const bool in = lane < 31 && (uint32_t)(n0 + lane) + 1u < len && k.towards(idn, bb);
        const bool nsc = in && ownn >= OWN_ACTIVE;
        double dx = __dsub_rn(xn, x);
        // (a target with a time of this leg, before whose pass there are none: an
        // assertion on Eq. 2 below)
        const bool neg = __double_as_longlong(dx) < 0, timed = in && ownn == s.stamp;
        const bool any_odd = __any_sync(FULL, neg || timed);
        if (any_odd && neg) dx = g_add(dx, L);
        double tau = __dsub_rn(dx, bb);
        if (__double_as_longlong(tau) < 0) tau = 0.0;
        const unsigned stops = __ballot_sync(FULL, lane < 31 && (nsc || !in));
        g_sums(tau, stops ? __ffs(stops) - 1 : 31, t, D);
        const bool lift = dbits(tau) < dbits(D);
        const unsigned fin = __ballot_sync(FULL, lane < 31 && (!in || nsc || !lift));
        const int f = fin ? __ffs(fin) - 1 : 31;  // the event that ends the run, or none
        const bool round = fin && !__shfl_sync(FULL, (int)in, f);
        const bool met = fin && !round && __shfl_sync(FULL, (int)lift, f);  // lift onto an active disk
        if (any_odd) {
            const double rt = shfl_f64(k.t, (lane + 1) & 31);
            if (timed && lane <= f && dbits(g_add(t, tau)) < dbits(rt))
                atomicAdd(s.lc + LC_HORIZON, 1ull);
        }
        n = n0 + f + (fin && !met ? 1 : 0);
        if ((round && len > 1) || n >= s.cap) {
            if (lane == 0 && round) atomicAdd(s.lc + LC_RINGLAP, 1ull);
            return false;
        }
        // events n0 .. n - 1
        const int e = n0 + lane;
        const bool has = e < n, stall = has && lane == f;
        const double ts = stall ? D : tau;
        const double tn_lift = shfl_f64(t, (lane + 1) & 31), dn_lift = shfl_f64(D, (lane + 1) & 31);
        const double tn_stall = __dadd_rn(t, D);
        double xe = __dadd_rn(x, ts);
        const bool wrap = has && dbits(xe) >= dbits(L);
        if (__any_sync(FULL, wrap) && wrap) xe = g_sub(xe, L);
        const double tn = stall ? tn_stall : tn_lift;
        if (s.cells && (has || (met && lane == f))) {
            const size_t at = (size_t)e * (size_t)s.k + (size_t)c;
            s.pxt[at] = make_double2(x, has ? ts : D);
            s.pcell[at] = row * (uint32_t)s.nc + (uint32_t)cell_coord(x, s.inv_a, s.nc);
        }
        if (has) {
            ulonglong2 *u = reinterpret_cast<ulonglong2 *>(grec_at(s, c, e));
            u[0] = make_ulonglong2((unsigned long long)id |
                                       ((unsigned long long)(stall ? NONE : idn) << 32),
                                   (unsigned long long)(uint32_t)e);
            u[1] = make_ulonglong2(dbits(x), dbits(t));
            u[2] = make_ulonglong2(0ull, dbits(tn));
            u[3] = make_ulonglong2(dbits(ts), dbits(xe));
            u[4] = make_ulonglong2(stall ? 0ull : dbits(xn), stall ? 0ull : dbits(dn_lift));
            if (!stall) {
                *gpath_at(s, c, e + 1) = idn;
                red_min_u64(s.key + idn, g_key(tn, c));
            }
        }
        if (fin) {
            end = met ? SP_NONSTATIC : SP_STALL;
            if (met) partner = __shfl_sync(FULL, ownn, f) & OWN_CHAIN;
            iend = __shfl_sync(FULL, id, f);
            t = shfl_f64(met ? t : tn, f);
            D = met ? shfl_f64(D, f) : 0.0;
            break;
        }
        t = shfl_f64(t, 31);
        D = shfl_f64(D, 31);
    }
    if (lane == 0) {
        GSpec r;
        r.n = n;
        r.touch = end == SP_STALL ? n : n + 1;
        r.end = end;
        r.partner = partner < (uint32_t)s.k ? (int32_t)partner : -1;
        r.tc = t;
        r.D = D;
        r.ci = iend;
        r.cut = end == SP_STALL ? 0x7FFFFFFF : n;
        r.pad[0] = r.pad[1] = 0;
        s.sp[c] = r;
    }
    __syncwarp();
    return true;
}

// Touch keys of chain c back to empty (one warp): every disk its last run
// alone posted a key for.
__device__ __forceinline__ void g_reset_keys(const GDev &s, int c, int lane) {
    const int nt = s.sp[c].touch;
    unsigned long long *const key = s.key;
    for (int e = lane; e < nt; e += 32) {
        const uint32_t id = *gpath_at(s, c, e);
        key[id] = ~0ull;
        if (s.strict) {
            const GDisk &r = s.g[id];
#pragma unroll
            for (int z = 0; z < 3; ++z)
                if (r.a[z] != NONE) key[r.a[z]] = ~0ull;
        }
    }
}

// The conflict flag (one warp, after the pass): chain c puts its word (epoch,
// chain) into s.fl for every disk its run alone read, its start disk and the
// arrow targets of every disk that was active -- or, for a cell-scan context,
// for every cell its scans covered. Two chains read one disk (scanned one
// cell) iff one of them is handed the other's word of this epoch; the epoch
// makes clearing unnecessary. Nothing waits for the result before the leg's
// totals, so the warps without a component do this while the others repair.
//
// The scan of a step covers rows cy - 1 .. cy + 1 and columns cx, cx + 1, ...
// up to the first m >= 1 whose threshold exceeds min(D, best) + eps. The
// cell scan forms best column by column; the columns up to the winner's have
// thresholds within the winner's time of flight (less a rounding far below
// eps), so the final best gives the same columns.
__device__ __noinline__ void g_flag_chain(const GDev &s, int c, uint32_t epoch, int lane) {
    const int nt = s.sp[c].touch;
    const unsigned long long tag = ((unsigned long long)epoch << 32) | ((unsigned)c + 1u);
    bool met = false;
    auto foreign = [&](unsigned long long w) {
        return (uint32_t)(w >> 32) == epoch && (uint32_t)w != (uint32_t)tag;
    };
    for (int e = lane; e < nt; e += 32) {
        const size_t at = (size_t)e * (size_t)s.k + (size_t)c;
        if (!s.cells) {
            const uint32_t id = s.path[at];
            const GDisk &r = s.g[id];
            uint32_t a[4] = {r.a[0], r.a[1], r.a[2], e == 0 ? id : NONE};
            unsigned long long w[4];
#pragma unroll
            for (int z = 0; z < 4; ++z) w[z] = a[z] != NONE ? atomicExch(s.fl + a[z], tag) : 0ull;
#pragma unroll
            for (int z = 0; z < 4; ++z) met |= foreign(w[z]);
            continue;
        }
        const double2 xt = s.pxt[at];
        const uint32_t cell = s.pcell[at];
        const int nc = s.nc, cy = (int)(cell / (uint32_t)nc), cx = (int)(cell % (uint32_t)nc);
        const double fx = __dsub_rn(xt.x, __dmul_rn((double)cx, s.sk.a));
        const float fxf = d2f_trunc(fx), lim_f = __fadd_rn(d2f_trunc(xt.y), s.sk.epsf);
        const int rdn = cy == 0 ? nc - 1 : cy - 1, rup = cy == nc - 1 ? 0 : cy + 1;
        unsigned long long *const f0 = s.fl + (size_t)rdn * (size_t)nc,
                                  *const f1 = s.fl + (size_t)cy * (size_t)nc,
                                  *const f2 = s.fl + (size_t)rup * (size_t)nc;
        bool more = true;
        for (int m0 = 0; more && m0 < nc; m0 += 3) {
            unsigned long long w[9];
#pragma unroll
            for (int z = 0; z < 3; ++z) {
                const int m = m0 + z;
                if (m >= nc ||
                    (m > 0 && more && beyond_k(s.sk, m, fx, fxf, lim_f, dbits(xt.y))))
                    more = false;
                int col = cx + m;
                if (col >= nc) col -= nc;
                w[3 * z] = more ? atomicExch(f0 + col, tag) : 0ull;
                w[3 * z + 1] = more ? atomicExch(f1 + col, tag) : 0ull;
                w[3 * z + 2] = more ? atomicExch(f2 + col, tag) : 0ull;
            }
#pragma unroll
            for (int z = 0; z < 9; ++z) met |= foreign(w[z]);
        }
    }
    if (__any_sync(FULL, met) && lane == 0) {
        atomicAdd(s.lc + LC_WEAK, 1ull);
        atomicAdd(s.lc + LC_WWEAK, 1ull);
    }
}

// After the pass (one warp): the first step of chain c's run that touches a
// disk another chain holds, the events before it published, the chain's
// state, the claims of the touched disks.
//
// The least key (earliest touch, then lower chain) holds a disk; a chain is
// cut at its first step that lifts onto a disk it does not hold. Published
// events are therefore on disks that no other chain's published events
// touch, and that makes them exact. Take the first event, in global time, at
// which a published chain A would differ from its run alone. A's disk is
// where it was in that run. A candidate that nobody touched before is where
// A read it; one that others touched lies farther ahead (motion is along +x,
// and no disk passes another within d of it in y) or is active; a disk that
// was active at the window's start lies no nearer than the winner or beyond
// reach there, or the run ended (SP_NONSTATIC). The winner itself A holds. So
// the least time of flight is the one of the run alone: no difference. What
// a chain only reads needs no claim of its own. (The repair's continuation
// claims what it reads: there a disk may already lie where another chain
// moved it at a later time.)
//
// With the claims on every disk read (three per event) 508 of 2048 chains on
// 262144 dense disks were blocked per leg; touched disks alone: about a
// third of that.
// Blocked chains of a pass, over all systems: chain f (numbered over the
// systems) is entry *cnt - base of list.
struct GBlocked {
    unsigned *cnt;
    int32_t *list;
    unsigned base;
};

// A pass's components start as single chains with final events (one warp).
__device__ __forceinline__ void g_begin_pass(const GDev &s, int c, int lane) {
    if (lane < 6) {
        int32_t *const a[6] = {s.uf, s.comp_of, s.fin, s.abort_to, s.child, s.ctl};
        const int32_t v[6] = {c, c, 1, -1, -1, 0};
        int32_t *p = a[0];
        int32_t w = v[0];
#pragma unroll
        for (int z = 1; z < 6; ++z) {
            p = lane == z ? a[z] : p;
            w = lane == z ? v[z] : w;
        }
        if (lane < 5) p[c] = w;
        if (lane == 5 && c == 0) {
            p[CTL_NABORT] = 0;
            p[CTL_NMEMB] = 0;
        }
    }
}

// The root of chain c's tree (no path is shortened: the trees stay as hooked).
__device__ __forceinline__ int g_root(const GDev &s, int c) {
    for (;;) {
        const int p = ((volatile int32_t *)s.uf)[c];
        if (p == c) return c;
        c = p;
    }
}

// A chain blocked by the pass (one thread): counted, listed for the repair,
// and in one component with its partner from here on. The component's members
// are its root's tree: a hooked root goes on its new root's list of children.
__device__ void g_note_blocked(const GDev &s, int c, int32_t partner, int f, const GBlocked &bl) {
    const unsigned ix = atomicAdd(bl.cnt, 1u) - bl.base;
    atomicAdd(s.lc + LC_BLOCKED, 1ull);
    atomicAdd(s.lc + LC_WBLOCKED, 1ull);
    s.fin[c] = 0;
    if (partner >= 0 && partner < s.k) {
        s.fin[partner] = 0;
        int a = c, b = partner;
        for (;;) {
            a = g_root(s, a);
            b = g_root(s, b);
            if (a == b) break;
            const int lo = min(a, b), hi = max(a, b);
            if (atomicCAS(s.uf + hi, hi, lo) == hi) {
                s.sib[hi] = atomicExch(s.child + lo, hi);
                break;
            }
        }
    }
    bl.list[ix] = f;
}

__device__ __noinline__ void g_resolve_chain(const GDev &s, int c, double tw, uint32_t epoch, int f,
                                             const GBlocked &bl) {
    const int lane = threadIdx.x & 31;
    // the chain's state and the first touched disks in one round of loads
    const GSpec sp = s.sp[c];
    const int32_t st0 = s.status[c], nr0 = s.nrec[c];
    uint32_t pid = lane < s.cap ? *gpath_at(s, c, lane) : NONE;
    if (st0 != ST_RUNNING) return;
    const int n = sp.n, nt = sp.touch, end = sp.end & SP_END;
    const bool serial = (sp.end & SP_LAP) != 0;
    const unsigned long long tag = ((unsigned long long)epoch << 32) | ((unsigned)c + 1u);
    int sfail = n;
    bool lost = false;
    uint32_t holder = NONE;
    for (int e0 = 0; e0 < nt && !lost; e0 += 32) {
        const int e = e0 + lane;
        // the first step this entry loses: its touch (by the step before), or
        // (strict) a read of the step it is active in
        int st = 0x7FFFFFFF;
        uint32_t h = NONE;
        if (e < nt) {
            const uint32_t id = e0 == 0 && lane < s.cap ? pid : *gpath_at(s, c, e);
            if (s.strict) {
                const GDisk &r = s.g[id];
#pragma unroll
                for (int z = 0; z < 3; ++z)
                    if (r.a[z] != NONE) {
                        const uint32_t hz = (uint32_t)__ldcg(s.key + r.a[z]);
                        if (hz != (uint32_t)c) {
                            st = e;
                            h = hz;
                        }
                    }
            }
            const uint32_t ht = (uint32_t)__ldcg(s.key + id);
            if (ht != (uint32_t)c) {
                st = e > 0 ? e - 1 : 0;
                h = ht;
            }
        }
        const int first = __reduce_min_sync(FULL, st);
        if (first != 0x7FFFFFFF) {
            const unsigned hm = __ballot_sync(FULL, st == first);
            holder = __shfl_sync(FULL, h, __ffs(hm) - 1);
            lost = true;
            sfail = first < n ? first : n;
        }
    }
    if (sp.cut <= sfail) {
        sfail = sp.cut;
        lost = true;
        holder = (uint32_t)sp.partner;
    }
    // publish records 0 .. sfail - 1; the lane of the last one keeps its time
    // and remaining length for the chain's state
    int lifts = 0;
    double lt = 0.0, ld = 0.0;
    for (int e0 = 0; e0 < sfail; e0 += serial ? 1 : 32) {
        const int e = e0 + lane;
        const bool mine = serial ? lane == 0 : e < sfail;
        uint32_t rj = NONE;
        if (mine) {
            const ulonglong2 *u = reinterpret_cast<const ulonglong2 *>(grec_at(s, c, nr0 + e));
            const ulonglong2 u0 = u[0], u2 = u[2], u3 = u[3], u4 = u[4];
            rj = (uint32_t)(u0.x >> 32);
            GDisk &r = s.g[(uint32_t)u0.x];
            *reinterpret_cast<ulonglong2 *>(&r.x) = make_ulonglong2(u3.y, u2.y);
            r.own = rj != NONE ? s.stamp : (OWN_STALLED | (uint32_t)c);
            r.claim = tag;
            lt = __longlong_as_double((long long)u2.y);
            ld = __longlong_as_double((long long)u4.y);
        }
        lifts += __popc(__ballot_sync(FULL, mine && rj != NONE));
        if (serial) __syncwarp();
    }
    const int ll = serial ? 0 : (sfail + 31) & 31;
    lt = shfl_f64(lt, ll);
    ld = shfl_f64(ld, ll);
    __syncwarp();
    if (lane == 0) {
        int st;
        uint32_t id;
        double tc, D;
        int32_t partner = -1;
        if (sfail < n) {
            id = *gpath_at(s, c, sfail);
            tc = sfail > 0 ? lt : s.tc[c];
            D = sfail > 0 ? ld : s.D[c];
            st = ST_BLOCKED;
            partner = (int32_t)holder;
        } else {
            id = sp.ci;
            tc = sp.tc;
            D = sp.D;
            st = end == SP_STALL ? ST_STALLED : ST_RUNNING;
            if (lost) {
                st = ST_BLOCKED;
                partner = (int32_t)holder;
            } else if (end == SP_NONSTATIC || end == SP_LIMIT) {
                st = ST_BLOCKED;
                partner = sp.partner;
            }
        }
        if (st != ST_STALLED) {
            GDisk &r = s.g[id];
            if (sfail > 0) {
                r.own = OWN_ACTIVE | (uint32_t)c;
                r.t = tc;
            }
            r.claim = tag;
        }
        s.ci[c] = id;
        s.tc[c] = tc;
        s.D[c] = D;
        s.status[c] = st;
        s.nrec[c] = nr0 + sfail;
        s.nlift[c] += lifts;
        s.partner[c] = partner;
        // events before the blocking time, and all before the window, are exact
        s.vt[c] = st == ST_BLOCKED ? fmax(tc, tw) : INFINITY;
        if (st == ST_BLOCKED) g_note_blocked(s, c, partner, f, bl);
        if (lifts) atomicAdd(s.lc + LC_P1LIFTS, (unsigned long long)lifts);
    }
    __syncwarp();
}

// ------------------------------------------------------------ repair steps

// Claims disk id for the pass (tag: epoch << 32 | chain + 1): the word of the
// chain that holds it in this epoch (chain + 1; that stays), or 0. A word of an
// earlier epoch is free, so nothing has to be cleared between passes.
__device__ __forceinline__ uint32_t g_holder(unsigned long long w, unsigned long long tag) {
    return (uint32_t)(w >> 32) == (uint32_t)(tag >> 32) ? (uint32_t)w : 0u;
}
__device__ __forceinline__ uint32_t g_claim(const GDev &s, uint32_t id, unsigned long long tag) {
    const unsigned long long w = __ldcg(&s.g[id].claim);
    const uint32_t h = g_holder(w, tag);
    return h ? h : g_holder(atomicCAS(&s.g[id].claim, w, tag), tag);
}

// What one step found.
struct GStep {
    double tau;        // tau* (lift) or D (stall)
    uint32_t j;        // target (lift)
    int lift;
    double xj, tj;     // the target's x and local time as read
    int conflict;      // a disk read is held by a chain of the other side
    uint32_t partner;  // that chain
};

// Is chain h, which holds a claim a repair step met, on the repairing side?
// Yes if this round's component lists it (memb == tag); with adopt, also if
// it was, or now is, taken over: a chain in no component of this round whose
// events are final since the round began joins the component (and any later
// merge that reaches the component takes it along: the next round's union-find
// adds it from comp_of).
__device__ __forceinline__ bool holder_ours(const GDev &s, int h, int root, uint64_t tag,
                                            bool adopt) {
    if (h < 0 || h >= s.k) return false;
    if (__ldcg((const unsigned long long *)s.memb + h) == tag) return true;
    if (!adopt) return false;
    int hc = __ldcg(s.comp_of + h);
    if (hc == h && h != root && __ldcg(s.fin + h) == 1) {
        const int prev = atomicCAS(s.comp_of + h, h, root);
        hc = prev == h ? root : prev;
    }
    return hc == root;
}

// The next event of chain c in a replay (Sec. 2.2) along the arrows a[] (with
// b[]) of its active disk i at x_i, t_i, with remaining length D. Every disk
// read -- i and the arrow targets -- is claimed for the pass, together with
// the loads; what was read is used only once the claims stand. A claim of
// another chain is a conflict unless that chain is listed in this round's
// component (memb == tag). (all: every chain is, nothing to claim.) Candidates are
// the static targets (Alg. 2: j not
// active); a target with t_i + tau < t_j became static after chain c's disk
// had passed it and is one lap away (lazy per-chain frame); ties go to the
// lower disk index.
__device__ GStep graph_step(const GDev &s, int c, int root, uint64_t tag, uint32_t epoch,
                            bool all, const uint32_t a[3], const double b[3], uint32_t i,
                            double xi, double ti, double D) {
    const uint32_t mine = (uint32_t)c + 1u;
    const unsigned long long ct = ((unsigned long long)epoch << 32) | mine;
    uint32_t old[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (!all && a[q] != NONE) old[q] = g_claim(s, a[q], ct);
    if (!all) old[3] = g_claim(s, i, ct);
    GDisk r[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (a[q] != NONE) r[q] = s.g[a[q]];
    GStep o;
    o.conflict = 0;
    o.partner = NONE;
    // time of flight to each static target (Sec. 2.2): forward image in x,
    // b_ij fixed with the arrow, clamped at 0
    unsigned long long bt = INF_BITS;
    int bq = -1;
    uint32_t bjid = NONE;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (g_open(a[q], b[q])) {  // (as a target at its place)
            double dx = __dsub_rn(g_unsigned(b[q]), xi);
            if (dneg(dx)) dx = __dadd_rn(dx, s.L);
            if (bq < 0 || dbits(dx) < bt) {
                bt = dbits(dx);
                bq = q;
                bjid = NONE;
            }
            continue;
        }
        if (a[q] == NONE || !g_static(r[q].own)) continue;
        const double rt = g_time(r[q].own, r[q].t, s.stamp);
        double dx = __dsub_rn(r[q].x, xi);
        if (dneg(dx)) dx = __dadd_rn(dx, s.L);
        double tau = __dsub_rn(dx, b[q]);
        if (dneg(tau)) tau = 0.0;
        if (dbits(rt) != 0ull && dbits(__dadd_rn(ti, tau)) < dbits(rt)) tau = __dadd_rn(tau, s.L);
        const unsigned long long tb = dbits(tau);
        if (bq < 0 || tb < bt || (tb == bt && a[q] < bjid)) {
            bt = tb;
            bq = q;
            bjid = a[q];
        }
    }
    // the claims: a taken one names the chain that holds the disk
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t w = old[q];
        if (w == 0u || w == mine) continue;
        const int h = (int)w - 1;
        if (holder_ours(s, h, root, tag, false)) continue;
        if (!o.conflict) {
            o.conflict = 1;
            o.partner = (uint32_t)h;
        }
    }
    if (bq >= 0 && bt < dbits(D) && bjid == NONE) g_undecided(s);
    if (bq >= 0 && bt < dbits(D) && bjid != NONE) {
        o.lift = 1;
        o.tau = __longlong_as_double((long long)bt);
        o.j = bjid;
        // selects, not an indexed (local-memory) load
        o.xj = bq == 0 ? r[0].x : bq == 1 ? r[1].x : r[2].x;
        o.tj = bq == 0   ? g_time(r[0].own, r[0].t, s.stamp)
               : bq == 1 ? g_time(r[1].own, r[1].t, s.stamp)
                         : g_time(r[2].own, r[2].t, s.stamp);
    } else {
        o.lift = 0;
        o.tau = D;
        o.j = NONE;
        o.xj = o.tj = 0.0;
    }
    return o;
}

// Executes chain c's step from disk i (a lifting, Eq. 1, or a stall at the
// breakpoint) and writes its record at index nr (the caller checked the
// capacity and counts records and liftings).
__device__ void graph_apply(const GDev &s, int c, uint32_t i, double xi, double ti, double D,
                            int lift, uint32_t j, double tau, double xj, double tj,
                            uint32_t seq, int32_t nr) {
    GEv u;
    u.i = i;
    u.seq = seq;
    u.pad = 0;
    u.x_old = xi;
    u.ti_old = ti;
    GDisk &ri = s.g[i];
    if (lift) {
        const double tnew = __dadd_rn(ti, tau);       // new t_j = new t_i (before x, Remark 11)
        const double xnew = wrap_add(xi, tau, s.L);   // i moves to contact
        GDisk &rj = s.g[j];
        rj.own = OWN_ACTIVE | (uint32_t)c;             // j active (the claim holds j)
        rj.t = tnew;
        ri.t = tnew;
        ri.x = xnew;
        ri.own = s.stamp;                              // i static
        u.j = j;
        u.tj_old = tj;
        u.t = tnew;
        u.tau = tau;
        u.xi = xnew;
        u.xj = xj;
        u.d_after = __dsub_rn(D, tau);                 // remaining length
    } else {
        const double tnew = __dadd_rn(ti, D);         // t_i reaches the breakpoint
        const double xnew = wrap_add(xi, D, s.L);     // i moves by D
        ri.x = xnew;
        ri.t = tnew;
        ri.own = OWN_STALLED | (uint32_t)c;           // stalled
        u.j = NONE;
        u.tj_old = 0.0;
        u.t = tnew;
        u.tau = D;
        u.xi = xnew;
        u.xj = 0.0;
        u.d_after = 0.0;                              // no length left
    }
    *grec_at(s, c, nr) = u;
}

// ------------------------------------------------------------------ legs

// The lifting log of the leg (one warp), in the chain's order.
__device__ __noinline__ void g_log_chain(const GDev &s, int c, int32_t leg, int lane) {
    const int32_t nl = s.nlift[c];
    if (nl > 0) {
        unsigned long long w = 0ull;
        if (lane == 0) w = atomicAdd(s.tc_cnt + TC_LOG_N, (unsigned long long)nl);
        w = shfl_u64(w, 0);
        const int32_t nr = s.nrec[c];
        for (int32_t e0 = 0; e0 < nr; e0 += 32) {
            const int32_t e = e0 + lane;
            const GEv *u = grec_at(s, c, e < nr ? e : 0);
            const bool is = e < nr && u->j != NONE;
            const unsigned m = __ballot_sync(FULL, is);
            const unsigned long long at = w + __popc(m & ((1u << lane) - 1u));
            if (is && (int64_t)at < s.log_cap) {
                ecmc_lift_t Lr;
                Lr.leg = leg;
                Lr.c = c;
                Lr.i = (int32_t)u->i;
                Lr.j = (int32_t)u->j;
                Lr.t = u->t;
                Lr.tau = u->tau;
                Lr.xi = u->xi;
                Lr.xj = u->xj;
                s.log[at] = Lr;
            }
            w += __popc(m);
        }
    }
}

// --------------------------------------------------------------- repairs

// Exact inverse of graph_apply for one record of chain c.
__device__ void g_undo(const GDev &s, int c, const GEv &u) {
    GDisk &ri = s.g[u.i];
    ri.x = u.x_old;
    ri.t = u.ti_old;
    ri.own = OWN_ACTIVE | (uint32_t)c;
    if (u.j != NONE) {
        GDisk &rj = s.g[u.j];
        rj.t = u.tj_old;
        rj.own = s.stamp;
        s.nlift[c] -= 1;
        atomicAdd(s.lc + LC_LIFTS, ~0ull);
    }
}

// Rolls the members of a component back to T* (their events before T* are
// exact): records with event time >= T* are undone, latest first. Records of
// repair rounds (seq >= REPAIR_SEQ0) may touch one disk from several members
// and are undone one at a time in descending seq; beneath them, the records
// of the window's parallel pass touch disks held by their own chain only,
// so each member undoes its own in parallel.
__device__ __noinline__ void g_rollback(const GDev &s, const int32_t *mem, int m, double Ts) {
    const int lane = threadIdx.x & 31;
    if (m <= 32) {
        // a member per lane, its last record in registers: an undo waits for
        // the member's next record at most
        const int c = lane < m ? mem[lane] : 0;
        int32_t nr = lane < m ? s.nrec[c] : 0;
        GEv u;
        bool top = false;  // u is a repair record to undo
        auto load = [&]() {
            top = false;
            if (nr > 0) {
                u = *grec_at(s, c, nr - 1);
                top = u.t >= Ts && u.seq >= REPAIR_SEQ0;
            }
        };
        load();
        for (;;) {
            const unsigned best = __reduce_max_sync(FULL, top ? u.seq : 0u);
            if (best == 0u) break;
            const unsigned bm = __ballot_sync(FULL, top && u.seq == best);
            if (lane == __ffs(bm) - 1) {
                g_undo(s, c, u);
                --nr;
                load();
            }
            __syncwarp();
        }
        if (lane < m) s.nrec[c] = nr;
        __syncwarp();
    } else {
        for (;;) {
            uint32_t bseq = 0;
            int bmem = -1;
            for (int e = lane; e < m; e += 32) {
                const int c = mem[e];
                const int32_t nr = s.nrec[c];
                if (nr == 0) continue;
                const GEv &u = *grec_at(s, c, nr - 1);
                if (!(u.t >= Ts) || u.seq < REPAIR_SEQ0) continue;
                if (bmem < 0 || u.seq > bseq || (u.seq == bseq && e < bmem)) {
                    bseq = u.seq;
                    bmem = e;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint32_t s2 = __shfl_xor_sync(FULL, bseq, o);
                const int m2 = __shfl_xor_sync(FULL, bmem, o);
                if (m2 >= 0 && (bmem < 0 || s2 > bseq || (s2 == bseq && m2 < bmem))) {
                    bseq = s2;
                    bmem = m2;
                }
            }
            if (bmem < 0) break;
            if (lane == 0) {
                const int c = mem[bmem];
                const int32_t nr = s.nrec[c];
                g_undo(s, c, *grec_at(s, c, nr - 1));
                s.nrec[c] = nr - 1;
            }
            __syncwarp();
        }
    }
    for (int e = lane; e < m; e += 32) {
        const int c = mem[e];
        int32_t nr = s.nrec[c];
        while (nr > 0) {
            const GEv &u = *grec_at(s, c, nr - 1);
            if (!(u.t >= Ts)) break;
            g_undo(s, c, u);
            --nr;
        }
        s.nrec[c] = nr;
    }
    __syncwarp();
}

// State of chain c after its last kept record (or at the leg start).
__device__ void g_resume(const GDev &s, int c) {
    const int32_t nr = s.nrec[c];
    if (nr == 0) {
        s.ci[c] = s.ci0[c];
        s.tc[c] = 0.0;
        s.D[c] = s.ell;
        s.status[c] = ST_RUNNING;
        return;
    }
    const GEv &u = *grec_at(s, c, nr - 1);
    if (u.j == NONE) {
        s.ci[c] = u.i;
        s.tc[c] = u.t;
        s.D[c] = 0.0;
        s.status[c] = ST_STALLED;
    } else {
        s.ci[c] = u.j;
        s.tc[c] = u.t;
        s.D[c] = u.d_after;
        s.status[c] = ST_RUNNING;
    }
}

// Pending event of member c (one thread), kept with the arrows it read.
__device__ __noinline__ void g_compute(const GDev &s, int c, int root, uint64_t tag,
                                       uint32_t epoch, bool all, bool &abort, int &met) {
    const uint32_t i = s.ci[c];
    const GDisk ri = s.g[i];
    const double ti = s.tc[c], D = s.D[c];
    const GStep o = graph_step(s, c, root, tag, epoch, all, ri.a, ri.b, i, ri.x, ti, D);
    if (o.conflict && !abort) {
        abort = true;
        met = (int)o.partner;
    }
    s.ev_T[c] = __dadd_rn(ti, o.tau);
    s.ev_tau[c] = o.tau;
    s.ev_j[c] = o.j;
    s.ev_lift[c] = o.lift;
    s.ev_xj[c] = o.xj;
    s.ev_tj[c] = o.tj;
#pragma unroll
    for (int q = 0; q < 3; ++q) s.ev_a[4 * (size_t)c + q] = ri.a[q];
}

// Restart mode: chain c back to time Ts. Its records at or after Ts are all
// of the current pass, whose disks each chain held alone, so every chain
// undoes its own (latest first) in parallel with the others.
__device__ void g_rollback_chain(const GDev &s, int c, double Ts) {
    int32_t nr = s.nrec[c];
    while (nr > 0) {
        const GEv &u = *grec_at(s, c, nr - 1);
        if (!(u.t >= Ts)) break;
        g_undo(s, c, u);
        --nr;
    }
    s.nrec[c] = nr;
    g_resume(s, c);
}

// After a component's replay: record abort or success for the next round.
// keep_vt (success by continuation): the members' vt becomes `now` instead of
// infinity, so that a later merge rolls them back to `now` or earlier (their
// events were applied chain by chain, not in time order).
__device__ void g_finish(const GDev &s, const int32_t *mem, int m, int root, bool abort,
                         int met, double now, bool keep_vt = false) {
    const int lane = threadIdx.x & 31;
    if (abort) {
        // events before `now` are exact; the chain met joins next round
        for (int e = lane; e < m; e += 32) s.vt[mem[e]] = now;
        if (lane == 0) {
            if (met >= 0 && met < s.k) {
                s.abort_to[root] = met;
                atomic_min_time(s.vt + met, now);
            }
            atomicAdd(s.ctl + CTL_NABORT, 1);
        }
    } else {
        for (int e = lane; e < m; e += 32) {
            s.fin[mem[e]] = 2;
            s.vt[mem[e]] = keep_vt ? now : INFINITY;
        }
    }
    __syncwarp();
}

// First repair round of a window, and later ones of a leg without windows: the
// blocked members continue from where they stopped, one after another (one
// warp), over the state the others left. What the pass published is a run of
// Alg. 4 (g_resolve_chain); so is what components did that met each other in
// the last round, whose events are on disks that only their own chains hold.
// (Rolling a merged component back instead: 83 us for a second round, on 97% of
// the legs of 2048 chains on 262144 dense disks.) If every
// continued step satisfies Eq. 2 on each arrow target as well, the whole is a
// run of Alg. 4 without a horizon violation, which by Lemma 2 ends where
// Alg. 2 ends: nothing has to be redone. A chain that finds the active disk of
// another blocked member among its arrow targets waits (Remark 10) while that
// member continues first. Otherwise the caller rolls the component back to T*
// and replays it in global order. The lanes share a step as in g_spec_chain;
// a step's claims are asked about one step later, when their round trip is
// over, and an event is written only once they stand.
//
// The disks that the continuation moves it holds, and one that another
// component holds ends it. A disk that it only reads need not be held (as in
// g_resolve_chain; strict: it is): nobody has touched it in this leg, and
// whatever moves it, at whatever time, moves it farther ahead of a disk whose
// target it was not. With every disk read held 30% more continuations met
// another component.
enum { CONT_DONE = 0, CONT_FAIL = 1, CONT_FOREIGN = 2 };

template <bool OPEN>
__device__ __noinline__ int g_continue(const GDev &s, const int32_t *mem, int m, int root,
                                       uint64_t tag, uint32_t epoch, int round, double tw,
                                       double tend, int *met, uint32_t *cnt_out) {
    const int lane = threadIdx.x & 31;
    const int l3 = lane % 3;
    const double L = s.L;
    GLevels &lv = g_levels();
    GDisk *const g = s.g;
    const uint32_t stamp = s.stamp;
    const bool bounded = dbits(tend) != INF_BITS || dbits(tw) != 0ull;
    const bool strict = s.strict != 0;
    const int n_lap = g_lap(s), cap = s.cap;
    uint32_t cnt = 0;
    int switches = 0, e = 0, cur = -1;
    int known = -1;  // a holder already found on this side
    for (;;) {
        if (cur < 0) {  // the next member still blocked
            while (e < m) {
                const unsigned bm =
                    __ballot_sync(FULL, e + lane < m && s.status[mem[e + lane]] == ST_BLOCKED);
                if (bm) {
                    e += __ffs(bm) - 1;
                    break;
                }
                e += 32;
            }
            if (e >= m) {
                *cnt_out = cnt;
                return CONT_DONE;
            }
            cur = mem[e];
        }
        const int c = cur;
        const uint32_t mine = (uint32_t)c + 1u;
        const unsigned long long ct = ((unsigned long long)epoch << 32) | mine;
        uint32_t i = s.ci[c];
        double ti = s.tc[c], D = s.D[c];
        const int32_t nr0 = s.nrec[c];
        const uint32_t seq0 = ((uint32_t)round << 24) | cnt;
        double xi = g[i].x;
        int cb = 0, sl = 0;  // the active disk's targets: lv.r[cb][sl .. sl + 2]
        g_fetch_first(g, i, lv.r[0]);
        uint32_t tid = g[i].a[l3];
        double tb = g[i].b[l3];
        unsigned none = g_none(tid);
        // the holder of a disk this lane claimed, asked one step later: what the
        // exchange found (0: free, mine), or the record's own word of this pass
        unsigned long long cas = 0ull;
        uint32_t held = 0u;
        if (lane == 31) held = g_claim(s, i, ct);
        // false: a disk read in the step before is held by the other side
        auto claims_stand = [&]() -> bool {
            const uint32_t h = held ? held : g_holder(cas, ct);
            const bool ask = h != 0u && h != mine && (int)h - 1 != known;
            if (!__any_sync(FULL, ask)) return true;
            const bool ours = !ask || holder_ours(s, (int)h - 1, root, tag, true);
            const unsigned fb = __ballot_sync(FULL, !ours);
            if (fb) {
                *met = (int)__shfl_sync(FULL, h, __ffs(fb) - 1) - 1;
                return false;
            }
            const unsigned ab = __ballot_sync(FULL, ask);
            known = (int)__shfl_sync(FULL, h, __ffs(ab) - 1) - 1;
            return true;
        };
        g_copy_wait();
        bool op = OPEN && g_open(tid, tb);
        if (OPEN && none) {
            g_open_targets(tid, tb, lv.r[0]);
            if (op) tb = 0.0;
        }
        GEvs E;
        E.i = NONE;
        E.x = E.t = E.D = E.tau = E.tj = 0.0;
        int n = 0, nf = 0, nl = 0, st = ST_RUNNING, next = -1, how = CONT_DONE;
        // events nf .. n - 1 to memory: records and the moved disks
        auto flush = [&](bool lift) {
            if (n == nf) return;
            const GFlush f = g_flush(s, c, nr0, seq0, nf, n, E, i, xi, ti, D, lift);
            if (f.has) {
                *reinterpret_cast<ulonglong2 *>(&g[E.i].x) =
                    make_ulonglong2(dbits(f.xn), dbits(f.t));
                g[E.i].own = f.j != NONE ? stamp : (OWN_STALLED | (uint32_t)c);
            }
            nf = n;
        };
        // back to the state before event n - 1
        auto drop = [&]() {
            --n;
            const int le = n & 31;
            i = __shfl_sync(FULL, E.i, le);
            xi = shfl_f64(E.x, le);
            ti = shfl_f64(E.t, le);
            D = shfl_f64(E.D, le);
        };
        for (;;) {
            const GDisk *const R = &lv.r[cb][sl];
            g_fetch(g, R, none, lv.r[cb ^ 1]);
            const bool ev = lane < 3 && tid != NONE;
            const bool evo = lane < 3 && (tid != NONE || (OPEN && op));
            const double rx = R[l3].x, rt = R[l3].t;
            const uint32_t own = R[l3].own;
            const unsigned long long cw = R[l3].claim;
            double dx = __dsub_rn(rx, xi);
            double tau = __dsub_rn(dx, tb);
            // the claims of the step before: if one failed, its event is none
            // (not written yet) and the component has met another chain
            if (!claims_stand()) {
                how = CONT_FOREIGN;
                if (n > nf) {
                    drop();
                    --nl;
                }
                break;
            }
            // this step's claims: a record whose word is of this pass names its
            // holder; of the others the winner is taken, once it is known
            // (strict: all), and the words of the rest are read again -- one that
            // is still free stands for a record that was not written
            held = ev ? g_holder(cw, ct) : 0u;
            cas = 0ull;
            if (strict && ev && held == 0u) cas = atomicCAS(&g[tid].claim, cw, ct);
            // Eq. 2, strict (a lap-away target fails it too), for every target
            // with a time of this leg; another chain's disk stops the step in
            // reach or where it fails Eq. 2
            double sum = __dadd_rn(ti, __double_as_longlong(tau) < 0 ? 0.0 : tau);
            const bool nsc = ev && own >= OWN_ACTIVE;
            const bool neg = evo && __double_as_longlong(dx) < 0;
            bool bad = ev && own == stamp && dbits(rt) != 0ull && !(dbits(sum) > dbits(rt));
            bool viol = false;
            uint32_t ns_owner = NONE;
            const bool any_odd = __any_sync(FULL, nsc || neg || bad);
            if (any_odd) {
                if (neg) {
                    tau = g_sub(g_add(dx, L), tb);
                    sum = g_add(ti, __double_as_longlong(tau) < 0 ? 0.0 : tau);
                }
                bad = ev && (nsc || (own == stamp && dbits(rt) != 0ull)) &&
                      !(dbits(sum) > dbits(rt));
                viol = __any_sync(FULL, bad && !nsc);
                const double tc0 = __double_as_longlong(tau) < 0 ? 0.0 : tau;
                const unsigned sb = __ballot_sync(FULL, nsc && (bad || dbits(tc0) < dbits(D)));
                if (sb) ns_owner = __shfl_sync(FULL, own, __ffs(sb) - 1) & OWN_CHAIN;
            }
            if (__double_as_longlong(tau) < 0) tau = 0.0;
            const unsigned long long tk = evo && !nsc ? dbits(tau) : INF_BITS;
            const int wl = g_winner(tk, tid);
            const unsigned long long bt = shfl_u64(tk, wl);
            bool lift = bt < dbits(D);
            const uint32_t bj = __shfl_sync(FULL, tid, wl);
            if (OPEN && lift && bj == NONE) {
                if (lane == 0) g_undecided(s);
                lift = false;
            }
            const double ts = lift ? __longlong_as_double((long long)bt) : D;
            const double T = lift ? shfl_f64(sum, wl) : g_add(ti, D);
            const double xj = shfl_f64(rx, wl);
            const double tj = shfl_f64(own == stamp ? rt : 0.0, wl);
            if (!strict && ev && held == 0u)
                cas = lift && lane == wl ? atomicCAS(&g[tid].claim, cw, ct)
                                         : __ldcg(&g[tid].claim);
            if (viol) {
                how = CONT_FAIL;
                break;
            }
            if (ns_owner != NONE) {
                const int h = (int)ns_owner;
                if (h != c && h < s.k && __ldcg((const unsigned long long *)s.memb + h) == tag &&
                    s.status[h] == ST_BLOCKED && switches < 4 * m + 4) {
                    next = h;  // wait for that member (Remark 10)
                    st = ST_BLOCKED;
                    ++switches;
                } else {
                    how = CONT_FAIL;
                }
                break;
            }
            if (bounded) {
                if (!(dbits(T) < dbits(tend))) break;  // pauses at the window end
                if (dbits(T) < dbits(tw)) {
                    how = CONT_FAIL;
                    break;
                }
            }
            if (nr0 + n >= cap) {
                how = CONT_FAIL;
                break;
            }
            if (lane == (n & 31)) {
                E.i = i;
                E.x = xi;
                E.t = ti;
                E.D = D;
                E.tau = ts;
                E.tj = lift ? tj : 0.0;
            }
            ++n;
            ti = T;
            if (!lift) {
                st = ST_STALLED;
                D = 0.0;
                break;
            }
            ++nl;
            D = __dsub_rn(D, ts);
            xi = xj;
            i = bj;
            tid = R[wl].a[l3];
            tb = R[wl].b[l3];
            none = g_none(tid);
            g_copy_wait();
            cb ^= 1;
            sl = 3 * wl;
            if (OPEN) {
                op = g_open(tid, tb);
                if (none) g_open_targets(tid, tb, &lv.r[cb][sl]);
                if (op) tb = 0.0;
            }
            if (n - nf == 32 || n > n_lap) {
                if (!claims_stand()) {
                    how = CONT_FOREIGN;
                    drop();
                    --nl;
                    break;
                }
                flush(true);
                if (n > n_lap) {
                    // the run may come round to a disk it moved: the level
                    // requested before that write is read again
                    __threadfence();
                    __syncwarp();
                    if (lane < 12) {
                        const uint32_t id = __shfl_sync(0xFFFu, tid, lane >> 2);
                        g_fetch_part(g, id, &lv.r[cb][sl + (lane >> 2)], lane & 3);
                    }
                    g_copy_wait();
                }
            }
        }
        g_copy_wait();
        // the last step's claims: a stall is its event; a pause, a failed Eq. 2
        // or a wait was decided on what it read
        if (how != CONT_FOREIGN && !claims_stand()) {
            how = CONT_FOREIGN;
            if (st == ST_STALLED) {
                drop();
                st = ST_RUNNING;
            }
        }
        flush(st != ST_STALLED);
        __syncwarp();
        // the events so far stand (a failure rolls them back with the rest)
        if (lane == 0) {
            if (nl > 0 && st != ST_STALLED) {
                g[i].own = OWN_ACTIVE | (uint32_t)c;
                g[i].t = ti;
            }
            s.nrec[c] = nr0 + n;
            s.nlift[c] += nl;
            if (nl) atomicAdd(s.lc + LC_LIFTS, (unsigned long long)nl);
            s.status[c] = how != CONT_DONE ? ST_BLOCKED : st;
            s.ci[c] = i;
            s.tc[c] = ti;
            s.D[c] = D;
        }
        __syncwarp();
        cnt += (uint32_t)n;
        if (how != CONT_DONE) {
            *cnt_out = cnt;
            return how;
        }
        cur = next;
    }
}

// The same in a frame of rings: a member goes on along its ring by stretches of
// 31 events as in g_leap_chain, with Eq. 2 asked of every target and every disk
// read claimed before anything is written. The words are exchanged after the
// records were read, so a word that was free stands for a record nobody has
// written since. (Claims beyond one that fails stay; the component they belong
// to is repaired again.) A run that comes round its ring is left to the replay.
// 1024 chains on 2^20 disks: the repair phase of a leg 33 us with a step per
// event, 17 by stretches.
__device__ __noinline__ int g_continue_ring(const GDev &s, const int32_t *mem, int m, int root,
                                            uint64_t tag, uint32_t epoch, int round, int *met,
                                            uint32_t *cnt_out) {
    const int lane = threadIdx.x & 31, up = (lane + 1) & 31;
    GDisk *const g = s.g;
    const double L = s.L;
    const uint32_t stamp = s.stamp;
    uint32_t cnt = 0;
    int switches = 0, e = 0, cur = -1;
    for (;;) {
        if (cur < 0) {  // the next member still blocked
            while (e < m) {
                const unsigned bm =
                    __ballot_sync(FULL, e + lane < m && s.status[mem[e + lane]] == ST_BLOCKED);
                if (bm) {
                    e += __ffs(bm) - 1;
                    break;
                }
                e += 32;
            }
            if (e >= m) {
                *cnt_out = cnt;
                return CONT_DONE;
            }
            cur = mem[e];
        }
        const int c = cur;
        const uint32_t mine = (uint32_t)c + 1u;
        const unsigned long long ct = ((unsigned long long)epoch << 32) | mine;
        uint32_t i = s.ci[c];
        double t = s.tc[c], D = s.D[c];
        const int32_t nr0 = s.nrec[c];
        const uint32_t seq0 = ((uint32_t)round << 24) | cnt;
        const uint4 at0 = s.pos[i];
        const uint32_t p0 = at0.x, first = at0.y, len = at0.z;
        int nl = 0, n = 0, st = ST_RUNNING, next = -1, how = CONT_DONE;
        for (bool more = true; more;) {
            uint32_t q = p0 - first + (uint32_t)(n + lane);
            if (q >= len) q %= len;
            const uint32_t id = s.rid[first + q];
            const GRingDisk k(g + id);
            const double x = k.x, xn = shfl_f64(x, up), rt = shfl_f64(k.t, up);
            const uint32_t ownn = __shfl_sync(FULL, k.own, up);
            const uint32_t idn = __shfl_sync(FULL, id, up);
            double bb;
            const bool in = lane < 31 && (uint32_t)(n + lane) + 1u < len && k.towards(idn, bb);
            const bool nsc = in && ownn >= OWN_ACTIVE;
            double dx = __dsub_rn(xn, x);
            const bool neg = __double_as_longlong(dx) < 0;
            if (__any_sync(FULL, neg) && neg) dx = g_add(dx, L);
            double tau = __dsub_rn(dx, bb);
            if (__double_as_longlong(tau) < 0) tau = 0.0;
            const unsigned stops = __ballot_sync(FULL, lane < 31 && (nsc || !in));
            g_sums(tau, stops ? __ffs(stops) - 1 : 31, t, D);
            const double sum = __dadd_rn(t, tau);
            const bool timed = ownn == stamp && dbits(rt) != 0ull;
            const bool bad = (nsc || timed) && !(dbits(sum) > dbits(rt));
            const bool lift = !nsc && dbits(tau) < dbits(D);
            const bool ends = !in || (bad && !nsc) || !lift;
            const unsigned fin = __ballot_sync(FULL, lane < 31 && ends);
            const int f = fin ? __ffs(fin) - 1 : 31;
            // what event f is, if it ends the run
            enum { STALLS = 0, FAILS = 1, WAITS = 2 };
            const int kind = __shfl_sync(FULL, !in || (bad && !nsc)                     ? FAILS
                                               : nsc && (bad || dbits(tau) < dbits(D)) ? WAITS
                                                                                       : STALLS,
                                         f);
            // the disks read, the active one and the targets of the events up to f
            uint32_t h = 0u;
            if (lane <= (fin ? f + 1 : 31)) {
                h = g_holder(k.claim, ct);
                if (h == 0u) h = g_holder(atomicCAS(&g[id].claim, k.claim, ct), ct);
            }
            const bool ask = h != 0u && h != mine;
            unsigned fb = 0u;
            if (__any_sync(FULL, ask)) {
                const bool ours = !ask || holder_ours(s, (int)h - 1, root, tag, true);
                fb = __ballot_sync(FULL, !ours);
            }
            const int nev = f + (fin && kind == STALLS ? 1 : 0);  // events of this stretch
            if (fb || nr0 + n + nev > s.cap) {  // none of them is written
                if (fb) *met = (int)__shfl_sync(FULL, h, __ffs(fb) - 1) - 1;
                how = fb ? CONT_FOREIGN : CONT_FAIL;
                i = __shfl_sync(FULL, id, 0);
                t = shfl_f64(t, 0);
                break;
            }
            const bool has = lane < nev, stall = has && lane == f;
            const double ts = stall ? D : tau, tn = stall ? g_add(t, D) : sum;
            const double dn = shfl_f64(D, up);
            double xe = __dadd_rn(x, ts);
            const bool wrap = has && dbits(xe) >= dbits(L);
            if (__any_sync(FULL, wrap) && wrap) xe = g_sub(xe, L);
            if (has) {
                ulonglong2 *u = reinterpret_cast<ulonglong2 *>(grec_at(s, c, nr0 + n + lane));
                u[0] = make_ulonglong2((unsigned long long)id |
                                           ((unsigned long long)(stall ? NONE : idn) << 32),
                                       (unsigned long long)(seq0 + (uint32_t)(n + lane)));
                u[1] = make_ulonglong2(dbits(x), dbits(t));
                u[2] = make_ulonglong2(!stall && ownn == stamp ? dbits(rt) : 0ull, dbits(tn));
                u[3] = make_ulonglong2(dbits(ts), dbits(xe));
                u[4] = make_ulonglong2(stall ? 0ull : dbits(xn), stall ? 0ull : dbits(dn));
                *reinterpret_cast<ulonglong2 *>(&g[id].x) = make_ulonglong2(dbits(xe), dbits(tn));
                g[id].own = stall ? (OWN_STALLED | (uint32_t)c) : stamp;
            }
            n += nev;
            nl += f;
            // the state before event f, or after the stall
            i = __shfl_sync(FULL, id, f);
            t = shfl_f64(stall ? tn : t, f);
            D = shfl_f64(stall ? 0.0 : D, f);
            more = fin == 0u;
            if (more) continue;
            if (kind == STALLS) st = ST_STALLED;
            if (kind == FAILS) how = CONT_FAIL;
            if (kind == WAITS) {
                const int hc = (int)(__shfl_sync(FULL, ownn, f) & OWN_CHAIN);
                if (hc != c && hc < s.k &&
                    __ldcg((const unsigned long long *)s.memb + hc) == tag &&
                    s.status[hc] == ST_BLOCKED && switches < 4 * m + 4) {
                    next = hc;  // wait for that member (Remark 10)
                    st = ST_BLOCKED;
                    ++switches;
                } else {
                    how = CONT_FAIL;
                }
            }
        }
        __syncwarp();
        // the events so far stand (a failure rolls them back with the rest)
        if (lane == 0) {
            if (nl > 0 && st != ST_STALLED) {
                g[i].own = OWN_ACTIVE | (uint32_t)c;
                g[i].t = t;
            }
            s.nrec[c] = nr0 + n;
            s.nlift[c] += nl;
            if (nl) atomicAdd(s.lc + LC_LIFTS, (unsigned long long)nl);
            s.status[c] = how != CONT_DONE ? ST_BLOCKED : st;
            s.ci[c] = i;
            s.tc[c] = t;
            s.D[c] = D;
        }
        __syncwarp();
        cnt += (uint32_t)n;
        if (how != CONT_DONE) {
            *cnt_out = cnt;
            return how;
        }
        cur = next;
    }
}

// Replay of a component with at most 10 members (one warp), rolled back to Ts:
// lane 3e + p holds target p of member e's active disk -- its record, as the
// replay has changed it -- so every member's next event is computed at once,
// and an event costs one round of loads, for the targets of the disk it
// activated (with the pending events in memory, one member per thread and
// three targets one after another it took ~10700 cycles, and the replays were
// most of a leg on dense boxes). The claims are those of graph_step, checked
// one event later.
constexpr int SMALL_REPLAY = 10;

template <bool OPEN>
__device__ __noinline__ bool g_replay_small(const GDev &s, const int32_t *mem, int m,
                                            uint32_t epoch, int round, double Ts, double tend,
                                            int *met_out, double *now_out, uint32_t *seq) {
    const int lane = threadIdx.x & 31;
    const int e = lane / 3, p = lane - 3 * e, base = 3 * e;
    const bool has = e < m;
    const double L = s.L;
    GDisk *const g = s.g;
    const uint32_t stamp = s.stamp;
    const bool bounded = dbits(tend) != INF_BITS;
    const int c = has ? mem[e] : 0x7FFFFFFF;
    const unsigned long long ct = ((unsigned long long)epoch << 32) | ((unsigned)c + 1u);
    uint32_t i = NONE, tid = NONE;
    double xi = 0.0, ti = 0.0, D = 0.0, tb = 0.0;
    int32_t nrec = 0, nl = 0;
    bool run = false;
    if (has) {
        i = s.ci[c];
        ti = s.tc[c];
        D = s.D[c];
        nrec = s.nrec[c];
        run = s.status[c] == ST_RUNNING;
    }
    if (run) {
        xi = g[i].x;
        tid = g[i].a[p];
        tb = g[i].b[p];
    }
    // this lane's target: place, time, owner and its own arrows
    double rx = 0.0, rt = 0.0, b0 = 0.0, b1 = 0.0, b2 = 0.0;
    uint32_t own = 0u, a0 = NONE, a1 = NONE, a2 = NONE;
    bool op = false;
    int met = -1;
    // The claims asked for and not checked yet: the holder that a record's word
    // of this pass names, or what the exchange for a free disk found.
    uint32_t held = 0u, held_i = 0u;
    unsigned long long cas = 0ull;
    auto take = [&](bool mine) {
        held = 0u;
        cas = 0ull;
        if (OPEN && mine) op = g_open(tid, tb);
        if (OPEN && mine && op) {  // (an open arrow: a target at its place)
            rx = g_unsigned(tb);
            rt = tb = 0.0;
            own = OWN_STATIC;
        }
        if (mine && tid != NONE) {
            const ulonglong2 *r = reinterpret_cast<const ulonglong2 *>(g + tid);
            const ulonglong2 u0 = __ldcg(r), u1 = __ldcg(r + 1), u2 = __ldcg(r + 2),
                             u3 = __ldcg(r + 3);
            rx = __longlong_as_double((long long)u0.x);
            rt = __longlong_as_double((long long)u0.y);
            own = (uint32_t)u1.x;
            a0 = (uint32_t)(u1.x >> 32);
            a1 = (uint32_t)u1.y;
            a2 = (uint32_t)(u1.y >> 32);
            b0 = __longlong_as_double((long long)u2.y);
            b1 = __longlong_as_double((long long)u3.x);
            b2 = __longlong_as_double((long long)u3.y);
            held = g_holder(u2.x, ct);
            if (held == 0u) cas = atomicCAS(&g[tid].claim, u2.x, ct);
        }
    };
    // true if a disk taken is held by a chain that is no member
    auto conflict = [&]() -> bool {
        const uint32_t h = held ? held : g_holder(cas, ct);
        const uint32_t me = (uint32_t)c + 1u;
        bool ask = h != 0u && h != me, ask_i = held_i != 0u && held_i != me;
        if (!__any_sync(FULL, ask || ask_i)) return false;
        for (int z = 0; z < m; ++z) {
            const uint32_t cz = (uint32_t)__shfl_sync(FULL, c, 3 * z) + 1u;
            ask = ask && h != cz;
            ask_i = ask_i && held_i != cz;
        }
        const unsigned bm = __ballot_sync(FULL, ask || ask_i);
        if (bm) met = (int)__shfl_sync(FULL, ask ? h : held_i, __ffs(bm) - 1) - 1;
        return bm != 0u;
    };
    if (run && p == 0) held_i = g_claim(s, i, ct);
    take(run);
    bool abort = false;
    double taken = Ts;  // time of the event after which the claims were asked for,
    int taker = -1;     // and the chain that asked
    double now = Ts;
    uint32_t cnt = *seq;
    if (conflict()) abort = true;
    held = held_i = 0u;
    cas = 0ull;
    while (!abort) {
        // every member's next event (Sec. 2.2): the least (tau, j) of its
        // static targets, one lap on where the target came after it had passed
        const bool stc = run && (tid != NONE || (OPEN && op)) && g_static(own);
        double dx = __dsub_rn(rx, xi);
        const bool neg = stc && __double_as_longlong(dx) < 0;
        if (__any_sync(FULL, neg) && neg) dx = g_add(dx, L);
        double tau = __dsub_rn(dx, tb);
        if (__double_as_longlong(tau) < 0) tau = 0.0;
        const bool tnz = stc && own == stamp && dbits(rt) != 0ull;
        if (__any_sync(FULL, tnz)) {
            if (tnz && dbits(g_add(ti, tau)) < dbits(rt)) tau = g_add(tau, L);
        }
        const unsigned long long tk = stc ? dbits(tau) : INF_BITS;
        const int l0 = min(base, 29);
        const unsigned long long t0 = shfl_u64(tk, l0), t1 = shfl_u64(tk, l0 + 1),
                                 t2 = shfl_u64(tk, l0 + 2);
        const uint32_t j0 = __shfl_sync(FULL, tid, l0), j1 = __shfl_sync(FULL, tid, l0 + 1),
                       j2 = __shfl_sync(FULL, tid, l0 + 2);
        unsigned long long bt = t0;
        uint32_t bj = j0;
        int w = 0;
        if (t1 < bt || (t1 == bt && j1 < bj)) {
            bt = t1;
            bj = j1;
            w = 1;
        }
        if (t2 < bt || (t2 == bt && j2 < bj)) {
            bt = t2;
            bj = j2;
            w = 2;
        }
        bool lift = bt < dbits(D);
        if (OPEN && lift && bj == NONE) {
            if (p == 0) g_undecided(s);
            lift = false;
        }
        const double ts = lift ? __longlong_as_double((long long)bt) : D;
        const double T = __dadd_rn(ti, ts);
        // the earliest (T, chain)
        const unsigned hi = run ? (unsigned)(dbits(T) >> 32) : ~0u;
        const unsigned mh = __reduce_min_sync(FULL, hi);
        if (mh == ~0u) break;  // every member has stalled
        const unsigned lo = hi == mh ? (unsigned)dbits(T) : ~0u;
        const unsigned ml = __reduce_min_sync(FULL, lo);
        const bool first = hi == mh && lo == ml;
        const unsigned mc = __reduce_min_sync(FULL, first ? (unsigned)c : ~0u);
        const int src = __ffs(__ballot_sync(FULL, first && (unsigned)c == mc)) - 1;
        const double Tn = shfl_f64(T, src);
        if (bounded && !(dbits(Tn) < dbits(tend))) break;  // the rest lies in a later window
        if (dbits(Tn) < dbits(now) && lane == 0) {
            atomicAdd(s.lc + LC_ORDER, 1ull);
            gdiag(s, 2, round, mc, Tn, now, Ts, m);
        }
        now = Tn;
        const int ce = (int)mc;
        const uint32_t ie = __shfl_sync(FULL, i, src);
        const bool le = __shfl_sync(FULL, (int)lift, src) != 0;
        const uint32_t je = le ? __shfl_sync(FULL, bj, src) : NONE;
        const int we = __shfl_sync(FULL, w, src), ls = src / 3 * 3 + we;
        const int32_t ne = __shfl_sync(FULL, nrec, src);
        if (ne >= s.cap) {  // out of records: reported by the host
            if (lane == 0) atomicAdd(s.lc + LC_ERR_REC, 1ull);
            abort = true;
            met = -1;
            break;
        }
        // a disk is written only once the claims on it stand: those asked for
        // after the last event are checked here if they are this member's, else
        // below, when this event has overlapped their round trip
        if (ce == taker) {
            if (conflict()) {
                abort = true;
                now = taken;
                break;
            }
            held = 0u;
            cas = 0ull;
        }
        const double xe = shfl_f64(xi, src), te = shfl_f64(ti, src), De = shfl_f64(D, src);
        const double tse = shfl_f64(ts, src), xj = shfl_f64(rx, ls);
        const double tj = shfl_f64(own == stamp ? rt : 0.0, ls);
        double xn = __dadd_rn(xe, tse);
        if (dbits(xn) >= dbits(L)) xn = g_sub(xn, L);
        const double Dn = __dsub_rn(De, tse);
        const uint32_t own_i = le ? stamp : (OWN_STALLED | (uint32_t)ce);
        if (lane < 5) {
            unsigned long long u0, u1;
            if (lane == 0) {
                u0 = (unsigned long long)ie | ((unsigned long long)je << 32);
                u1 = (unsigned long long)(((uint32_t)round << 24) | cnt);
            } else if (lane == 1) {
                u0 = dbits(xe);
                u1 = dbits(te);
            } else if (lane == 2) {
                u0 = le ? dbits(tj) : 0ull;
                u1 = dbits(Tn);
            } else if (lane == 3) {
                u0 = dbits(tse);
                u1 = dbits(xn);
            } else {
                u0 = le ? dbits(xj) : 0ull;
                u1 = le ? dbits(Dn) : 0ull;
            }
            reinterpret_cast<ulonglong2 *>(grec_at(s, ce, ne))[lane] = make_ulonglong2(u0, u1);
        } else if (lane == 5) {
            *reinterpret_cast<ulonglong2 *>(&g[ie].x) = make_ulonglong2(dbits(xn), dbits(Tn));
            g[ie].own = own_i;
        } else if (le && lane == 6) {
            g[je].own = OWN_ACTIVE | (uint32_t)ce;
            g[je].t = Tn;
        }
        ++cnt;
        // the copies of the two disks in the other lanes
        if (tid == ie) {
            rx = xn;
            rt = Tn;
            own = own_i;
        }
        if (le && tid == je) {
            rt = Tn;
            own = OWN_ACTIVE | (uint32_t)ce;
        }
        const uint32_t q0 = __shfl_sync(FULL, a0, ls), q1 = __shfl_sync(FULL, a1, ls),
                       q2 = __shfl_sync(FULL, a2, ls);
        const double d0 = shfl_f64(b0, ls), d1 = shfl_f64(b1, ls), d2 = shfl_f64(b2, ls);
        const bool acts = has && c == ce;
        __syncwarp();
        // (if one failed, what was read then is no basis for anything from the
        // time of that event on)
        if (conflict()) {
            abort = true;
            now = taken;
        }
        if (acts) {
            ++nrec;
            ti = Tn;
            if (le) {
                ++nl;
                i = je;
                xi = xj;
                D = Dn;
                tid = p == 0 ? q0 : p == 1 ? q1 : q2;
                tb = p == 0 ? d0 : p == 1 ? d1 : d2;
            } else {
                D = 0.0;
                run = false;
            }
        }
        take(le && !abort && acts);
        taken = Tn;
        taker = ce;
    }
    if (!abort && conflict()) {
        abort = true;
        now = taken;
    }
    if (has && p == 0) {
        s.status[c] = run ? ST_RUNNING : ST_STALLED;
        s.ci[c] = i;
        s.tc[c] = ti;
        s.D[c] = D;
        s.nrec[c] = nrec;
        s.nlift[c] += nl;
        if (nl) atomicAdd(s.lc + LC_LIFTS, (unsigned long long)nl);
    }
    __syncwarp();
    *met_out = met;
    *now_out = now;
    *seq = cnt;
    return abort;
}

// The members of the component of blocked chain a (one warp): the root's tree,
// 16 members at a time. The list grows from the warp's buffer into parts of
// comp_mem (each twice the last: 4 k words hold all of them). False if another
// blocked chain's warp has taken the component for this pass.
//
// So a pass's components need no phase of their own. (One block made them in
// shared memory or, beyond 2048 chains, in global memory, between the resolve
// and the repair: 8 us of a leg at 1024 chains, ~300 of 605 us at 16384.)
constexpr int MEMBER_BUF = 64;
__device__ __noinline__ bool g_members(const GDev &s, int a, uint32_t epoch, int *root_out,
                                       int32_t **mem_out, int *m_out, int *cap_out) {
    __shared__ int32_t buf[8][MEMBER_BUF];
    const int lane = threadIdx.x & 31;
    int32_t *mem = buf[threadIdx.x >> 5];
    const int root = g_root(s, a);
    // (asked now, answered while the members are gathered)
    int prev = 0;
    if (lane == 0) prev = atomicExch(s.taken + root, (int32_t)epoch);
    int cap = MEMBER_BUF, n = 1, done = 0;
    __syncwarp();
    if (lane == 0) mem[0] = root;
    __syncwarp();
    while (done < n) {
        if (n + 32 > cap) {
            // (only the component's one owner takes parts of comp_mem)
            if (__shfl_sync(FULL, prev, 0) == (int32_t)epoch) return false;
            int off = 0;
            if (lane == 0) off = atomicAdd(s.ctl + CTL_NMEMB, 2 * cap);
            off = __shfl_sync(FULL, off, 0);
            int32_t *const to = s.comp_mem + off;
            for (int e = lane; e < n; e += 32) to[e] = mem[e];
            mem = to;
            cap *= 2;
            __syncwarp();
        }
        const int e = done + lane, end = min(n, done + 16);
        int ch = -1, sb = -1;
        if (e < end) {
            const int c = mem[e];
            ch = ((volatile int32_t *)s.child)[c];
            if (e > 0) sb = ((volatile int32_t *)s.sib)[c];
        }
        const unsigned mc = __ballot_sync(FULL, ch >= 0), ms = __ballot_sync(FULL, sb >= 0);
        const unsigned below = (1u << lane) - 1u;
        if (ch >= 0) mem[n + __popc(mc & below)] = ch;
        if (sb >= 0) mem[n + __popc(mc) + __popc(ms & below)] = sb;
        n += __popc(mc) + __popc(ms);
        done = end;
        __syncwarp();
    }
    *root_out = root;
    *mem_out = mem;
    *m_out = n;
    *cap_out = cap;
    return __shfl_sync(FULL, prev, 0) != (int32_t)epoch;
}

// Replay of a larger component: its members spread over the lanes (member e on
// lane e mod 32); after each event only the members whose arrows read a disk it
// changed recompute.
__device__ __noinline__ bool g_replay_large(const GDev &s, const int32_t *mem, int m, int root,
                                            uint64_t tag, uint32_t epoch, int round, double Ts,
                                            double tend, int *met_out, double *now_out,
                                            uint32_t *seq) {
    const int lane = threadIdx.x & 31;
    const bool all = m == s.k;
    bool abort = false;
    int met = -1;
    // this lane's earliest pending event (ev_T: infinity for a member that stands)
    unsigned long long bT = INF_BITS;
    int bc = 0x7FFFFFFF, bl = lane;
    auto take = [&](int c) {
        const unsigned long long T = dbits(s.ev_T[c]);
        if (T < bT || (T == bT && c < bc && T != INF_BITS)) {
            bT = T;
            bc = c;
        }
    };
    for (int e = lane; e < m; e += 32) {
        const int c = mem[e];
        if (s.status[c] == ST_RUNNING)
            g_compute(s, c, root, tag, epoch, all, abort, met);
        else
            s.ev_T[c] = INFINITY;
        take(c);
    }
    double now = Ts;
    uint32_t cnt = *seq;
    for (;;) {
        {
            const unsigned ab = __ballot_sync(FULL, abort);
            if (ab) {
                met = __shfl_sync(FULL, met, __ffs(ab) - 1);
                abort = true;
                break;
            }
        }
        bl = lane;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long T2 = shfl_xor_u64(bT, o);
            const int c2 = __shfl_xor_sync(FULL, bc, o);
            const int l2 = __shfl_xor_sync(FULL, bl, o);
            if (T2 < bT || (T2 == bT && c2 < bc)) {
                bT = T2;
                bc = c2;
                bl = l2;
            }
        }
        if (bc == 0x7FFFFFFF) break;
        if (!(bT < dbits(tend))) break;  // the rest lies in a later window
        const double Tn = __longlong_as_double((long long)bT);
        if (dbits(Tn) < dbits(now) && lane == 0) {
            atomicAdd(s.lc + LC_ORDER, 1ull);
            gdiag(s, 2, round, bc, Tn, now, Ts, m);
        }
        now = Tn;
        uint32_t ib = NONE, jb = NONE;
        int st = ST_RUNNING;
        if (lane == bl) {
            const uint32_t i = s.ci[bc];
            const double ti = s.tc[bc], D = s.D[bc];
            GStep o;
            o.lift = s.ev_lift[bc];
            o.tau = s.ev_tau[bc];
            o.j = s.ev_j[bc];
            o.xj = s.ev_xj[bc];
            o.tj = s.ev_tj[bc];
            const double xi = s.g[i].x;
            const int32_t nr = s.nrec[bc];
            if (nr >= s.cap) {
                atomicAdd(s.lc + LC_ERR_REC, 1ull);
                st = ST_BLOCKED;
            } else {
                graph_apply(s, bc, i, xi, ti, D, o.lift, o.j, o.tau, o.xj, o.tj,
                            ((uint32_t)round << 24) | cnt, nr);
                s.nrec[bc] = nr + 1;
                if (o.lift) {
                    s.nlift[bc] += 1;
                    atomicAdd(s.lc + LC_LIFTS, 1ull);
                }
                st = o.lift ? ST_RUNNING : ST_STALLED;
            }
            ib = i;
            if (st == ST_RUNNING) {
                jb = o.j;
                s.ci[bc] = o.j;
                s.tc[bc] = __dadd_rn(ti, o.tau);
                s.D[bc] = __dsub_rn(D, o.tau);
            } else if (st == ST_STALLED) {
                s.tc[bc] = __dadd_rn(ti, D);
                s.D[bc] = 0.0;
                s.status[bc] = ST_STALLED;
                s.ev_T[bc] = INFINITY;
            }
        }
        ++cnt;
        st = __shfl_sync(FULL, st, bl);
        ib = __shfl_sync(FULL, ib, bl);
        jb = __shfl_sync(FULL, jb, bl);
        __syncwarp();
        if (st == ST_BLOCKED) {  // out of records: reported by the host
            abort = true;
            met = -1;
            break;
        }
        // one look at every member, four at once: does it read a disk that changed,
        // and the earliest event of this lane's (two passes, member by member: 1253
        // ms a leg of 4096 chains on 16384 dense disks, 848 so)
        const int ce = bc;
        bT = INF_BITS;
        bc = 0x7FFFFFFF;
        auto is = [&](uint32_t a) { return a != NONE && (a == ib || a == jb); };
        for (int e0 = lane; e0 < m; e0 += 4 * 32) {
            int c[4];
            unsigned long long T[4];
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) c[u] = e0 + 32 * u < m ? mem[e0 + 32 * u] : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                T[u] = c[u] >= 0 ? dbits(s.ev_T[c[u]]) : INF_BITS;
                v[u] = c[u] >= 0 ? *reinterpret_cast<const uint4 *>(s.ev_a + 4 * (size_t)c[u])
                                 : make_uint4(NONE, NONE, NONE, NONE);
            }
#pragma unroll 1
            for (int u = 0; u < 4; ++u) {
                const unsigned long long t = u == 0 ? T[0] : u == 1 ? T[1] : u == 2 ? T[2] : T[3];
                const uint4 a = u == 0 ? v[0] : u == 1 ? v[1] : u == 2 ? v[2] : v[3];
                const int q = u == 0 ? c[0] : u == 1 ? c[1] : u == 2 ? c[2] : c[3];
                if (t == INF_BITS) continue;
                const bool redo = q == ce || is(a.x) || is(a.y) || is(a.z);
                if (redo) g_compute(s, q, root, tag, epoch, all, abort, met);
                const unsigned long long tn = redo ? dbits(s.ev_T[q]) : t;
                if (tn < bT || (tn == bT && q < bc)) {
                    bT = tn;
                    bc = q;
                }
            }
        }
        __syncwarp();
    }
    *met_out = met;
    *now_out = now;
    *seq = cnt;
    return abort;
}

// Systems of more chains may have all of them made one component (k_run_graph).
constexpr int ONE_MIN = 64;

// A component of this round (one warp; room for cap members in mem): continue
// its blocked chains, or else roll its members back to T* and replay them in
// global event-time order (Alg. 2) up to the window's end. A replay of the
// first round that needs a disk of a chain in no component takes that chain
// in and starts again: left to the next round, it made one of 70 us on nearly
// every leg of 2048 chains on 262144 dense disks.
__device__ __noinline__ void g_repair_component(const GDev &s, int32_t *mem, int m, int cap,
                                                int root, int round, uint32_t epoch,
                                                uint32_t wr_tag, double tw, double tend) {
    const int lane = threadIdx.x & 31;
    double Ts = INFINITY;
    // the members listed for this round of this pass (wr_tag names both)
    const uint64_t tag = ((uint64_t)wr_tag << 32) | (uint32_t)root;
    for (int e = lane; e < m; e += 32) {
        const int c = mem[e];
        Ts = fmin(Ts, s.vt[c]);
        s.memb[c] = tag;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Ts = fmin(Ts, __shfl_xor_sync(FULL, Ts, o));
    Ts = fmax(Ts, tw);  // earlier windows are final
    if (lane == 0) atomicAdd(s.lc + LC_REPAIRED, (unsigned long long)m);
    __syncwarp();
    uint32_t seq = 0;  // events of this repair so far: what is kept of one attempt
                       // comes before the next one's in order
    // (a later round of a leg without claim windows: chains that a repair which
    // met another component left unfinished)
    const bool whole = dbits(tend) == INF_BITS && dbits(tw) == 0ull;
    if (round > 1 && whole) {
        for (int e = lane; e < m; e += 32)
            if (s.status[mem[e]] == ST_RUNNING) s.status[mem[e]] = ST_BLOCKED;
        __syncwarp();
    }
    // (all chains as one component: replayed in order from the start)
    const bool all = round > 1 && m == s.k && s.k > ONE_MIN;
    if ((round == 1 || whole) && !all) {
        int met = -1;
        const int how = s.ring && !s.strict
                            ? g_continue_ring(s, mem, m, root, tag, epoch, round, &met, &seq)
                        : s.open
                            ? g_continue<true>(s, mem, m, root, tag, epoch, round, tw, tend, &met,
                                               &seq)
                            : g_continue<false>(s, mem, m, root, tag, epoch, round, tw, tend, &met,
                                                &seq);
        if (how == CONT_DONE) {
            if (lane == 0) atomicAdd(s.lc + LC_CONTINUED, (unsigned long long)m);
            g_finish(s, mem, m, root, false, -1, Ts, true);
            return;
        }
        if (how == CONT_FOREIGN) {
            // its events so far stand for the merged component to go on from (or
            // to roll back to T*: all of this round's events lie after it)
            g_finish(s, mem, m, root, true, met, Ts);
            return;
        }
        // What was done is a run of Alg. 4 without a violation, so every event
        // before the earliest time an unfinished chain stands at is exact
        // (Remark 6): the replay starts there, not where the pass was cut.
        if (whole) {
            Ts = INFINITY;
            for (int e = lane; e < m; e += 32)
                if (s.status[mem[e]] == ST_BLOCKED) Ts = fmin(Ts, s.tc[mem[e]]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) Ts = fmin(Ts, __shfl_xor_sync(FULL, Ts, o));
        }
    }
    for (;;) {
        g_rollback(s, mem, m, Ts);
        for (int e = lane; e < m; e += 32) g_resume(s, mem[e]);
        __syncwarp();
        int met = -1;
        double now = Ts;
        const bool abort =
            m <= SMALL_REPLAY
                ? (s.open ? g_replay_small<true>(s, mem, m, epoch, round, Ts, tend, &met, &now, &seq)
                          : g_replay_small<false>(s, mem, m, epoch, round, Ts, tend, &met, &now,
                                                  &seq))
                : g_replay_large(s, mem, m, root, tag, epoch, round, Ts, tend, &met, &now,
                                 &seq);
        int more = 0;
        if (abort && whole && round == 1 && m < cap && met >= 0 && met < s.k && lane == 0) {
            // a chain of no component: it joins this one at once
            int h = __ldcg(s.comp_of + met);
            if (h == met && met != root && __ldcg(s.fin + met) == 1)
                h = atomicCAS(s.comp_of + met, met, root) == met ? root : -1;
            if (h == root) {
                mem[m] = met;
                s.memb[met] = tag;
                atomicAdd(s.lc + LC_REPAIRED, 1ull);
                more = 1;
            }
        }
        if (!__shfl_sync(FULL, more, 0)) {
            g_finish(s, mem, m, root, abort, met, now);
            return;
        }
        ++m;
        Ts = now;  // (the events before are exact)
        __syncwarp();
    }
}

// ------------------------------------------- persistent multi-leg kernel

struct GCtl {
    int64_t budget;  // liftings for this run (0: none)
    int64_t lifts, legs, conflict_legs, repaired, continued, horizon, order_err, p1_lifts,
        repair_lifts, restarts, blocked, cwindows, row_windows;
    int64_t leg0;    // legs run before this launch (lifting log)
    uint8_t *flags;  // per-leg conflict flags (device) or null
    int32_t flags_cap;
    int32_t done;    // budget reached or error
    int32_t err;     // LC_ERR_* seen, or too many repair rounds
    int32_t failed;  // 1 until a leg is done without one
    int32_t dbg;     // an internal check recorded in GDev::dbg (set at the end)
    int32_t open;    // an open arrow left a step undecided: nothing of the launch stands
};

enum { GG_WORK = 0, GG_ANY, GG_ERR, GG_REMAIN0, GG_REMAIN1, GG_COUNT, GG_PASSES,
       GG_NBLK, GG_N };
enum { GPH_BEGIN = 0, GPH_PASS1, GPH_REPAIR, GPH_END, GPH_N };

// One launch: R systems (their descriptions in device memory), their chains
// and conflict components flattened by prefix offsets.
struct GBatchDev {
    const GDev *reps;              // [R]
    GCtl *ctl;                     // [R]
    const int32_t *chain_base;     // [R + 1]
    int32_t *comp_base;            // [R + 1]
    unsigned int *bar;             // [1] grid barrier
    int32_t *g;                    // [GG_N]
    int32_t *blocked;              // [chain_base[R]] blocked chains of a pass
    unsigned long long *phase_ns;  // [GPH_N] device time per phase (block 0 clock)
    int32_t R, max_legs, windows, pad;
    unsigned long long wait_ns;    // bound on every grid-barrier wait
};

__device__ __forceinline__ double g_window_start(const GDev &s, int w) {
    return w == 0 ? 0.0 : __ddiv_rn(__dmul_rn((double)w, s.ell), (double)s.windows);
}

__device__ __forceinline__ double g_window_end(const GDev &s, int w) {
    return w + 1 >= s.windows ? INFINITY
                              : __ddiv_rn(__dmul_rn((double)(w + 1), s.ell), (double)s.windows);
}

// system of flattened item f, with base[r] <= f < base[r + 1]
__device__ __forceinline__ int g_find_rep(const int32_t *base, int R, int f) {
    int lo = 0, hi = R;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (base[mid] <= f)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

__device__ __forceinline__ bool g_rep_on(const GBatchDev &B, int r) { return !B.ctl[r].done; }

// A system with no liftings budget runs every leg of the launch: its next leg
// is begun by its chains at this leg's end. With a budget, the leg's totals
// decide first.
__device__ __forceinline__ bool g_next_at_end(const GBatchDev &B, int r, int leg) {
    return B.ctl[r].budget == 0 && leg + 1 < B.max_legs;
}

// The system's description in the warp's slot of shared memory (constant
// during a launch; a field of the global copy would be re-read from L2 after
// every store).
__device__ __forceinline__ const GDev &g_warp_dev(GDev *slot, int *rep, const GDev *reps, int r) {
    if (*(volatile int *)rep != r) {
        constexpr int WORDS = (int)(sizeof(GDev) / sizeof(uint32_t));
        const uint32_t *src = reinterpret_cast<const uint32_t *>(reps + r);
        uint32_t *dst = reinterpret_cast<uint32_t *>(slot);
        for (int q = threadIdx.x & 31; q < WORDS; q += 32) dst[q] = src[q];
        __syncwarp();
        if ((threadIdx.x & 31) == 0) *(volatile int *)rep = r;
        __syncwarp();
    }
    return *slot;
}

// The leg's stamp and the touch keys of claim window w in the warp's copy of the
// description.
__device__ __forceinline__ void g_set_stamp(GDev *slot, int leg, int w, int lane) {
    if (lane == 0) {
        slot->stamp = slot->stamp0 + (uint32_t)leg + 1u;
        if (slot->windows > 1) slot->key = slot->keys + ((w & 1) != 0 ? slot->n : 0);
    }
    __syncwarp();
}

// Chain c at the start of window w > 0: its keys of the last window go (nobody
// reads that set in this window; in a phase of its own, with a barrier, a window
// took 16.7 us instead of 14.5).
__device__ __noinline__ void g_drop_keys(GDev *slot, int c, int leg, int w, int lane) {
    g_set_stamp(slot, leg, w - 1, lane);
    g_reset_keys(*slot, c, lane);
    __syncwarp();
    g_set_stamp(slot, leg, w, lane);
}

// The flags of a pass with claim windows or restarts, while chains resolve: what a
// chain read its run alone left, so of few chains the warps without one find it (a
// call of its own: the loop inside the kernel cost batches without claim windows
// 0.8%).
__device__ __noinline__ void g_flag_strict(const GDev *reps, const GCtl *ctl, const int32_t *base,
                                           int R, GDev *slot, int *rep, int f, int nwarps,
                                           uint32_t pass) {
    const int total = base[R], lane = threadIdx.x & 31;
    for (; f < total; f += nwarps) {
        const int r = g_find_rep(base, R, f);
        if (ctl[r].done) continue;
        const GDev &s = g_warp_dev(slot, rep, reps, r);
        g_flag_chain(s, f - base[r], s.epoch0 + pass, lane);
    }
}

constexpr int GRUN_THREADS = 256;
constexpr int GRUN_MIN_BLOCKS = 2;
constexpr int MAX_RESTARTS = 16;  // per leg, then the local repair takes over

// One cooperative launch runs up to max_legs legs of every system. Per leg
// and claim window: the parallel pass (one warp per chain), the resolve, then
// repair rounds (one warp per component: in the first round the one of its
// blocked chains, in later ones, whose components one block per system finds,
// from a queue) until no component met another chain; the leg end with each
// system's totals. Phases are separated by grid barriers whose waits are
// bounded (ECMC_ETIMEOUT). Restart mode takes one system.
//
// Bound by latency: a leg of 1024 chains on 2^20 lattice disks takes 32 us, of
// which the runs alone 5, the publishing 8, the continuations 8 to 17, three
// barriers 3; DRAM and the FP64 pipes are nearly idle.
__global__ void __launch_bounds__(GRUN_THREADS, GRUN_MIN_BLOCKS) k_run_graph(GBatchDev B) {
    extern __shared__ int32_t uf_sm[];  // UF_SMEM_BYTES: the union-find working set
    __shared__ int warp_tot[32];
    __shared__ int tot[2];
    __shared__ int sflag;
    __shared__ double dmin[GRUN_THREADS / 32];
    __shared__ GDev wdev[GRUN_THREADS / 32];
    __shared__ int wrep[GRUN_THREADS / 32];
    if ((threadIdx.x & 31) == 0) wrep[threadIdx.x >> 5] = -1;
    __syncthreads();
    GDev *const my_dev = wdev + (threadIdx.x >> 5);
    int *const my_rep = wrep + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    // warps interleaved over the blocks: chains spread over all SMs
    const int gw = blockIdx.x + gridDim.x * (threadIdx.x >> 5);
    const int R = B.R;
    const int total_chains = B.chain_base[R];
    const bool restart = R == 1 && B.reps[0].restart;
    // Without claim windows or restarts a leg has one pass. Its chains begin the
    // leg there (the stamps make clearing local times unnecessary), and the flag
    // is found and the touch keys go during the repair. (In a phase of their own
    // before the pass, and with the resolve and the leg end: a batch of 128 21.3
    // ms, 20.0 so, 12 served requests 25.4 and 23.7.) One such system also needs no leg end: s.lc
    // alternates by leg, and the totals of a leg are taken by one warp while the
    // next one resolves. Of several systems the budgets decide which go on.
    const bool simple = !B.reps[0].strict;
    const bool fast = R == 1 && simple;
    const bool timer = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned long long t_prev = timer ? gtimer() : 0ull;
    auto mark = [&](int ph) {
        if (timer) {
            const unsigned long long t = gtimer();
            B.phase_ns[ph] += t - t_prev;
            t_prev = t;
        }
    };
    auto barrier = [&]() -> bool { return grid_sync(B.bar, B.g + GG_ERR, &sflag, B.wait_ns); };
    // true in the last block to get here, of all blocks (each comes once per
    // use; the block barrier, then the master thread's fences, release before
    // the count and acquire after it, as in the grid barrier)
    auto last_block = [&]() -> bool {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const int old = atomicAdd(B.g + GG_COUNT, 1);
            sflag = (old + 1) % (int)gridDim.x == 0;
            if (sflag) __threadfence();
        }
        __syncthreads();
        const bool last = sflag != 0;
        __syncthreads();
        return last;
    };
    // conflict components of system r after round 1 (one block)
    auto uf_system = [&](int r, int round) {
        if (threadIdx.x < 32) (void)g_warp_dev(wdev, wrep, B.reps, r);
        __syncthreads();
        const GDev &s = wdev[0];
        // (a system with a chain out of records has failed its leg: no merge cures
        // that, and every further round would fail alike)
        const bool need = g_rep_on(B, r) && __ldcg(s.ctl + CTL_NABORT) != 0 &&
                          __ldcg(s.lc + LC_ERR_REC) == 0ull;
        if (need && round <= 255) {
            // the chains taken over in the last round
            for (int c = threadIdx.x; c < s.k; c += blockDim.x) {
                const int to = s.comp_of[c];
                if (to != c) uf_union(s.uf, c, to);
            }
            __syncthreads();
            uf_block(s, warp_tot, tot, uf_sm);
            // Where most chains are one component the rest belongs to it sooner
            // or later (every round would redo it with a few more): all chains
            // become one, which meets nobody. 4096 chains on 16384 dense disks:
            // 51 rounds and 7 s a leg otherwise, 1 s so. The same ends a repair of
            // very many rounds.
            int big = 0;
            const int ncomp = s.ctl[CTL_NCOMP];
            for (int q = threadIdx.x; q < ncomp; q += blockDim.x)
                big |= 2 * (s.comp_off[q + 1] - s.comp_off[q]) > s.k;
            if (__syncthreads_or(big || round >= 64) && s.k > ONE_MIN && ncomp > 0) {
                for (int c = threadIdx.x; c < s.k; c += blockDim.x) {
                    s.uf[c] = 0;
                    s.comp_of[c] = 0;
                    s.fin[c] = 0;
                    s.comp_mem[c] = c;
                }
                if (threadIdx.x == 0) {
                    s.comp_root[0] = 0;
                    s.comp_off[0] = 0;
                    s.comp_off[1] = s.k;
                    s.ctl[CTL_NCOMP] = 1;
                    s.ctl[CTL_NMEMB] = s.k;
                }
            }
        } else if (threadIdx.x == 0) {
            s.ctl[CTL_NCOMP] = 0;
            if (need) atomicAdd(s.lc + LC_ERR_CAP, 1ull);  // too many rounds
        }
        __syncthreads();
    };
    // prefix of component counts over systems (one block)
    auto comp_prefix = [&]() {
        const int chunk = (R + blockDim.x - 1) / blockDim.x;
        const int lo = min(R, (int)threadIdx.x * chunk), hi = min(R, lo + chunk);
        int sum = 0;
        for (int r = lo; r < hi; ++r) sum += __ldcg(B.reps[r].ctl + CTL_NCOMP);
        int off = block_exscan(sum, warp_tot, tot);
        for (int r = lo; r < hi; ++r) {
            B.comp_base[r] = off;
            off += __ldcg(B.reps[r].ctl + CTL_NCOMP);
            // every block read the abort counts before it counted itself
            B.reps[r].ctl[CTL_NABORT] = 0;
        }
        if (threadIdx.x == 0) {
            B.comp_base[R] = tot[0];
            B.g[GG_WORK] = 0;
            B.g[GG_ANY] = tot[0];
        }
    };
    unsigned long long *const lc0 = B.reps[0].lc;
    // the totals of leg `leg` of system r from its counters, which go back to
    // zero (one thread)
    auto totals = [&](int r, unsigned long long *lcp) -> bool {
        GCtl *const cp = B.ctl + r;
        GCtl c = *cp;
        if (c.done) return true;
        unsigned long long lc[LC_N];
#pragma unroll
        for (int q = 0; q < LC_N; ++q) lc[q] = __ldcg(lcp + q);
        const int64_t lifts = (int64_t)(lc[LC_P1LIFTS] + lc[LC_LIFTS]);
        const int flag = lc[LC_WEAK] != 0ull;
        if (c.flags && c.legs < c.flags_cap) c.flags[c.legs] = (uint8_t)flag;
        c.lifts += lifts;
        c.p1_lifts += (int64_t)lc[LC_P1LIFTS];
        if (flag) c.repair_lifts += lifts;
        c.legs += 1;
        c.conflict_legs += flag;
        c.repaired += (int64_t)lc[LC_REPAIRED];
        c.continued += (int64_t)lc[LC_CONTINUED];
        c.restarts += (int64_t)lc[LC_RESTARTS];
        c.blocked += (int64_t)lc[LC_BLOCKED];
        c.cwindows += simple ? flag : (int64_t)lc[LC_CWINDOWS];
        if (B.reps[r].ring && B.reps[r].cells && lc[LC_RINGLAP] == 0ull) c.row_windows += B.windows;
        c.horizon += (int64_t)lc[LC_HORIZON];
        c.order_err += (int64_t)lc[LC_ORDER];
        if (lc[LC_ERR_REC] != 0ull || lc[LC_ERR_CAP] != 0ull) c.err = 1;
        if (lc[LC_OPEN] != 0ull) c.open = 1;
        c.failed = c.err || c.open;
        if (c.failed || (c.budget > 0 && c.lifts >= c.budget)) c.done = 1;
        *cp = c;
#pragma unroll
        for (int q = 0; q < LC_N; ++q) lcp[q] = 0ull;
        return c.done != 0;
    };
    uint32_t pass = 0;  // passes of the launch (the same count in every thread)
    GBlocked bl = {(unsigned *)(B.g + GG_NBLK), B.blocked, 0u};
    int leg = 0;
    for (; leg < B.max_legs; ++leg) {
        if (fast) {
            GDev &s = *my_dev;
            (void)g_warp_dev(my_dev, my_rep, B.reps, 0);
            if (lane == 0) {
                s.lc = lc0 + (leg & 1) * LC_N;
                s.stamp = s.stamp0 + (uint32_t)leg + 1u;
            }
            __syncwarp();
        }
        // leg start of the systems whose last leg did not begin this one
        bool begin_here = false;
        for (int r = 0; r < R && !simple; ++r)
            if (g_rep_on(B, r) && !(leg > 0 && g_next_at_end(B, r, leg - 1))) begin_here = true;
        if (begin_here) {
            for (int f = gw; f < total_chains; f += nwarps) {
                const int r = g_find_rep(B.chain_base, R, f);
                if (!g_rep_on(B, r) || (leg > 0 && g_next_at_end(B, r, leg - 1))) continue;
                const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
                const int c = f - B.chain_base[r];
                g_begin_state(s, c, s.ci[c], lane);
            }
            if (!barrier()) return;
        }
        mark(GPH_BEGIN);
        // restart mode (one claim window): a pass that meets a conflict is cut
        // at T*, the earliest time a chain stopped -- every event before it is
        // exact (Remark 6) -- all chains are rolled back to T*, and T* becomes
        // the next breakpoint of the leg: a new pass from T* (Sec. 3.4, second
        // restart strategy). A pass that cannot progress (T* at its own
        // start), or the last one allowed, is repaired locally.
        double tw_r = 0.0;
        int sub = 0;
        bool any = false;  // (fast) the leg had something to repair
        auto flags = [&]() {
            for (int f = gw; f < total_chains; f += nwarps) {
                const int r = g_find_rep(B.chain_base, R, f), c = f - B.chain_base[r];
                if (!g_rep_on(B, r)) continue;
                const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
                g_flag_chain(s, c, s.epoch0 + pass, lane);
                g_reset_keys(s, c, lane);
            }
        };
        for (int w = 0; w < B.windows; ++w) {
            int nblk = 0;  // blocked chains of the pass, of all systems
            for (;;) {
                ++pass;
                if (gt == 0) B.g[GG_WORK] = 0;
                for (int f = gw; f < total_chains; f += nwarps) {
                    const int r = g_find_rep(B.chain_base, R, f);
                    if (!g_rep_on(B, r)) continue;
                    const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
                    if (!fast) g_set_stamp(my_dev, leg, w, lane);
                    g_begin_pass(s, f - B.chain_base[r], lane);
                    if (s.ring && simple && g_leap_chain(s, f - B.chain_base[r])) continue;
                    if (w > 0) g_drop_keys(my_dev, f - B.chain_base[r], leg, w, lane);
                    const double t0 = restart ? tw_r : g_window_start(s, w);
                    if (s.open)
                        g_spec_chain<true>(s, f - B.chain_base[r], t0, g_window_end(s, w), simple);
                    else
                        g_spec_chain<false>(s, f - B.chain_base[r], t0, g_window_end(s, w), simple);
                }
                if (!barrier()) return;
                if (gt == 0 && w == 0 && sub == 0) B.g[GG_REMAIN0 + ((leg + 1) & 1)] = 0;
                // (the leg's own counters are the other half of s.lc)
                if (fast && leg > 0 && gw == nwarps - 1 && lane == 0)
                    (void)totals(0, lc0 + ((leg - 1) & 1) * LC_N);
                for (int f = gw; f < total_chains; f += nwarps) {
                    const int r = g_find_rep(B.chain_base, R, f);
                    if (!g_rep_on(B, r)) continue;
                    const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
                    if (!fast) g_set_stamp(my_dev, leg, w, lane);
                    g_resolve_chain(s, f - B.chain_base[r], restart ? tw_r : g_window_start(s, w),
                                    s.epoch0 + pass, f, bl);
                }
                if (!simple && sub == 0)
                    g_flag_strict(B.reps, B.ctl, B.chain_base, R, my_dev, my_rep,
                                  nwarps - 1 - gw, nwarps, pass);
                if (!barrier()) return;
                mark(GPH_PASS1);
                {
                    const unsigned now = (unsigned)__ldcg(B.g + GG_NBLK);
                    nblk = (int)(now - bl.base);
                    bl.base = now;
                }
                if (!restart) break;
                const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, 0);
                g_set_stamp(my_dev, leg, w, lane);
                if (__ldcg(s.lc + LC_WBLOCKED) == 0ull) break;
                if (blockIdx.x == 0) {  // T*: the earliest stop of this pass
                    double m = INFINITY;
                    for (int c = threadIdx.x; c < s.k; c += blockDim.x)
                        if (s.status[c] == ST_BLOCKED) m = fmin(m, s.vt[c]);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(FULL, m, o));
                    if (lane == 0) dmin[threadIdx.x >> 5] = m;
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) m = fmin(m, dmin[q]);
                        s.tstar[0] = fmax(m, tw_r);
                    }
                    __syncthreads();
                }
                if (!barrier()) return;
                const double Ts = __ldcg(s.tstar);
                if (!(dbits(Ts) > dbits(tw_r)) || sub >= MAX_RESTARTS) break;  // local repair
                for (int f = gw; f < total_chains; f += nwarps) g_reset_keys(s, f, lane);
                if (!barrier()) return;
                // (every thread has read the blocked count: back to 0)
                if (gt == 0) {
                    s.lc[LC_WBLOCKED] = 0ull;
                    s.lc[LC_RESTARTS] += 1ull;
                }
                for (int c = gt; c < s.k; c += (int)(gridDim.x * blockDim.x))
                    g_rollback_chain(s, c, Ts);
                if (!barrier()) return;
                tw_r = Ts;
                ++sub;
            }
            // the window's flag: the reads of two chains met (its counter is added
            // to again behind the next pass's barrier)
            for (int r = gt; r < R && !simple; r += (int)(gridDim.x * blockDim.x))
                if (g_rep_on(B, r) && __ldcg(B.reps[r].lc + LC_WWEAK) != 0ull) {
                    atomicAdd(B.reps[r].lc + LC_CWINDOWS, 1ull);
                    B.reps[r].lc[LC_WWEAK] = 0ull;
                }
            // repair rounds
            for (int round = 1; nblk > 0; ++round) {
                int ncomp = nblk;
                if (round > 1) {
                    for (int r = blockIdx.x; r < R; r += gridDim.x) uf_system(r, round);
                    // the last block to finish its union-finds takes the prefix
                    if (last_block()) comp_prefix();
                    if (!barrier()) return;
                    ncomp = __ldcg(B.g + GG_ANY);
                    if (ncomp == 0) break;
                }
                // round 1: an entry per blocked chain, the first ones to the last
                // warps (of few chains, those without one of their own); the
                // others, and later rounds, from a queue
                for (int z = round == 1 ? nwarps - 1 - gw : -1;;) {
                    if (z < 0) {
                        if (lane == 0) z = atomicAdd(B.g + GG_WORK, 1);
                        z = __shfl_sync(FULL, z, 0) + (round == 1 ? nwarps : 0);
                    }
                    if (z >= ncomp) break;
                    const int f = round == 1 ? __ldcg(B.blocked + z) : z;
                    const int32_t *const base = round == 1 ? B.chain_base : B.comp_base;
                    const int r = g_find_rep(base, R, f), q = f - base[r];
                    const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
                    if (!fast) g_set_stamp(my_dev, leg, w, lane);
                    int root, m;
                    int32_t *mem;
                    int cap = 0;
                    bool mine = true;
                    if (round == 1) {
                        mine = g_members(s, q, s.epoch0 + pass, &root, &mem, &m, &cap);
                    } else {
                        root = s.comp_root[q];
                        const int off = s.comp_off[q];
                        m = s.comp_off[q + 1] - off;
                        mem = s.comp_mem + off;
                    }
                    if (mine)
                        g_repair_component(s, mem, m, cap, root, round, s.epoch0 + pass,
                                           ((uint32_t)(leg * B.windows + w) << 8) | (uint32_t)round,
                                           restart ? tw_r : g_window_start(s, w),
                                           g_window_end(s, w));
                    if (round == 1 && ncomp <= nwarps) break;
                    z = -1;
                }
                if (simple && round == 1) flags();
                if (!barrier()) return;
                // no component met another chain: the window is repaired
                int aborted = 0;
                for (int r = threadIdx.x; r < R; r += blockDim.x)
                    if (g_rep_on(B, r) && __ldcg(B.reps[r].ctl + CTL_NABORT) != 0) aborted = 1;
                if (!__syncthreads_or(aborted)) break;
            }
            if (simple && nblk == 0) flags();
            any = nblk > 0;
            mark(GPH_REPAIR);
        }
        if (fast) {
            // a leg without components has passed no barrier since its keys went
            if (!any && !barrier()) return;
            const GDev &s = *my_dev;
            if (s.log_on)
                for (int f = gw; f < total_chains; f += nwarps)
                    g_log_chain(s, f, (int32_t)(B.ctl[0].leg0 + leg), lane);
            mark(GPH_END);
            // every thread decides alike: the leg's counters are final since
            // the barrier, the totals before it since the leg's first one
            const GCtl *const cp = B.ctl;
            const int64_t lifts = (int64_t)__ldcg((const unsigned long long *)&cp->lifts) +
                                  (int64_t)(__ldcg(s.lc + LC_P1LIFTS) + __ldcg(s.lc + LC_LIFTS));
            // (one round of loads)
            const bool err =
                (__ldcg(s.lc + LC_ERR_REC) | __ldcg(s.lc + LC_ERR_CAP)) != 0ull;
            if (err || (cp->budget > 0 && lifts >= cp->budget)) break;
            continue;
        }
        // leg end: the log and the touch keys of the last window; the last
        // block takes each system's totals
        for (int f = gw; f < total_chains; f += nwarps) {
            const int r = g_find_rep(B.chain_base, R, f);
            if (!g_rep_on(B, r)) continue;
            const GDev &s = g_warp_dev(my_dev, my_rep, B.reps, r);
            const int c = f - B.chain_base[r];
            if (!simple) {
                g_set_stamp(my_dev, leg, B.windows - 1, lane);
                g_reset_keys(s, c, lane);
            }
            if (s.log_on) g_log_chain(s, c, (int32_t)(B.ctl[r].leg0 + B.ctl[r].legs), lane);
            if (!simple && g_next_at_end(B, r, leg)) g_begin_state(s, c, s.ci[c], lane);
        }
        if (last_block())
            for (int r = threadIdx.x; r < R; r += blockDim.x)
                if (!B.ctl[r].done && !totals(r, B.reps[r].lc))
                    atomicAdd(B.g + GG_REMAIN0 + (leg & 1), 1);
        if (!barrier()) return;
        mark(GPH_END);
        if (__ldcg(B.g + GG_REMAIN0 + (leg & 1)) == 0) break;
    }
    // (the last block out: every other thread has decided on these counters)
    if (fast && last_block() && threadIdx.x == 0) {
        const int last = leg < B.max_legs ? leg : B.max_legs - 1;
        (void)totals(0, lc0 + (last & 1) * LC_N);
    }
    if (gt == 0) B.g[GG_PASSES] = (int32_t)pass;
    // the systems whose internal checks recorded a failure (GDev::dbg[0])
    if (blockIdx.x == 0)
        for (int r = threadIdx.x; r < R; r += blockDim.x)
            if (B.reps[r].dbg && __ldcg(B.reps[r].dbg) != 0.0) B.ctl[r].dbg = 1;
}

// Exports positions (per disk id), local times and active disks.
// (each may be null). failed: a word that is not 0 if nothing is to be written
// (or null).
__global__ void k_g_export(GDev s, double *x, double *t, int32_t *active, const int32_t *failed) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= s.n || (failed && *failed)) return;
    if (x) x[q] = s.g[q].x;
    if (t) t[q] = g_time(s.g[q].own, s.g[q].t, s.stamp0);
    if (active && q < s.k) active[q] = (int32_t)s.ci[q];
}

// Every disk back where it was when its frame was built (start).
__global__ void k_g_restore(GDev s, const double *start) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= s.n) return;
    GDisk &r = s.g[q];
    *reinterpret_cast<ulonglong2 *>(&r.x) = make_ulonglong2(dbits(start[q]), 0ull);
    r.own = OWN_STATIC;
    r.claim = 0ull;
}

// Direction change: the disks' x and y are exchanged (x from y_old, y from
// x_old); the graph is then rebuilt for the new frame.
__global__ void k_g_swap_xy(GDev s, double *xnew) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= s.n) return;
    const double xo = s.g[q].x;
    xnew[q] = s.y[q];
    s.y[q] = xo;
}

}  // namespace

// ------------------------------------------------------------------ host

struct GraphCtx {
    GDev s;
    int nc = 0;
    double box = 0.0;
    cudaStream_t st = nullptr;
    std::vector<void *> allocs;
    uint8_t *d_flags = nullptr;
    int32_t flags_cap = 0;
    int64_t log_legs = 0;  // legs logged so far (leg index of the log)
    GBatchScratch *launch = nullptr;  // launch tables of graph_run
    void *build_tmp = nullptr;        // scratch of graph_build
    GRing ring = {};
    int C = 4;                          // slots per cell of a build
    bool try_ring[2] = {false, false};  // per axis: its last frame was of rings, or none was
    int axis = 0;
    // Arrows may be open (the frame is new, and few legs may be all it runs): the
    // build that would complete them, and whether a launch has run since.
    bool places = false;  // s.pos is there; without rings it keeps the frame's start
    bool open = false, fresh = false;
    bool one_leg = false;  // one leg is all it runs
    GBuild build;
    std::vector<std::pair<void **, size_t>> pending;
    int64_t bytes = 0;  // device memory held
};

namespace {

// Device arrays of a context: requested one by one, then placed in a single
// allocation (each on a 256-byte boundary) by gcommit.
template <typename T>
void galloc(GraphCtx *g, T **ptr, size_t count) {
    *ptr = nullptr;
    g->pending.emplace_back((void **)ptr, std::max<size_t>(count, 1) * sizeof(T));
}

int gcommit(GraphCtx *g, std::string &err) {
    size_t total = 0;
    for (auto &r : g->pending) total += (r.second + 255) & ~(size_t)255;
    void *base = nullptr;
    if (total) {
        if (dm_alloc(&base, total) != 0) {
            g->pending.clear();
            err = "cudaMalloc failed (graph state)";
            return ECMC_ENOMEM;
        }
        g->allocs.push_back(base);
        g->bytes += (int64_t)total;
    }
    size_t off = 0;
    for (auto &r : g->pending) {
        *r.first = (char *)base + off;
        off += (r.second + 255) & ~(size_t)255;
    }
    g->pending.clear();
    return 0;
}

// Parts of a build's scratch (kept by the context for direction changes). All
// ones to start with: the FP32 coordinates, the ids per slot, the rows' least y;
// zero: the y bins, the counts (overfull cells, rows that are no rings, disks
// listed), the rows' largest y. Then the y limits of the blocks of columns and
// the list of disks.
struct BuildParts {
    size_t cid, ylo, zero, err, yhi, ylim, far, total;
    BuildParts(int64_t n, double L, double d, int nc, int C) {
        const size_t nslot = (size_t)nc * nc * C;
        const size_t nb = (size_t)((int)std::ceil(L / (d / 128.0)) + 1);
        auto after = [](size_t at, size_t bytes) { return (at + bytes + 15) & ~(size_t)15; };
        cid = after(0, nslot * sizeof(float2));
        ylo = after(cid, nslot * 4);
        zero = after(ylo, (size_t)nc * 8);  // (the bins)
        err = after(zero, (nb / 32 + 1) * 4);
        yhi = after(err, sizeof(BuildCounts));
        ylim = after(yhi, (size_t)nc * 8);
        far = after(ylim, (size_t)nc * (size_t)((nc + FAR_COLS - 1) / FAR_COLS) * sizeof(float4));
        total = after(far, 2 * (size_t)n * sizeof(uint32_t));
    }
};

static size_t graph_build_bytes(const GraphCtx *g) {
    return BuildParts(g->s.n, g->s.L, g->s.d, g->nc, g->C).total;
}

static int launched(const char *what, std::string &err) {
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) return 0;
    err = std::string(what) + ": " + cudaGetErrorString(e);
    return ECMC_ECUDA;
}

// The constants of a build.
static GBuild build_params(const GraphCtx *g) {
    const GDev &s = g->s;
    GBuild b;
    memset(&b, 0, sizeof b);
    b.n = s.n;
    b.nc = g->nc;
    b.L = s.L;
    b.d = s.d;
    b.d2 = s.d * s.d;
    b.a = g->box / g->nc;
    b.inv_a = (double)g->nc / s.L;
    const double w = s.d / 128.0;
    b.Lf = (float)s.L;
    b.af = (float)b.a;
    b.wf = (float)w;
    b.inv_wf = 1.0f / b.wf;
    b.half_f = (float)(0.5 * s.d);
    b.df = (float)s.d;
    b.del = (float)std::ldexp(b.a, -20);
    b.nb = (int)std::ceil(s.L / w) + 1;
    b.nblk = (g->nc + FAR_COLS - 1) / FAR_COLS;
    b.g = s.g;
    return b;
}

// The first half of a frame's build, queued on the context's stream: every
// disk in a cell, and whether the rows are rings (asked again on an axis only
// while they were: rows that motion across them has mixed stay mixed).
// check: coordinates outside [0, L), which count as the nearest cell's, are
// counted.
static int graph_place(GraphCtx *g, const double *x, const double *y, bool check, GBuild *out,
                       std::string &err) {
    GDev &s = g->s;
    const int nc = g->nc;
    GBuild b = build_params(g);
    b.x = x;
    b.y = y;
    b.yout = s.y;
    b.check = check ? 1 : 0;
    const BuildParts at(s.n, s.L, s.d, nc, g->C);
    // scratch of the build, kept by the context for the next direction change
    if (!g->build_tmp) {
        if (dm_alloc(&g->build_tmp, at.total) != 0) {
            g->build_tmp = nullptr;
            err = "cudaMalloc failed (graph build)";
            return ECMC_ENOMEM;
        }
        g->bytes += (int64_t)at.total;
    }
    char *tmp = (char *)g->build_tmp;
    b.cxy = (float2 *)tmp;
    b.scid = (uint32_t *)(tmp + at.cid);
    b.bits = (uint32_t *)(tmp + at.zero);
    g->ring.ylo = (unsigned long long *)(tmp + at.ylo);
    g->ring.yhi = (unsigned long long *)(tmp + at.yhi);
    b.count = (BuildCounts *)(tmp + at.err);
    b.ylim = (float4 *)(tmp + at.ylim);
    b.far = (uint32_t *)(tmp + at.far);
    cudaStream_t st = g->st;
    // (all ones: NaN coordinates and EMPTY ids)
    cudaMemsetAsync(tmp, 0xFF, at.zero, st);
    cudaMemsetAsync(tmp + at.zero, 0, at.ylim - at.zero, st);
    const unsigned nblk = (unsigned)((s.n + 255) / 256);
    if (g->C == 4)
        k_gb_cells<4><<<nblk, 256, 0, st>>>(b);
    else
        k_gb_cells<8><<<nblk, 256, 0, st>>>(b);
    if (g->try_ring[g->axis]) {
        const int chunks = ring_chunks(nc);
        const dim3 grid((unsigned)chunks, (unsigned)nc);
        if (g->C == 4)
            k_ring_count<4><<<grid, RING_CHUNK, 0, st>>>(b, g->ring);
        else
            k_ring_count<8><<<grid, RING_CHUNK, 0, st>>>(b, g->ring);
        k_ring_rows<<<1, 1024, 0, st>>>(b, g->ring, chunks);
    }
    *out = b;
    return launched("graph build", err);
}

// Legs that a frame's first launch may run with open arrows. An open arrow tells
// of a place at least (NEAR_COLS - 1) a - d ahead of the disk when the frame was
// built; a chain moves a disk by ell a leg at most, and on dense boxes by the
// gaps. Calls of few legs do not earn the search for these arrows back (with it
// 10^6 triangular disks at eta 0.60 took 1080 us to create, 460 so); before longer
// ones, and before a launch with other systems, it is done first. A launch in
// which a step comes to such a place is undone and run again with all arrows.
//
// On small boxes the search is cheap, and doing it apart costs as much again (two
// turns of 65536 disks and 16 legs: 923 us with it at the turn, 957 before the
// legs): only boxes of OPEN_DISKS or more, or a single leg, go without.
constexpr int64_t OPEN_DISKS = (int64_t)1 << 17;

static int open_legs(const GraphCtx *g) {
    return (int)std::min(8.0, NEAR_COLS * (g->box / g->nc) / g->s.ell);
}

// What a frame with open arrows keeps behind the disks' places (s.pos has 16 bytes
// a disk): the chains' disks, and the length of the log before the first launch.
static int32_t *graph_kept(const GraphCtx *g) { return (int32_t *)((double *)g->s.pos + g->s.n); }
static unsigned long long *graph_log_kept(const GraphCtx *g) {
    return (unsigned long long *)g->s.pos + g->s.n + (g->s.k + 1) / 2;
}

// The disks that k_gb_arrows listed, or (OPEN) those with open arrows.
template <int C, bool OPEN>
static void graph_far(const GraphCtx *g, cudaStream_t st) {
    const GBuild &b = g->build;
    // (with open arrows left open nothing listed needs the columns beyond)
    if (OPEN || !b.start) {
        const unsigned nb = (unsigned)std::min<size_t>(
            ((size_t)g->nc * (size_t)b.nblk * FAR_COLS + 255) / 256, 1216);
        k_gb_blocks<C><<<nb, 256, 0, st>>>(b, OPEN ? &b.count->open : &b.count->listed);
    }
    const unsigned nf = (unsigned)std::min<int64_t>(
        (b.n * FAR_LANES + FAR_THREADS - 1) / FAR_THREADS, FAR_BLOCKS);
    k_gb_far<C, OPEN><<<nf, FAR_THREADS, 0, st>>>(b);
}

// The second half: the records, along the rings (rings) or with the arrows of
// G(3), and the chains on their start disks (null: where they are).
static int graph_records(GraphCtx *g, const GBuild &b, bool rings, const int32_t *active,
                         std::string &err) {
    GDev &s = g->s;
    cudaStream_t st = g->st;
    s.ring = rings && g->try_ring[g->axis];
    g->try_ring[g->axis] = s.ring != 0;
    if (s.ring) {
        const dim3 grid((unsigned)ring_chunks(g->nc), (unsigned)g->nc);
        if (g->C == 4)
            k_ring_place<4><<<grid, RING_CHUNK, 0, st>>>(b, g->ring, s);
        else
            k_ring_place<8><<<grid, RING_CHUNK, 0, st>>>(b, g->ring, s);
    }
    g->fresh = true;
    g->open = !s.ring && s.cells && !s.strict && g->places && open_legs(g) >= 1 &&
              (g->one_leg || s.n >= OPEN_DISKS);
    g->build = b;
    g->build.start = g->open ? (double *)s.pos : nullptr;
    const unsigned ablk = (unsigned)(((size_t)g->nc * g->nc + BUILD_CELLS - 1) / BUILD_CELLS);
    if (s.ring && s.cells) {
        k_ring_records<<<(unsigned)((s.n + 255) / 256), 256, 0, st>>>(b, s);
    } else if (g->C == 4) {
        k_gb_arrows<4><<<ablk, 256, 0, st>>>(g->build);
        graph_far<4, false>(g, st);
    } else {
        k_gb_arrows<8><<<ablk, 256, 0, st>>>(g->build);
        graph_far<8, false>(g, st);
    }
    k_g_init_chains<<<(unsigned)((s.k + 127) / 128), 128, 0, st>>>(
        s, active, g->open ? graph_kept(g) : nullptr);
    return launched("graph build", err);
}

// Open arrows completed, on stream st.
static void graph_complete(GraphCtx *g, cudaStream_t st) {
    g->build.x = g->build.start;
    g->build.y = g->s.y;
    g->build.start = nullptr;
    if (g->C == 4)
        graph_far<4, true>(g, st);
    else
        graph_far<8, true>(g, st);
    g->open = false;
}

// A launch that an open arrow left undecided is undone: disks, chains and the
// length of the log as they were when the frame was built; the arrows completed.
static void graph_undo(GraphCtx *g, cudaStream_t st) {
    const GDev &s = g->s;
    k_g_restore<<<(unsigned)((s.n + 255) / 256), 256, 0, st>>>(s, g->build.start);
    k_g_init_chains<<<(unsigned)((s.k + 127) / 128), 128, 0, st>>>(s, graph_kept(g), nullptr);
    cudaMemsetAsync(s.dbg, 0, 16 * 8, st);
    if (s.log_on) cudaMemcpyAsync(s.tc_cnt, graph_log_kept(g), 8, cudaMemcpyDeviceToDevice, st);
    graph_complete(g, st);
}

// A frame from positions x, y and active disks (device): both halves, with a
// wait for the first one's counts between. check: the inputs are not known to be
// good (s.rid is zero then, for the ids seen). active: null, the disks are where
// they were.
static int graph_build(GraphCtx *g, const double *x, const double *y, const int32_t *active,
                       bool check, std::string &err) {
    const GDev &s = g->s;
    GBuild b;
    int rc = graph_place(g, x, y, check, &b, err);
    if (rc) return rc;
    if (check)
        graph_check_inputs(nullptr, nullptr, active, s.n, s.k, s.L, s.rid, nullptr,
                           &b.count->bad_id, g->st);
    BuildCounts h;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, b.count, sizeof h, cudaMemcpyDeviceToHost, g->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        err = std::string("graph build: ") + cudaGetErrorString(e);
        return ECMC_ECUDA;
    }
    if (h.bad_xy || h.bad_id) {
        err = h.bad_xy ? "coordinate outside [0, L)" : "active ids must be distinct and in [0, n)";
        return ECMC_EINVAL;
    }
    if (h.full) {
        err = "more disks in a cell than it has slots (overlapping input?)";
        return ECMC_ECAPACITY;
    }
    return graph_records(g, b, h.mixed == 0ull, active, err);
}

// Flag words of a context: one per disk, or per cell.
static size_t flag_words(const GDev &s) {
    return s.cells ? (size_t)s.nc * (size_t)s.nc : (size_t)s.n;
}

}  // namespace

// The device arrays of a context: take(pointer, count) for each.
template <class Take>
static void graph_arrays(GraphCtx *g, Take take) {
    GDev &s = g->s;
    const size_t n = (size_t)s.n, k = (size_t)s.k;
    const size_t path = k * ((size_t)s.cap + 2);
    take(&s.g, n);
    take(&s.y, n);
    take(&s.pos, g->places ? n : 0);
    take(&g->ring.off, g->places ? (size_t)g->nc * ring_chunks(g->nc) + 1 : 0);
    if (s.cells) {
        take(&s.pxt, path);
        take(&s.pcell, path);
    }
    take(&s.path, path);
    take(&s.ci, k);
    take(&s.ci0, k);
    take(&s.D, k);
    take(&s.tc, k);
    take(&s.status, k);
    take(&s.partner, k);
    take(&s.nlift, k);
    take(&s.tstar, 1);
    take(&s.rec, k * (size_t)s.cap);
    take(&s.ev_T, k);
    take(&s.ev_tau, k);
    take(&s.ev_xj, k);
    take(&s.ev_tj, k);
    take(&s.ev_j, k);
    take(&s.ev_a, 4 * k);
    take(&s.ev_lift, k);
    take(&s.vt, k);
    take(&s.uf, k);
    take(&s.fin, k);
    take(&s.comp_of, k);
    take(&s.abort_to, k);
    take(&s.comp_cnt, k);
    take(&s.comp_off, k + 1);
    take(&s.comp_root, k);
    take(&s.comp_mem, 4 * k);  // (g_members)
    take(&s.child, k);
    take(&s.sib, k);
    take(&s.ctl, CTL_N);
    if (s.log_on) take(&s.log, (size_t)s.log_cap);
    // all ones in a new context, from here on
    take(&s.keys, s.windows > 1 ? 2 * n : n);
    take(&s.memb, k);
    // zero, from here on
    take(&s.sp, k);
    take(&s.nrec, k);
    take(&s.taken, k);
    take(&s.lc, 2 * LC_N);
    take(&s.dbg, 16);
    take(&s.tc_cnt, TC_N);
    take(&s.fl, flag_words(s));
    take(&s.rid, n);
}

// Requests for all of them (galloc; gcommit allocates, graph_plan_bytes adds up).
static void graph_plan(GraphCtx *g) {
    graph_arrays(g, [&](auto **p, size_t count) { galloc(g, p, count); });
}

// Blocks of the persistent launch that fit on the current device at once (0:
// no cooperative launch there): queried once per device.
static int graph_max_grid() {
    static std::mutex mu;
    static int cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && cached[dev] > 0) return cached[dev];
    int n_sm = 1, blocks = 0, coop = 0;
    if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_run_graph, GRUN_THREADS,
                                                      UF_SMEM_BYTES) != cudaSuccess ||
        !coop || blocks < 1) {
        (void)cudaGetLastError();
        return 0;
    }
    const int grid = n_sm * std::min(blocks, GRUN_MIN_BLOCKS);
    if (dev >= 0 && dev < 64) cached[dev] = grid;
    return grid;
}

// A context's fields that follow from its parameters.
static void graph_params(GraphCtx *g, const ecmc_params *p, int nc) {
    g->nc = nc;
    g->box = p->box;
    GDev &s = g->s;
    memset(&s, 0, sizeof s);
    s.n = p->n;
    s.k = p->n_chains;
    s.nc = nc;
    s.cap = p->undo_cap > 0 ? p->undo_cap : 1024;
    s.windows = p->windows > 0 ? p->windows : 1;
    s.L = p->box;
    s.d = p->d;
    s.ell = p->ell;
    s.inv_a = (double)nc / p->box;
    s.strict = (s.windows > 1 || (p->flags & ECMC_RESTART)) ? 1 : 0;
    s.restart = (p->flags & ECMC_RESTART) ? 1 : 0;
    s.cells = (p->flags & ECMC_GRAPH) ? 0 : 1;
    const double a = p->box / nc;
    // slots per cell: at most 4 centres at mutual distance >= d fit in a cell
    // with a < sqrt(2) d, at most 6 for a < 1.664 d
    g->C = a < std::sqrt(2.0) * p->d * (1.0 - 1e-9) ? 4 : 8;
    // a leg along rings must not come round the box; a context may go without
    // (256 disks, 4 chains: a leg 31 us along the arrows of G(3), 23 along rings;
    // 2^20 disks, 1024 chains: 63 and 32)
    g->try_ring[0] = g->try_ring[1] =
        !(p->flags & ECMC_NO_ROWPASS) && p->ell < p->box - 3.0 * a;
    g->places = g->try_ring[0];
    // FP32 image of the scan's stop rule thr(m) = ((m a) - fx) - d > RN(cur +
    // eps): thr_f = ((m af - fxf) - df) and lim_f = trunc(cur) + epsf, with af,
    // df, epsf the FP32 roundings, fxf = trunc(fx). Each of the four FP32
    // roundings and the two truncations errs by at most 2^-23 of a term of
    // magnitude at most m a + a + d + cur + eps <= L + a + d + ell + eps (m < nc,
    // |fx| <= a, cur <= ell), so |(thr_f - lim_f) - (thr - lim)| < 2^-22 (L + a +
    // d + ell + eps) (the FP64 roundings are 2^29 times smaller). stop_e is 4
    // times that.
    const double eps = std::ldexp(p->box, -30);
    s.sk.a = a;
    s.sk.d = p->d;
    s.sk.eps = eps;
    s.sk.af = (float)a;
    s.sk.df = (float)p->d;
    s.sk.epsf = (float)eps;
    s.sk.stop_e = (float)std::ldexp(p->box + a + p->d + p->ell + eps + 1.0, -20);
    s.log_on = (p->flags & ECMC_LOG_LIFTINGS) ? 1 : 0;
    s.log_cap = s.log_on ? (p->log_cap > 0 ? p->log_cap : ((int64_t)1 << 22)) : 0;
}

// Counters, run results, flag words, touch keys, member tags and the ids seen of
// a new context (arrays side by side in the order of graph_arrays).
static cudaError_t graph_clear(GraphCtx *g) {
    GDev &s = g->s;
    s.key = s.keys;
    char *const ones = (char *)s.keys, *const zero = (char *)s.sp, *const end = (char *)(s.rid + s.n);
    const cudaError_t e = cudaMemsetAsync(ones, 0xFF, (size_t)(zero - ones), g->st);
    return e != cudaSuccess ? e : cudaMemsetAsync(zero, 0, (size_t)(end - zero), g->st);
}

int graph_create(const ecmc_params *p, int nc, const double *x, const double *y,
                 const int32_t *active, cudaStream_t st, GraphCtx **out, std::string &err) {
    *out = nullptr;
    if (p->n_chains > MAX_CHAINS) {
        err = "too many chains";
        return ECMC_EINVAL;
    }
    GraphCtx *g = new (std::nothrow) GraphCtx();
    if (!g) {
        err = "host allocation";
        return ECMC_ENOMEM;
    }
    g->st = st;
    graph_params(g, p, nc);
    graph_plan(g);
    int rc = gcommit(g, err);
    if (rc) {
        graph_destroy(g);
        return rc;
    }
    if (graph_clear(g) != cudaSuccess) {
        (void)cudaGetLastError();
        err = "clearing the graph state";
        rc = ECMC_ECUDA;
    }
    if (!rc) rc = graph_build(g, x, y, active, true, err);
    if (!rc && graph_max_grid() < 1) {
        err = "cooperative launch unavailable";
        rc = ECMC_ECUDA;
    }
    if (rc) {
        graph_destroy(g);
        return rc;
    }
    *out = g;
    return 0;
}

// Launch tables of the persistent kernel: one device block [reps | chain_base
// | comp_base | ctl | bar | g | phase] (256-byte aligned parts), uploaded
// whole before a launch and read back from ctl on after it.
struct GBatchScratch {
    int cap = 0;
    int64_t chains = 0;
    unsigned char *block = nullptr;
    // (and the flags of a run of one system, up to FLAG_TABLE legs)
    size_t off_flags = 0, off_base = 0, off_comp = 0, off_ctl = 0, off_bar = 0, off_g = 0, off_phase = 0,
           off_list = 0, total = 0;
    std::vector<unsigned char> host;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

void graph_batch_free(GBatchScratch *b) {
    if (!b) return;
    dm_free(b->block);
    if (b->ev0) cudaEventDestroy(b->ev0);
    if (b->ev1) cudaEventDestroy(b->ev1);
    delete b;
}

constexpr int32_t FLAG_TABLE = 1024;

static int launch_reserve(GBatchScratch **scratch, int n, int64_t chains, std::string &err) {
    GBatchScratch *b = *scratch;
    if (b && b->cap >= n && b->chains >= chains) return 0;
    const int cap = b && b->cap >= n ? b->cap : std::max(n, b ? 2 * b->cap : 1);
    chains = std::max(chains, b ? b->chains : 0);
    graph_batch_free(b);
    *scratch = nullptr;
    b = new (std::nothrow) GBatchScratch();
    if (!b) {
        err = "host allocation";
        return ECMC_ENOMEM;
    }
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    (void)take((size_t)cap * sizeof(GDev));
    b->off_base = take((size_t)(cap + 1) * sizeof(int32_t));
    b->off_comp = take((size_t)(cap + 1) * sizeof(int32_t));
    b->off_ctl = take((size_t)cap * sizeof(GCtl));
    b->off_bar = take(sizeof(unsigned int));
    b->off_g = take(GG_N * sizeof(int32_t));
    b->off_phase = take(GPH_N * sizeof(unsigned long long));
    b->off_flags = take(FLAG_TABLE);
    b->total = off;
    b->host.assign(off, 0);
    b->off_list = take((size_t)chains * sizeof(int32_t));  // (device only)
    if (dm_alloc_t(&b->block, off) != 0 || cudaEventCreate(&b->ev0) != cudaSuccess ||
        cudaEventCreate(&b->ev1) != cudaSuccess) {
        (void)cudaGetLastError();
        graph_batch_free(b);
        err = "launch tables";
        return ECMC_ENOMEM;
    }
    b->cap = cap;
    b->chains = chains;
    *scratch = b;
    return 0;
}

// Epochs (32-bit pass counts) and stamps (30-bit leg counts) of a context; far
// before one wraps (a launch makes fewer than 2^29 passes and 2^24 legs) both
// start again.
__global__ void k_g_clear_epochs(GDev s) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= s.n) return;
    GDisk &r = s.g[q];
    r.claim = 0ull;
    r.t = g_time(r.own, r.t, s.stamp0);
    if (g_static(r.own)) r.own = dbits(r.t) != 0ull ? 1u : 0u;
}

int graph_batch_run(GBatchScratch **scratch, GraphCtx *const *gs, int32_t n, int32_t max_legs,
                    const uint64_t *budgets, cudaStream_t st, GraphTotals *tots,
                    int32_t *legs_out, double *ms_out, std::string &err,
                    unsigned long long wait_ns) {
    if (ms_out) *ms_out = 0.0;
    if (n < 1 || max_legs < 0) {
        err = "bad batch size or leg count";
        return ECMC_EINVAL;
    }
    const int W = gs[0]->s.windows;
    for (int r = 0; r < n; ++r) {
        if (!gs[r] || gs[r]->s.windows != W) {
            err = "all contexts of a batch need the same claim windows";
            return ECMC_EINVAL;
        }
        if (gs[r]->s.restart && (n > 1 || scratch != &gs[r]->launch)) {
            err = "restart-mode contexts run alone (ecmc_run_to_breakpoint)";
            return ECMC_EINVAL;
        }
        if ((int64_t)max_legs * W >= ((int64_t)1 << 24)) {
            err = "too many legs x windows for one call (< 2^24)";
            return ECMC_EINVAL;
        }
    }
    for (int r = 0; r < n; ++r) {
        memset(&tots[r], 0, sizeof tots[r]);
        if (legs_out) legs_out[r] = 0;
    }
    if (max_legs == 0) return 0;
    int64_t chains = 0;
    for (int r = 0; r < n; ++r) chains += gs[r]->s.k;
    if (chains > 0x7FFFFFFF) {
        err = "too many chains in a batch";
        return ECMC_EINVAL;
    }
    int rc = launch_reserve(scratch, n, chains, err);
    if (rc) return rc;
    GBatchScratch *b = *scratch;
    auto cu = [&](cudaError_t e, const char *what) {
        if (e != cudaSuccess && !rc) {
            (void)cudaGetLastError();
            err = std::string(what) + ": " + cudaGetErrorString(e);
            rc = ECMC_ECUDA;
        }
    };
    unsigned char *h = b->host.data();
    memset(h, 0, b->total);
    GDev *S = (GDev *)h;
    int32_t *base = (int32_t *)(h + b->off_base);
    GCtl *ctl = (GCtl *)(h + b->off_ctl);
    chains = 0;
    for (int r = 0; r < n; ++r) {
        GraphCtx *g = gs[r];
        if (g->st != st) cu(cudaStreamSynchronize(g->st), "context stream");
        if (max_legs > FLAG_TABLE && g->flags_cap < max_legs) {
            dm_free(g->d_flags);
            g->d_flags = nullptr;
            g->flags_cap = 0;
            if (dm_alloc_t(&g->d_flags, (size_t)max_legs) != 0) {
                err = "flags allocation";
                return ECMC_ENOMEM;
            }
            g->flags_cap = max_legs;
        }
        // (open arrows are for one system and few legs from the frame's start)
        if (g->open && !(n == 1 && g->fresh && max_legs <= open_legs(g))) graph_complete(g, st);
        if (g->open && g->s.log_on)
            cu(cudaMemcpyAsync(graph_log_kept(g), g->s.tc_cnt, 8, cudaMemcpyDeviceToDevice, st),
               "log");
        g->fresh = false;
        if (g->s.epoch0 > 0xC0000000u || g->s.stamp0 > 0x3E000000u) {
            k_g_clear_epochs<<<(unsigned)((g->s.n + 255) / 256), 256, 0, st>>>(g->s);
            cu(cudaGetLastError(), "epochs");
            cu(cudaMemsetAsync(g->s.fl, 0, flag_words(g->s) * 8, st), "epochs");
            cu(cudaMemsetAsync(g->s.taken, 0, (size_t)g->s.k * 4, st), "epochs");
            g->s.epoch0 = 0;
            g->s.stamp0 = 1;  // (the last leg's times, for ecmc_positions)
        }
        S[r] = g->s;
        S[r].open = g->open ? 1 : 0;
        ctl[r].budget = budgets ? (int64_t)budgets[r] : 0;
        // (only a run of one system reports its flags)
        ctl[r].flags = n > 1                    ? nullptr
                       : max_legs <= FLAG_TABLE ? (uint8_t *)(b->block + b->off_flags)
                                                : g->d_flags;
        ctl[r].flags_cap = max_legs;
        ctl[r].leg0 = g->log_legs;
        base[r] = (int32_t)chains;
        chains += g->s.k;
        // member tags restart with the launch's window count
        cu(cudaMemsetAsync(g->s.memb, 0xFF, (size_t)g->s.k * 8, st), "memb");
    }
    base[n] = (int32_t)chains;
    cu(cudaMemcpyAsync(b->block, h, b->total, cudaMemcpyHostToDevice, st), "tables");
    if (rc) return rc;
    GBatchDev B;
    B.reps = (const GDev *)b->block;
    B.ctl = (GCtl *)(b->block + b->off_ctl);
    B.chain_base = (const int32_t *)(b->block + b->off_base);
    B.comp_base = (int32_t *)(b->block + b->off_comp);
    B.bar = (unsigned int *)(b->block + b->off_bar);
    B.g = (int32_t *)(b->block + b->off_g);
    B.phase_ns = (unsigned long long *)(b->block + b->off_phase);
    B.blocked = (int32_t *)(b->block + b->off_list);
    B.R = n;
    B.max_legs = max_legs;
    B.windows = W;
    B.pad = 0;
    B.wait_ns = wait_ns;
    const int grid = graph_max_grid();
    if (grid < 1) {
        err = "cooperative launch unavailable";
        return ECMC_ECUDA;
    }
    void *args[] = {&B};
    cu(cudaEventRecord(b->ev0, st), "event");
    cu(cudaLaunchCooperativeKernel((void *)k_run_graph, grid, GRUN_THREADS, args, UF_SMEM_BYTES,
                                   st),
       "launch");
    cu(cudaEventRecord(b->ev1, st), "event");
    cu(cudaMemcpyAsync(h + b->off_ctl, b->block + b->off_ctl, b->total - b->off_ctl,
                       cudaMemcpyDeviceToHost, st),
       "tables");
    cu(cudaStreamSynchronize(st), "run");
    if (rc) return rc;
    const int32_t *gg = (const int32_t *)(h + b->off_g);
    const unsigned long long *ph = (const unsigned long long *)(h + b->off_phase);
    float ms = 0.f;
    cu(cudaEventElapsedTime(&ms, b->ev0, b->ev1), "elapsed");
    if (ms_out) *ms_out = ms;
    bool cap_err = false;
    // (a launch that gave up on a wait may have made any number of passes)
    const bool timed_out = gg[GG_ERR] == ECMC_ETIMEOUT;
    const uint32_t passes =
        timed_out ? (uint32_t)max_legs * (uint32_t)W * (MAX_RESTARTS + 2u) : (uint32_t)gg[GG_PASSES];
    for (int r = 0; r < n; ++r) {
        const GCtl &c = ctl[r];
        if (c.open && !timed_out) {  // (n == 1)
            gs[r]->s.epoch0 += passes;
            gs[r]->s.stamp0 += (uint32_t)c.legs;
            graph_undo(gs[r], st);
            cu(cudaGetLastError(), "open arrows");
            return rc ? rc
                      : graph_batch_run(scratch, gs, n, max_legs, budgets, st, tots, legs_out,
                                        ms_out, err, wait_ns);
        }
        gs[r]->log_legs += c.legs;
        gs[r]->s.epoch0 += passes;
        gs[r]->s.stamp0 += timed_out ? (uint32_t)max_legs : (uint32_t)c.legs;
        GraphTotals &t = tots[r];
        t.legs = c.legs;
        t.lifts = c.lifts;
        t.conflict_legs = c.conflict_legs;
        t.repaired = c.repaired;
        t.continued = c.continued;
        t.restarts = c.restarts;
        t.horizon = c.horizon;
        t.order_err = c.order_err;
        t.p1_lifts = c.p1_lifts;
        t.repair_lifts = c.repair_lifts;
        t.blocked = c.blocked;
        t.cwindows = c.cwindows;
        t.row_windows = c.row_windows;
        if (n == 1) {
            t.ms = ms;
            t.pass1_ms = ph[GPH_PASS1] * 1e-6;
            t.repair_ms = ph[GPH_REPAIR] * 1e-6;
            t.other_ms = (ph[GPH_BEGIN] + ph[GPH_END]) * 1e-6;
        }
        if (legs_out) legs_out[r] = (int32_t)c.legs;
        if (c.err) cap_err = true;
    }
    if (timed_out) {
        err = "a grid barrier wait passed its time limit";
        return ECMC_ETIMEOUT;
    }
    if (cap_err) {
        err = "undo records or repair rounds overflowed";
        return ECMC_ECAPACITY;
    }
    for (int r = 0; r < n; ++r) {
        double dg[7];
        if (ctl[r].dbg &&
            cudaMemcpy(dg, gs[r]->s.dbg, sizeof dg, cudaMemcpyDeviceToHost) == cudaSuccess &&
            dg[0] != 0.0) {
            char buf[240];
            snprintf(buf, sizeof buf,
                     "internal check %g failed: %.17g %.17g %.17g %.17g %.17g %.17g", dg[0], dg[1],
                     dg[2], dg[3], dg[4], dg[5], dg[6]);
            err = buf;
            return ECMC_ECUDA;
        }
    }
    return 0;
}

int graph_run(GraphCtx *g, int32_t n_legs, uint64_t budget, uint8_t *flags_host,
              int32_t *legs_done, GraphTotals *tot, std::string &err,
              unsigned long long wait_ns) {
    memset(tot, 0, sizeof *tot);
    if (legs_done) *legs_done = 0;
    if (n_legs <= 0) return 0;
    int32_t legs = 0;
    const int rc = graph_batch_run(&g->launch, &g, 1, n_legs, &budget, g->st, tot, &legs, nullptr,
                                   err, wait_ns);
    if (legs_done) *legs_done = legs;
    if (flags_host && legs > 0 && n_legs <= FLAG_TABLE) {
        memcpy(flags_host, g->launch->host.data() + g->launch->off_flags, (size_t)legs);
    } else if (flags_host && legs > 0) {
        const cudaError_t e = cudaMemcpyAsync(flags_host, g->d_flags, (size_t)legs,
                                              cudaMemcpyDeviceToHost, g->st);
        if (e != cudaSuccess || cudaStreamSynchronize(g->st) != cudaSuccess) {
            (void)cudaGetLastError();
            err = "flags";
            return rc ? rc : ECMC_ECUDA;
        }
    }
    return rc;
}

int graph_export(GraphCtx *g, double *x, double *t, const double **y, const int32_t **active) {
    const GDev &s = g->s;
    *y = s.y;
    *active = (const int32_t *)s.ci;
    if (x || t)
        k_g_export<<<(unsigned)((s.n + 255) / 256), 256, 0, g->st>>>(s, x, t, nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? 0 : ECMC_ECUDA;
}

int graph_arrows(GraphCtx *g, int32_t *a, double *b, std::string &err) {
    const GDev &s = g->s;
    cudaStream_t st = g->st;
    // strided copies straight out of the 64-byte records
    cudaError_t e = cudaSuccess;
    if (a)
        e = cudaMemcpy2DAsync(a, 3 * sizeof(uint32_t), &s.g[0].a[0], sizeof(GDisk),
                              3 * sizeof(uint32_t), (size_t)s.n, cudaMemcpyDeviceToHost, st);
    if (b && e == cudaSuccess)
        e = cudaMemcpy2DAsync(b, 3 * sizeof(double), &s.g[0].b[0], sizeof(GDisk),
                              3 * sizeof(double), (size_t)s.n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        err = std::string("graph arrows: ") + cudaGetErrorString(e);
        return ECMC_ECUDA;
    }
    return 0;
}

int graph_transpose(GraphCtx *g, std::string &err) {
    GDev &s = g->s;
    double *xnew = nullptr;
    if (dm_alloc_t(&xnew, (size_t)s.n * 8) != 0) {
        err = "transpose scratch";
        return ECMC_ENOMEM;
    }
    k_g_swap_xy<<<(unsigned)((s.n + 255) / 256), 256, 0, g->st>>>(s, xnew);
    // records (x, t = 0) and arrows for the new frame
    g->axis ^= 1;
    int rc = graph_build(g, xnew, s.y, nullptr, false, err);
    if (rc == ECMC_ECAPACITY) {
        // (a cell overfull by overlapping disks; the records were not built) the
        // context stays as it was
        g->axis ^= 1;
        if (cudaMemcpyAsync(s.y, xnew, (size_t)s.n * 8, cudaMemcpyDeviceToDevice, g->st) !=
            cudaSuccess) {
            (void)cudaGetLastError();
            rc = ECMC_ECUDA;
        }
    }
    // (the build's kernels read xnew: done before the block goes back)
    if (cudaStreamSynchronize(g->st) != cudaSuccess && rc == 0) {
        (void)cudaGetLastError();
        err = "transpose";
        rc = ECMC_ECUDA;
    }
    dm_free(xnew);
    return rc;
}

int graph_liftings(GraphCtx *g, ecmc_lift_t *buf, int64_t cap, int64_t *n_out,
                   std::string &err) {
    const GDev &s = g->s;
    if (!s.log_on) {
        err = "lifting log not enabled";
        return ECMC_EINVAL;
    }
    unsigned long long n = 0;
    if (cudaMemcpy(&n, s.tc_cnt + TC_LOG_N, sizeof n, cudaMemcpyDeviceToHost) != cudaSuccess) {
        err = "log count";
        return ECMC_ECUDA;
    }
    *n_out = (int64_t)n;
    if ((int64_t)n > s.log_cap) {
        err = "lifting log overflowed log_cap";
        return ECMC_ECAPACITY;
    }
    std::vector<ecmc_lift_t> all((size_t)n);
    if (n && cudaMemcpy(all.data(), s.log, n * sizeof(ecmc_lift_t), cudaMemcpyDeviceToHost) !=
                 cudaSuccess) {
        err = "log copy";
        return ECMC_ECUDA;
    }
    std::stable_sort(all.begin(), all.end(), [](const ecmc_lift_t &a, const ecmc_lift_t &b) {
        return a.leg != b.leg ? a.leg < b.leg : a.c < b.c;
    });
    if (buf && cap > 0)
        memcpy(buf, all.data(), (size_t)std::min<int64_t>(cap, (int64_t)n) * sizeof(ecmc_lift_t));
    return 0;
}

void graph_destroy(GraphCtx *g) {
    if (!g) return;
    if (cudaStreamSynchronize(g->st) != cudaSuccess) (void)cudaGetLastError();
    for (void *p : g->allocs) dm_free(p);
    dm_free(g->build_tmp);
    dm_free(g->d_flags);
    graph_batch_free(g->launch);
    delete g;
}

int64_t graph_device_bytes(const GraphCtx *g) { return g ? g->bytes : 0; }

int64_t graph_plan_bytes(const ecmc_params *p, int nc) {
    GraphCtx *g = new (std::nothrow) GraphCtx();
    if (!g) return -1;
    graph_params(g, p, nc);
    graph_plan(g);
    int64_t total = (int64_t)graph_build_bytes(g);
    for (auto &r : g->pending) total += (int64_t)((r.second + 255) & ~(size_t)255);
    g->pending.clear();
    delete g;
    return total;
}

// -------------------------------------------- one leg on given memory

namespace {

// Tables of a launch of one system, as they lie on the device.
struct LegTables {
    GDev dev;
    int32_t chain_base[2], comp_base[2];
    GCtl ctl;
    unsigned bar;
    int32_t g[GG_N];
    unsigned long long phase[GPH_N];
};

// Places the arrays of a leg in [base, ...) on 256-byte boundaries (base null:
// only counts).
struct LegArrays {
    LegTables *tables;
    int32_t *blocked;
};

size_t leg_arrays(GraphCtx *g, unsigned char *base, LegArrays *out) {
    size_t off = 0;
    auto take = [&](auto **p, size_t count) {
        off = (off + 255) & ~(size_t)255;
        *p = base ? reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + off) : nullptr;
        off += std::max<size_t>(count, 1) * sizeof(**p);
    };
    graph_arrays(g, take);
    take(&out->tables, 1);
    take(&out->blocked, (size_t)g->s.k);
    char *tmp;
    take(&tmp, graph_build_bytes(g));
    g->build_tmp = tmp;
    return off;
}

}  // namespace

size_t graph_leg_bytes(const ecmc_params *p, int nc) {
    GraphCtx g;
    graph_params(&g, p, nc);
    LegArrays a;
    return leg_arrays(&g, nullptr, &a);
}

int graph_leg(const ecmc_params *p, int nc, unsigned char *base, double *x, const double *y,
              int32_t *active, double *t_out, cudaStream_t st, uint8_t *flag, int64_t *lifts,
              std::string &err) {
    GraphCtx g;
    g.st = st;
    graph_params(&g, p, nc);
    LegArrays a;
    (void)leg_arrays(&g, base, &a);
    GDev &s = g.s;
    int rc = 0;
    auto cu = [&](cudaError_t e) {
        if (e != cudaSuccess && !rc) {
            (void)cudaGetLastError();
            rc = ECMC_ECUDA;
        }
    };
    const int grid = graph_max_grid();
    if (grid < 1) return ECMC_ECUDA;
    g.one_leg = true;
    cu(graph_clear(&g));
    if (!rc) rc = graph_build(&g, x, y, active, true, err);
    if (rc) return rc;
    LegTables t;
    for (;;) {
        memset(&t, 0, sizeof t);
        t.dev = s;
        t.dev.open = g.open ? 1 : 0;
        t.chain_base[1] = s.k;
        t.ctl.failed = 1;
        GBatchDev B;
        B.reps = &a.tables->dev;
        B.ctl = &a.tables->ctl;
        B.chain_base = a.tables->chain_base;
        B.comp_base = a.tables->comp_base;
        B.bar = &a.tables->bar;
        B.g = a.tables->g;
        B.blocked = a.blocked;
        B.phase_ns = a.tables->phase;
        B.R = 1;
        B.max_legs = 1;
        B.windows = 1;
        B.pad = 0;
        B.wait_ns = BARRIER_TIMEOUT_NS;
        cu(cudaMemcpyAsync(a.tables, &t, sizeof t, cudaMemcpyHostToDevice, st));
        void *args[] = {&B};
        cu(cudaLaunchCooperativeKernel((void *)k_run_graph, grid, GRUN_THREADS, args,
                                       UF_SMEM_BYTES, st));
        if (!rc) {
            // (a leg out of records leaves the inputs as they are; one that gave up
            // on a wait never counted itself)
            const int32_t *const failed = &a.tables->ctl.failed;
            GDev done = s;
            done.stamp0 = s.stamp0 + 1;  // (the leg's times)
            k_g_export<<<(unsigned)((s.n + 255) / 256), 256, 0, st>>>(done, x, t_out, active,
                                                                      failed);
            cu(cudaGetLastError());
        }
        cu(cudaMemcpyAsync(&t, a.tables, sizeof t, cudaMemcpyDeviceToHost, st));
        cu(cudaStreamSynchronize(st));
        if (rc) return rc;
        if (!t.ctl.open || t.g[GG_ERR]) break;
        s.epoch0 += (uint32_t)t.g[GG_PASSES];
        s.stamp0 += 1;
        graph_undo(&g, st);
        cu(cudaMemsetAsync(s.memb, 0xFF, (size_t)s.k * 8, st));
        cu(cudaGetLastError());
    }
    if (t.ctl.err) return ECMC_ECAPACITY;
    if (t.g[GG_ERR] || t.ctl.dbg) return ECMC_ECUDA;
    if (flag) *flag = t.ctl.conflict_legs != 0;
    if (lifts) *lifts = t.ctl.lifts;
    return 0;
}
