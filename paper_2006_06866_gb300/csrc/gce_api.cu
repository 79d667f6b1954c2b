// C ABI of the CE search library: argument checks, the handle's device
// workspace, the per-call kernel sequence (init -> scan -> trial constants ->
// per-curve prep -> persistent CE kernel -> top-k merge), its capture into
// CUDA graphs, and the launch-shape autotuner.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <new>
#include <numeric>
#include <string>
#include <tuple>
#include <vector>

#include "gce_internal.cuh"
#include "gce_topk.cuh"
#include "gce_workspace.h"

using namespace gce;

namespace gce {

int most_tpt(int mode) { return mode == GCE_PHASE_FP64 ? 2 : 4; }

// The counter range of a job's SPLIT32 fold: narrow with a Pdot axis (every fold
// re-reduced), else the shape's (mid: warps with many cycles re-reduce).
int split_range(int mode, int n_pdots, int slot_range) {
    if (mode != GCE_PHASE_SPLIT32) return RANGE_WIDE;
    return n_pdots > 1 ? RANGE_NARROW : slot_range == 1 ? RANGE_MID : RANGE_WIDE;
}

// The launch shape of a job that was not tuned: 128 threads, and as many trials per
// thread as leave about 16 warps of counters on an SM.  More trials share a point's
// loads (and with a Pdot axis its period part) and give the fold independent chains;
// more warps hide the sweeps.  SM cycles per warp and point-trial, 40 curves x 600
// points x 1e5 trials, SPLIT32 / FIXED32, against the shape used before (256 x 2):
//   15 bins 128 x 4 3.53 / 4.23 (3.80 / 4.64), 20 bins 3.89 / 4.53 (4.11 / 4.88), 24
//   bins 4.41 / 4.87 and 128 x 2 4.29 / 5.01; 16 Pdot values: 15 bins 128 x 4 4.59 /
//   4.70 (5.51 / 5.46), 31 bins 5.78 / 6.15 (6.29 / 6.74), 40 bins 7.27 / 7.76 and
//   128 x 2 6.93 / 7.59; 50 bins 128 x 2 6.67 / 7.78 (8.84 / 7.55), 50 overlapping
//   bins 128 x 1 6.12 / 7.29 (9.15 / 7.38) and with Pdot 128 x 2 8.01 / 8.83 (8.01 /
//   8.69); 100 bins 128 x 1 11.2 / 11.6 (29.2 / 13.8).
// (A plan takes 256 threads where 128 leave fewer warps on an SM.)  With a Pdot axis
// a thread's trials are consecutive Pdot values, so few values leave some of its
// trials empty: the trials per thread also minimise the padded axis times the cost of
// a trial (1, 1.18, 1.7 at 4, 2, 1, from the figures above).
gce_tuning default_tuning(const gce_config *cfg, int n_pdots) {
    const int mode = cfg->phase_mode;
    const bool overlap = (cfg->flags & GCE_FLAG_OVERLAP) != 0;
    gce_tuning t;
    t.block = 128;
    t.ctas_per_sm = 0;
    t.chunk = 2048;
    t.slot_range = 1;
    const bool pd_axis = n_pdots > 1;
    const int slots = slots_per_trial(mode, cfg->n_phase_bins, split_range(mode, n_pdots, 1));
    t.tpt = slots <= (pd_axis ? 33 : 26) ? 4 : slots <= (overlap && !pd_axis ? 48 : 64) ? 2 : 1;
    t.tpt = std::min(t.tpt, most_tpt(mode));
    if (pd_axis) {
        auto cost = [&](int tpt) {
            return (double)((n_pdots + tpt - 1) / tpt * tpt) * (tpt == 4 ? 1.0 : tpt == 2 ? 1.18 : 1.7);
        };
        for (int tpt = t.tpt / 2; tpt >= 1; tpt /= 2)
            if (cost(tpt) < cost(t.tpt)) t.tpt = tpt;
    }
    return t;
}

// Jobs of so few warps (with one trial per thread) that fit_to_job leaves the default
// shape.  A tuned shape serves jobs of its own class: one tuned on a survey batch costs a
// single curve what its own shape gains (2000 points x 1000 periods, SPLIT32, the CE
// kernel: 0.088 ms with a batch's 128 x 4, 0.022 with its own), and the other way round.
static bool small_job(int mode, long long n_trials, int n_curves, int n_sm) {
    return (n_trials + 31) / 32 * n_curves <= (mode == GCE_PHASE_FP64 ? 24 : 20) * 4ll * n_sm;
}

// Fewer trials per thread where the job's trials would not fill the device
// otherwise.  w: warps per scheduler with one trial per thread.  SM cycles per warp
// and point-trial of 300-point curves, SPLIT32 at 1 / 2 / 4 trials per thread: w =
// 2.6 16.3 / 18.9 / -, w = 5.1 13.6 / 10.8 / 13.1, w = 8.2 - / 8.9 / 9.8, w = 16 - /
// 6.9 / 7.5, w = 41 - / 5.8 / 5.7; FP64, whose warps wait longer, w = 8.2 12.8 / 13.8,
// w = 16 10.5 / 9.2.
// Jobs with the significance keep at least two wherever 256 threads x 2 trials have
// always fitted (100 slots): its moments are summed per list of 64 trials.
// Returns whether the CTA's warps should share one trial set: their points are then
// counted 4 or 8 at a time, which pays while a curve's points, walked by a single
// warp, outlast the barriers.  Against the shapes above, at w = 0.05 / 0.26 / 1.0 /
// 2.6 / 4.1: 2000 points 286 -> 114, 57 -> 24, 16.9 -> 10.4, 7.8 -> 6.4, 7.6 -> 5.8
// (FIXED32); 811 points 385 -> 207, 77 -> 47, 22.6 -> 15.5, 10.1 -> 9.1, 9.2 -> 7.9;
// 300 points 670 -> 532, 139 -> 98, 37 -> 31, 16.7 -> 16.7, 13.8 -> 14.4; 100 points
// 1600 -> 1400, 320 -> 281, 84 -> 80, 36 -> 38, 29 -> 35.
bool fit_to_job(gce_tuning &t, const gce_config *cfg, int n_pdots, long long n_trials,
                       int n_curves, long long n_points, int n_sm, bool stats) {
    const int mode = cfg->phase_mode;
    const long long warps = (n_trials + 31) / 32 * n_curves, schedulers = 4ll * n_sm;
    const bool few = warps <= (mode == GCE_PHASE_FP64 ? 9 : 3) * schedulers;
    const bool keep2 =
        stats && slots_per_trial(mode, cfg->n_phase_bins, split_range(mode, n_pdots, 0)) <= 100;
    if (!(cfg->flags & GCE_FLAG_OVERLAP)) {
        const bool very_few = 10 * warps <= 3 * schedulers;
        // mean points per curve >= 200 w
        if (very_few || (warps <= 6 * schedulers &&
                         n_points / n_curves * schedulers >= 200 * warps)) {
            t.block = very_few ? 256 : 128;
            t.tpt = very_few && !keep2 ? 1 : 2;
            return true;
        }
    }
    if (mode == GCE_PHASE_FP64) {
        // As many as a FIXED32 job, which runs the same fold (a caller's own or the
        // tuner's shape has at most two).  100 curves x 1000 points x 2e4 periods, the
        // CE kernel: 0.85 ms with two, 0.80 with four; 23 x 487 x 1e4 x 16 Pdot 1.03 /
        // 0.87; 300 x 50..2000 x 1e4 0.80 / 0.70.  Near 20 w, where four leave one wave
        // and a bit, 20 x 200 points 0.076 / 0.079, from 25 w on 0.089 / 0.086.
        gce_config fixed = *cfg;
        fixed.phase_mode = GCE_PHASE_FIXED32;
        t.tpt = default_tuning(&fixed, n_pdots).tpt;
    }
    if (small_job(mode, n_trials, n_curves, n_sm)) t.tpt = std::min(t.tpt, 2);
    if (few && !stats) t.tpt = 1;
    if (keep2) {
        t.tpt = std::max(t.tpt, 2);
        if (few) t.block = 64;
    }
    return false;
}

}  // namespace gce

namespace {

// mode, n_phase, n_mag, log2 bucket of N, Pdot axis (n_pdots > 1: period-major tiles),
// size class (small_job)
typedef std::tuple<int, int, int, int, int, int> TuneKey;
// own: the tuner found the job's own shape the fastest (default_tuning, fit_to_job)
struct Tuned {
    gce_tuning t;
    bool own;
};

enum JobKind { JOB_GRID = 0, JOB_TOPK = 1, JOB_SINGLE = 2, JOB_COUNTS = 3 };

struct GraphKey {
    int kind, mode, n_curves, n_periods, n_pdots, n_phase, n_mag, k, block, tpt, grid, chunk,
        table_smem, grab;
    long long n_points;
    bool operator<(const GraphKey &o) const {
        return std::tie(kind, mode, n_curves, n_periods, n_pdots, n_phase, n_mag, k, block, tpt,
                        grid, chunk, table_smem, grab, n_points) <
               std::tie(o.kind, o.mode, o.n_curves, o.n_periods, o.n_pdots, o.n_phase, o.n_mag,
                        o.k, o.block, o.tpt, o.grid, o.chunk, o.table_smem, o.grab, o.n_points);
    }
};

// Everything a captured call sequence bakes into its nodes besides the launch
// shape (which the GraphKey holds): the caller's arrays, the epoch, the flags,
// and the handle's own workspace and pinned staging buffers.  A call whose
// fingerprint equals the cached graph's replays that graph as it is.
struct Fingerprint {
    uintptr_t v[40];
    int n = 0;
    void add(const void *p) { v[n++] = (uintptr_t)p; }
    void add_u(unsigned long long x) { v[n++] = (uintptr_t)x; }
    bool operator==(const Fingerprint &o) const {
        return n == o.n && std::memcmp(v, o.v, sizeof(uintptr_t) * (size_t)n) == 0;
    }
};

// The inputs of a launch shape's fitting (mode, bins, longest curve,
// slot range, the tuning's block / tpt / chunk / CTA cap) and its result, so
// that repeated calls skip the driver queries of the fitting.
typedef std::tuple<int, int, int, int, int, int, int, int, int> ShapeKey;
struct LaunchShape {
    int block, tpt, chunk, table_smem, occ;
    size_t smem;
};

constexpr int kCheckedArrays = 14;
constexpr int kWorkspaceBuffers = 12;

struct CachedGraph {
    cudaGraphExec_t exec = nullptr;
    Fingerprint fp;
    int launches = 0;  // kernels the sequence launches
};

}  // namespace

struct gce_handle_s {
    int device = 0;
    int n_sm = 0;
    int smem_optin = 0;
    std::string last_error;
    DevBuf payload, tau, seg, trialc, order, offsets, cand, stats, table, state, in_times, in_mags,
        in_periods, in_pdots, out_H, out_idx, band_stats, cand2, stats2;
    int table_n = -1;                    // largest count the table covers
    bool ask_memory = false;             // a growth to the coarse form has failed (job_buffers)
    int *h_order = nullptr;              // pinned staging
    long long *h_offsets = nullptr;
    size_t h_cap = 0;
    JobState *h_state = nullptr;         // pinned copy target for the check flags
    cudaEvent_t staged = nullptr;        // after the last job: workspace and staging buffers free
    bool staged_pending = false;
    cudaStream_t last_stream = nullptr;  // the stream of that event, and its id
    unsigned long long last_id = 0;
    int staged_n = -1;                   // curves whose offsets and order the buffers hold
    cudaEvent_t k0 = nullptr, k1 = nullptr;  // around the CE kernel (GCE_FLAG_TIME_KERNEL)
    bool timed = false;
    int launches = 0;                    // kernels the last job launched (directly or in its graph)
    std::map<TuneKey, Tuned> tune;
    std::map<GraphKey, CachedGraph> graphs;
    std::map<ShapeKey, LaunchShape> shapes;  // launch shapes already fitted to the device
    const void *checked[kCheckedArrays] = {};  // arrays of the last call found on the device
};

static std::string g_create_error;

static gce_status fail(gce_handle h, gce_status st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    if (h) h->last_error = buf;
    else g_create_error = buf;
    return st;
}

#define CUDA_TRY(h, expr)                                                                   \
    do {                                                                                    \
        cudaError_t e_ = (expr);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return fail((h), GCE_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e_)); \
    } while (0)

static const DevMemory kDevMemory = {
    [](void **p, size_t bytes) {
        if (cudaMalloc(p, bytes) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    },
    [](void *p) { cudaFree(p); },
    []() { return cudaDeviceSynchronize() == cudaSuccess; },
    []() {
        size_t free_bytes = 0, total = 0;
        if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) cudaGetLastError();
        return free_bytes;
    }};

static gce_status growth_status(gce_handle h, Growth g, size_t bytes) {
    if (g == GROWN) return GCE_OK;
    if (g == WAIT_FAILED)
        return fail(h, GCE_ERR_CUDA, "cudaDeviceSynchronize failed: %s", cudaGetErrorString(cudaGetLastError()));
    return fail(h, GCE_ERR_NOMEM, "device allocation of %zu bytes failed", bytes);
}

static gce_status ensure(gce_handle h, DevBuf &b, size_t bytes) {
    return growth_status(h, grow(kDevMemory, b, bytes), bytes);
}

static int point_bytes(int mode) {
    return coarse_mode(mode) ? (int)sizeof(CoarsePoint) : mode == GCE_PHASE_FP64 ? 8 : 16;
}

static size_t trial_bytes(int mode) {
    switch (mode) {
        case GCE_PHASE_FP64: return sizeof(ModeTraits<GCE_PHASE_FP64>::trial_t);
        case GCE_PHASE_SPLIT32: return sizeof(ModeTraits<GCE_PHASE_SPLIT32>::trial_t);
        default: return sizeof(ModeTraits<GCE_PHASE_FIXED32>::trial_t);
    }
}

static int ilog2_ceil(long long v) {
    int e = 0;
    while ((1ll << e) < v) ++e;
    return e;
}

static bool tuning_ok(const gce_tuning &t, int mode) {
    const bool block_ok = t.block == 64 || t.block == 128 || t.block == 256 || t.block == 512;
    const bool tpt_ok = t.tpt == 1 || t.tpt == 2 || (t.tpt == 4 && mode != GCE_PHASE_FP64);
    return block_ok && tpt_ok && t.ctas_per_sm >= 0 && t.ctas_per_sm <= 32 &&
           t.chunk >= 256 && t.chunk <= 8192 && t.chunk % 256 == 0 &&
           (t.slot_range == 0 || t.slot_range == 1);
}

static TuneKey tune_key(const gce_config *cfg, int n_obs, int pd_axis, bool small) {
    return TuneKey(cfg->phase_mode, cfg->n_phase_bins, cfg->n_mag_bins,
                   ilog2_ceil(std::max(n_obs, 1)), pd_axis, small ? 1 : 0);
}

// The cached shape for the key (a Pdot-axis job without its own entry uses the
// plain one), or the default one (*tuned = false).
static gce_tuning lookup_tuning(gce_handle h, const gce_config *cfg, int n_max, int n_pdots,
                                bool small, bool *tuned) {
    const int pd_axis = n_pdots > 1 ? 1 : 0;
    auto it = h->tune.find(tune_key(cfg, n_max, pd_axis, small));
    if (it == h->tune.end() && pd_axis) it = h->tune.find(tune_key(cfg, n_max, 0, small));
    *tuned = it != h->tune.end() && !it->second.own;
    return *tuned ? it->second.t : default_tuning(cfg, n_pdots);
}

extern "C" const char *gce_status_string(gce_status s) {
    switch (s) {
        case GCE_OK: return "ok";
        case GCE_ERR_INVALID: return "invalid argument or input value";
        case GCE_ERR_CUDA: return "CUDA error";
        case GCE_ERR_NOMEM: return "device memory exhausted";
        case GCE_ERR_UNSUPPORTED: return "input outside the range of the chosen phase fold";
        default: return "unknown status";
    }
}

extern "C" const char *gce_last_error(gce_handle h) {
    return h ? h->last_error.c_str() : g_create_error.c_str();
}

extern "C" gce_status gce_check_job(const int64_t *h_offsets, int32_t n_curves,
                                    int32_t n_periods, int32_t n_pdots, const gce_config *cfg,
                                    int32_t k) {
    if (!cfg) return GCE_ERR_INVALID;
    if (cfg->n_phase_bins < 1 || cfg->n_phase_bins > GCE_MAX_PHASE_BINS) return GCE_ERR_INVALID;
    if (cfg->n_mag_bins < 1 || cfg->n_mag_bins > GCE_MAX_MAG_BINS) return GCE_ERR_INVALID;
    if (cfg->phase_mode != GCE_PHASE_FP64 && cfg->phase_mode != GCE_PHASE_SPLIT32 &&
        cfg->phase_mode != GCE_PHASE_FIXED32)
        return GCE_ERR_INVALID;
    if (!std::isfinite(cfg->t0)) return GCE_ERR_INVALID;
    if ((cfg->flags & GCE_FLAG_OVERLAP) && cfg->n_phase_bins < 2) return GCE_ERR_INVALID;
    if (n_curves < 0 || n_periods < 1 || n_pdots < 1) return GCE_ERR_INVALID;
    const long long n_trials = (long long)n_periods * n_pdots;
    if (n_trials >= (1ll << 32)) return GCE_ERR_INVALID;
    if (k < 0 || k > GCE_MAX_TOPK || k > n_trials) return GCE_ERR_INVALID;
    if (n_curves > 0) {
        if (!h_offsets || h_offsets[0] != 0) return GCE_ERR_INVALID;
        for (int32_t c = 0; c < n_curves; ++c) {
            const long long n = h_offsets[c + 1] - h_offsets[c];
            if (n < 1 || n > GCE_MAX_CURVE_POINTS) return GCE_ERR_INVALID;
        }
    }
    return GCE_OK;
}

extern "C" gce_status gce_create(gce_handle *out, int32_t device) {
    if (!out) return fail(nullptr, GCE_ERR_INVALID, "gce_create: NULL output pointer");
    *out = nullptr;
    int n_dev = 0;
    cudaError_t e = cudaGetDeviceCount(&n_dev);
    if (e != cudaSuccess)
        return fail(nullptr, GCE_ERR_CUDA, "cudaGetDeviceCount: %s", cudaGetErrorString(e));
    if (device < 0 || device >= n_dev)
        return fail(nullptr, GCE_ERR_INVALID, "device %d out of range (%d devices)", device, n_dev);
    e = cudaSetDevice(device);
    if (e != cudaSuccess)
        return fail(nullptr, GCE_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(e));
    gce_handle h = new (std::nothrow) gce_handle_s();
    if (!h) return fail(nullptr, GCE_ERR_NOMEM, "host allocation failed");
    h->device = device;
    cudaDeviceGetAttribute(&h->n_sm, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&h->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (cudaEventCreateWithFlags(&h->staged, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreate(&h->k0) != cudaSuccess || cudaEventCreate(&h->k1) != cudaSuccess ||
        cudaMallocHost((void **)&h->h_state, sizeof(JobState)) != cudaSuccess) {
        e = cudaGetLastError();
        gce_destroy(h);
        return fail(nullptr, GCE_ERR_CUDA, "handle setup: %s", cudaGetErrorString(e));
    }
    if (ensure(h, h->state, sizeof(JobState)) != GCE_OK) {
        gce_destroy(h);
        return fail(nullptr, GCE_ERR_NOMEM, "workspace allocation failed");
    }
    *out = h;
    return GCE_OK;
}

extern "C" gce_status gce_destroy(gce_handle h) {
    if (!h) return GCE_ERR_INVALID;
    cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    for (auto &kv : h->graphs) cudaGraphExecDestroy(kv.second.exec);
    DevBuf *bufs[] = {&h->payload, &h->tau, &h->seg, &h->trialc, &h->order, &h->offsets, &h->cand, &h->stats,
                      &h->table, &h->state, &h->in_times, &h->in_mags, &h->in_periods,
                      &h->in_pdots, &h->out_H, &h->out_idx, &h->band_stats, &h->cand2,
                      &h->stats2};
    for (DevBuf *b : bufs)
        if (b->p) cudaFree(b->p);
    if (h->h_order) cudaFreeHost(h->h_order);
    if (h->h_offsets) cudaFreeHost(h->h_offsets);
    if (h->h_state) cudaFreeHost(h->h_state);
    if (h->staged) cudaEventDestroy(h->staged);
    if (h->k0) cudaEventDestroy(h->k0);
    if (h->k1) cudaEventDestroy(h->k1);
    delete h;
    return GCE_OK;
}

namespace {

struct Job {
    int kind;
    const double *times, *mags, *periods, *pdots;
    const int64_t *h_offsets;
    int n_curves, n_periods, n_pdots;
    const gce_config *cfg;
    int k;
    float *out;                  // grid (JOB_GRID, JOB_SINGLE)
    float *topk_H;               // JOB_TOPK
    int64_t *topk_idx;
    double *mean, *std_dev;      // JOB_TOPK with significance (rho != nullptr)
    float *rho;
    long long n_cells;           // JOB_COUNTS
    const int64_t *cell_curve, *cell_trial;
    uint32_t *counts;
    const gce_tuning *force;     // tuning override (autotuner)
    bool own;                    // the job's own shape, whatever is cached (autotuner)
    const unsigned char *bands;  // multi-filter input (nullptr: one filter, raw magnitudes)
    int n_bands;
};

struct Plan {
    long long n_points, n_trials, n_items, n_long_items;
    long long n_lists;    // top-k candidate lists per curve: tiles x warps
    int stats_per;        // moment records per candidate list
    int n_long, n_short;  // curves taken curve-major / tile-major (see MainArgs)
    int n_max, n_tiles, n_ptiles, pd_major, range, half, kv, block, tpt, grid, chunk, table_smem,
        grab;
    int n_groups, tiles_per_group;  // top-k: first merge level (0 groups: none)
    // the payload's fold mode: kernel_mode(), or the job's phase mode itself for the
    // diagnostic jobs and where the coarse payload (32 bytes per point and per trial
    // instead of FP64's 8 and 16 or FIXED32's 16 and 32) does not fit the device
    int prep_mode, kmode;  // kmode: the CE kernel's (main_mode)
    size_t smem;
};

// A launch shape fitted to the device for the plan's fold, slots and longest curve
// (cached per handle).
gce_status fit_shape(gce_handle h, const gce_config *cfg, const Plan &pl, const gce_tuning &t,
                     LaunchShape &ls) {
    const int kmode = pl.kmode, kv = pl.kv;
    const ShapeKey skey(kmode, cfg->n_phase_bins, cfg->n_mag_bins, pl.n_max,
                        pl.range * 8 + pl.half * 4 + kv, t.block, t.tpt, t.chunk, t.ctas_per_sm);
    auto sit = h->shapes.find(skey);
    if (sit != h->shapes.end()) {
        ls = sit->second;
        return GCE_OK;
    }
    ls.block = t.block;
    ls.tpt = t.tpt;
    ls.chunk = std::min(t.chunk, ((pl.n_max + 31) / 32) * 32);
    // the c ln c table in shared memory: the whole table when it has at most
    // 2048 entries (16 KB), so that lookups need no bounds test; longer curves
    // read counts above it from global memory
    ls.table_smem = std::min(pl.n_max + 1, 2048);
    // shrink the staged chunk, then the table, then trials per thread, then the
    // block, until the CTA fits in shared memory
    auto size = [&]() {
        return main_smem_bytes(kmode, trial_threads(kv, ls.block), ls.tpt, ls.chunk, cfg->n_phase_bins,
                               cfg->n_mag_bins, ls.table_smem, pl.range, pl.half);
    };
    auto limit = [&]() {
        return main_dynamic_smem_limit(kmode, ls.tpt, ls.block, kv, (size_t)h->smem_optin);
    };
    ls.smem = size();
    while (ls.smem > limit()) {
        if (ls.chunk > 512) ls.chunk = half_chunk(ls.chunk);
        else if (ls.table_smem > 256) ls.table_smem /= 2;
        else if (ls.tpt > 1) ls.tpt /= 2;
        else if (ls.block > 64) ls.block /= 2;
        else if (ls.chunk > 64) ls.chunk = half_chunk(ls.chunk);
        else break;
        ls.smem = size();
    }
    if (ls.smem > limit())
        return fail(h, GCE_ERR_UNSUPPORTED, "launch shape needs %zu bytes of shared memory", ls.smem);
    CUDA_TRY(h, main_kernel_attrs(kmode, ls.tpt, ls.block, kv, (size_t)h->smem_optin));
    const void *kern = main_kernel_ptr(kmode, ls.tpt, ls.block, kv);
    CUDA_TRY(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ls.occ, kern, ls.block, ls.smem));
    if (ls.occ < 1) return fail(h, GCE_ERR_UNSUPPORTED, "launch shape does not fit on an SM");
    // A smaller staged chunk costs only more staging passes: take it whenever it
    // admits more CTAs per SM (the counters leave little room at many phase bins, so
    // the tuned chunk can sit just past an occupancy step).
    // Every halving down to 256 points is tried; the largest chunk that reaches
    // the best occupancy is kept.
    int best_chunk = ls.chunk;
    size_t best_smem = ls.smem;
    for (int c = ls.chunk; c > 256;) {
        c = std::max(256, half_chunk(c));
        ls.chunk = c;
        const size_t sm2 = size();
        int occ2 = 0;
        CUDA_TRY(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, kern, ls.block, sm2));
        if (occ2 > ls.occ) {
            ls.occ = occ2;
            best_chunk = c;
            best_smem = sm2;
        }
    }
    ls.chunk = best_chunk;
    ls.smem = best_smem;
    h->shapes[skey] = ls;
    return GCE_OK;
}

// Curves of at most this many points are scheduled tile-major (Plan).
constexpr long long kShortCurve = 256;

gce_status make_plan(gce_handle h, const Job &j, Plan &pl) {
    const gce_config *cfg = j.cfg;
    pl.n_points = (long long)j.h_offsets[j.n_curves];
    pl.n_trials = (long long)j.n_periods * j.n_pdots;
    long long nmax = 1;
    for (int c = 0; c < j.n_curves; ++c) nmax = std::max<long long>(nmax, j.h_offsets[c + 1] - j.h_offsets[c]);
    pl.n_max = (int)nmax;
    bool tuned = true;
    gce_tuning t;
    if (j.force) t = *j.force;
    else if (j.own) t = default_tuning(cfg, j.n_pdots), tuned = false;
    else
        t = lookup_tuning(h, cfg, pl.n_max, j.n_pdots,
                          small_job(cfg->phase_mode, pl.n_trials, j.n_curves, h->n_sm), &tuned);
    const bool shared_set = !tuned && fit_to_job(t, cfg, j.n_pdots, pl.n_trials, j.n_curves,
                                                 pl.n_points, h->n_sm, j.rho != nullptr);
    pl.range = split_range(cfg->phase_mode, j.n_pdots, t.slot_range);
    // one Pdot value: the staging holds 8-byte half points
    pl.half = j.n_pdots == 1 ? 1 : 0;
    pl.prep_mode = (j.kind == JOB_GRID || j.kind == JOB_TOPK)
                       ? job_prep_mode(cfg, pl.n_trials, j.n_pdots, j.n_curves, h->n_sm)
                       : cfg->phase_mode;
    pl.kmode = main_mode(pl.prep_mode, cfg->phase_mode);
    // the kernel instantiation: overlapping bins, a shared trial set, or neither
    pl.kv = kernel_variant((cfg->flags & GCE_FLAG_OVERLAP) != 0);
    if (shared_set && pl.kv == KV_SNAP) pl.kv = KV_SHARED;
    const int kv = pl.kv;
    LaunchShape ls;
    if (gce_status st = fit_shape(h, cfg, pl, t, ls)) return st;
    if (!tuned && pl.kv != KV_SHARED && ls.block == 128 && ls.occ * ls.block < 512) {
        gce_tuning wide = t;
        wide.block = 256;
        LaunchShape lw;
        const std::string last = h->last_error;
        if (fit_shape(h, cfg, pl, wide, lw) != GCE_OK) h->last_error = last;
        else if (lw.tpt == ls.tpt && lw.occ * lw.block > ls.occ * ls.block) ls = lw;
    }
    pl.block = ls.block;
    pl.tpt = ls.tpt;
    pl.chunk = ls.chunk;
    pl.table_smem = ls.table_smem;
    pl.smem = ls.smem;
    int occ = ls.occ;
    const TileGrid tg = job_tiles(j.n_periods, j.n_pdots, trial_threads(kv, pl.block), pl.tpt);
    pl.n_tiles = (int)tg.n_tiles;
    pl.n_ptiles = tg.n_ptiles;
    pl.pd_major = tg.pd_major;
    pl.n_items = (long long)j.n_curves * pl.n_tiles;
    // curves of at most kShortCurve points run tile-major: a CTA then takes one
    // tile for several curves and loads its trial constants once
    pl.n_short = 0;
    for (int c = 0; c < j.n_curves; ++c)
        if (j.h_offsets[c + 1] - j.h_offsets[c] <= kShortCurve) ++pl.n_short;
    pl.n_long = j.n_curves - pl.n_short;
    pl.n_long_items = (long long)pl.n_long * pl.n_tiles;
    // each warp of a tile writes its own candidate list and its trial lists' moments
    pl.n_lists = (long long)pl.n_tiles * (trial_threads(kv, pl.block) / 32);
    pl.stats_per = pl.tpt == 4 ? 2 : 1;
    pl.n_groups = j.kind == JOB_TOPK ? topk_groups(pl.n_lists, j.k, &pl.tiles_per_group) : 0;
    if (j.kind != JOB_TOPK) pl.tiles_per_group = 0;
    if (t.ctas_per_sm > 0) occ = std::min(occ, t.ctas_per_sm);
    long long g = (long long)h->n_sm * occ;
    g = std::min(g, std::max(pl.n_items, 1ll));
    pl.grid = (int)g;
    // about 128 grabs per CTA: large enough to amortise the counter, small enough
    // that the last grabs leave little tail
    long long grab = pl.n_items / (g * 128);
    pl.grab = (int)std::max(1ll, std::min(grab, 64ll));
    return GCE_OK;
}

// Event around the CE kernel; under stream capture it becomes an event-record node.
gce_status mark(gce_handle h, cudaEvent_t e, cudaStream_t s, bool capturing) {
    if (capturing) CUDA_TRY(h, cudaEventRecordWithFlags(e, s, cudaEventRecordExternal));
    else CUDA_TRY(h, cudaEventRecord(e, s));
    return GCE_OK;
}

// Enqueue the whole sequence of one call on stream s (possibly under capture).
// pdl: launch the kernels with programmatic dependence.
gce_status enqueue(gce_handle h, const Job &j, const Plan &pl, cudaStream_t s, bool capturing,
                   bool pdl) {
    const gce_config *cfg = j.cfg;
    const int mode = pl.prep_mode;
    const int kmode = pl.kmode;
    JobState *st = (JobState *)h->state.p;
    int n_launch = 0;  // kernels this sequence launches, for gce_last_launches
    CUDA_TRY(h, launch_init(st, h->h_offsets, h->h_order, (long long *)h->offsets.p,
                            (int *)h->order.p, j.n_curves, s));
    CUDA_TRY(h, launch_scan(j.times, j.mags, pl.n_points, j.periods, j.n_periods, j.pdots,
                            j.n_pdots, cfg->t0, st, pdl, s));
    n_launch += 2;
    TrialArgs ta;
    ta.periods = j.periods;
    ta.pdots = j.pdots;
    ta.n_periods = j.n_periods;
    ta.n_pdots = j.n_pdots;
    ta.trialc = h->trialc.p;
    ta.state = st;
    CUDA_TRY(h, launch_trials(mode, ta, pdl, s));
    ++n_launch;
    PrepArgs pa;
    pa.times = j.times;
    pa.mags = j.mags;
    pa.offsets = (const long long *)h->offsets.p;
    pa.n_curves = j.n_curves;
    pa.n_mag = cfg->n_mag_bins;
    pa.t0 = cfg->t0;
    pa.payload = h->payload.p;
    pa.seg = (int *)h->seg.p;
    pa.tau = (double *)h->tau.p;
    pa.state = st;
    pa.bands = j.bands;
    pa.band_stats = (const double2 *)h->band_stats.p;
    pa.n_bands = j.bands ? j.n_bands : 0;
    if (j.bands) {
        CUDA_TRY(h, launch_band_stats(j.mags, j.bands, pa.offsets, j.n_curves, j.n_bands,
                                      (double2 *)h->band_stats.p, st, pdl, s));
        ++n_launch;
    }
    CUDA_TRY(h, launch_prep(mode, pa, pdl, s));
    ++n_launch;
    MainArgs ma;
    ma.payload = h->payload.p;
    ma.offsets = (const long long *)h->offsets.p;
    ma.seg = (const int *)h->seg.p;
    ma.trialc = h->trialc.p;
    ma.order = (const int *)h->order.p;
    ma.table = (const unsigned long long *)h->table.p;
    ma.n_trials = pl.n_trials;
    ma.n_periods = j.n_periods;
    ma.n_pdots = j.n_pdots;
    ma.n_tiles = pl.n_tiles;
    ma.n_ptiles = pl.n_ptiles;
    ma.pd_major = pl.pd_major;
    ma.range = pl.range;
    ma.n_items = pl.n_items;
    ma.n_long_items = pl.n_long_items;
    ma.n_long = pl.n_long;
    ma.n_short = pl.n_short;
    ma.grab = pl.grab;
    ma.n_phase = cfg->n_phase_bins;
    ma.n_mag = cfg->n_mag_bins;
    ma.chunk = pl.chunk;
    ma.table_smem = pl.table_smem;
    ma.out = nullptr;
    ma.cand = nullptr;
    ma.k = 0;
    ma.stats = nullptr;
    ma.overlap = (cfg->flags & GCE_FLAG_OVERLAP) ? 1 : 0;
    ma.half = pl.half;
    ma.kv = pl.kv;
    ma.pdl = pdl ? 1 : 0;
    ma.tau = (const double *)h->tau.p;
    ma.periods = j.periods;
    ma.pdots = j.pdots;
    ma.plain = mode == kmode ? 0 : 1;
    ma.state = st;
    const bool timed = (cfg->flags & GCE_FLAG_TIME_KERNEL) != 0;
    gce_status ms;
    switch (j.kind) {
        case JOB_GRID:
            ma.out = j.out;
            if (timed && (ms = mark(h, h->k0, s, capturing)) != GCE_OK) return ms;
            CUDA_TRY(h, launch_main(kmode, pl.tpt, pl.block, pl.grid, pl.smem, ma, s));
            ++n_launch;
            if (timed && (ms = mark(h, h->k1, s, capturing)) != GCE_OK) return ms;
            break;
        case JOB_TOPK:
            ma.cand = (unsigned long long *)h->cand.p;
            ma.k = j.k;
            if (j.rho) ma.stats = (TileStats *)h->stats.p;
            if (timed && (ms = mark(h, h->k0, s, capturing)) != GCE_OK) return ms;
            CUDA_TRY(h, launch_main(kmode, pl.tpt, pl.block, pl.grid, pl.smem, ma, s));
            ++n_launch;
            if (timed && (ms = mark(h, h->k1, s, capturing)) != GCE_OK) return ms;
            if (pl.n_groups > 0) {
                // many tiles per curve: reduce groups of tiles first, then merge the groups
                TileStats *stats2 = j.rho ? (TileStats *)h->stats2.p : nullptr;
                CUDA_TRY(h, launch_topk_reduce((const unsigned long long *)h->cand.p, j.n_curves,
                                               (int)pl.n_lists, j.k, pl.tiles_per_group, pl.n_groups,
                                               pl.stats_per, ma.stats, (unsigned long long *)h->cand2.p, stats2,
                                               st, pdl, s));
                CUDA_TRY(h, launch_topk_merge((const unsigned long long *)h->cand2.p, j.n_curves,
                                              pl.n_groups, j.k, 1, j.topk_H, (long long *)j.topk_idx,
                                              stats2, j.mean, j.std_dev, j.rho, st, pdl, s));
                n_launch += 2;
            } else {
                CUDA_TRY(h, launch_topk_merge((const unsigned long long *)h->cand.p, j.n_curves,
                                              (int)pl.n_lists, j.k, pl.stats_per, j.topk_H,
                                              (long long *)j.topk_idx, ma.stats, j.mean, j.std_dev, j.rho, st, pdl, s));
                ++n_launch;
            }
            break;
        case JOB_SINGLE:
            ma.out = j.out;
            if (timed && (ms = mark(h, h->k0, s, capturing)) != GCE_OK) return ms;
            for (int c = 0; c < j.n_curves; ++c) CUDA_TRY(h, launch_single(ma, c, 0, s));
            n_launch += j.n_curves;
            if (timed && (ms = mark(h, h->k1, s, capturing)) != GCE_OK) return ms;
            break;
        case JOB_COUNTS:
            CUDA_TRY(h, cudaMemsetAsync(j.counts, 0,
                                        sizeof(uint32_t) * (size_t)j.n_cells * cfg->n_mag_bins *
                                            cfg->n_phase_bins, s));
            CUDA_TRY(h, launch_counts(mode, ma, j.n_cells, (const long long *)j.cell_curve,
                                      (const long long *)j.cell_trial, (unsigned int *)j.counts, s));
            if (j.n_cells > 0) ++n_launch;
            break;
    }
    h->launches += n_launch;
    return GCE_OK;
}

// A device array must be on the handle's device: memory the runtime reports as
// another device's is rejected (managed and host-registered memory is left to
// the driver).
bool on_device(const void *ptr, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return a.type != cudaMemoryTypeDevice || a.device == dev;
}

gce_status run_job(gce_handle h, const Job &j, cudaStream_t s) {
    if (!h) return GCE_ERR_INVALID;
    h->launches = 0;
    const gce_status chk = gce_check_job(j.h_offsets, j.n_curves, j.n_periods, j.n_pdots, j.cfg,
                                         j.kind == JOB_TOPK ? j.k : 0);
    if (chk != GCE_OK) return fail(h, chk, "argument check failed");
    if (j.kind == JOB_TOPK && j.k < 1) return fail(h, GCE_ERR_INVALID, "k must be >= 1");
    if (j.kind == JOB_SINGLE && j.cfg->phase_mode != GCE_PHASE_FP64)
        return fail(h, GCE_ERR_INVALID, "the one-launch-per-curve baseline is FP64 only");
    if (j.n_curves == 0) return GCE_OK;
    if (!j.times || !j.mags || !j.periods || !j.pdots)
        return fail(h, GCE_ERR_INVALID, "NULL input array");
    if ((j.kind == JOB_GRID || j.kind == JOB_SINGLE) && !j.out)
        return fail(h, GCE_ERR_INVALID, "NULL output array");
    if (j.kind == JOB_TOPK && (!j.topk_H || !j.topk_idx))
        return fail(h, GCE_ERR_INVALID, "NULL output array");
    if (j.kind == JOB_TOPK && (j.rho || j.mean || j.std_dev) && !(j.rho && j.mean && j.std_dev))
        return fail(h, GCE_ERR_INVALID, "significance needs all of mean, std and rho");
    if (j.kind == JOB_COUNTS && j.n_cells > 0 && (!j.cell_curve || !j.cell_trial || !j.counts))
        return fail(h, GCE_ERR_INVALID, "NULL cell array");
    if (j.bands && (j.n_bands < 1 || j.n_bands > GCE_MAX_BANDS))
        return fail(h, GCE_ERR_INVALID, "n_bands must be 1 .. %d", GCE_MAX_BANDS);
    CUDA_TRY(h, cudaSetDevice(h->device));
    // The job waits on the device for the handle's last one, which may still use the
    // workspace, unless that ran on the very same stream (a small call is bound by the
    // host, and the wait would take 1 to 3 of its 36 us).  A stream's handle value does
    // not identify it: a destroyed stream's is given out again, so the ids are compared,
    // and the per-thread default stream has one value in every thread, so it never
    // counts as the same.  A stream that the caller is capturing cannot wait for an
    // event from outside the capture: there the host waits.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (s != nullptr) CUDA_TRY(h, cudaStreamIsCapturing(s, &cap));
    const bool captured = cap != cudaStreamCaptureStatusNone;
    unsigned long long stream_id = 0;
    if (s != nullptr && !captured) CUDA_TRY(h, cudaStreamGetId(s, &stream_id));
    if (h->staged_pending && captured) {
        CUDA_TRY(h, cudaEventSynchronize(h->staged));
        h->staged_pending = false;
    } else if (h->staged_pending &&
               (s != h->last_stream || stream_id != h->last_id || s == cudaStreamPerThread)) {
        CUDA_TRY(h, cudaStreamWaitEvent(s, h->staged, 0));
    }
    {
        // arrays already checked by the previous call (same argument, same
        // pointer) need no new query
        const void *arrays[kCheckedArrays] = {j.times, j.mags, j.periods, j.pdots, j.out,
                                              j.topk_H, j.topk_idx, j.mean, j.std_dev, j.rho,
                                              j.cell_curve, j.cell_trial, j.counts, j.bands};
        for (int i = 0; i < kCheckedArrays; ++i) {
            if (arrays[i] && arrays[i] != h->checked[i] && !on_device(arrays[i], h->device)) {
                std::fill(h->checked, h->checked + kCheckedArrays, nullptr);
                return fail(h, GCE_ERR_INVALID, "an array is on another device than the handle's");
            }
            h->checked[i] = arrays[i];
        }
    }

    Plan pl;
    gce_status st = make_plan(h, j, pl);
    if (st != GCE_OK) return st;

    // workspace (the first three buffers' size depends on the payload's form)
    const bool new_table = pl.n_max > h->table_n;
    const size_t nc = (size_t)j.n_curves, lists = nc * (size_t)pl.n_lists;
    const bool topk = j.kind == JOB_TOPK;
    auto needs = [&](int mode, Need (&need)[kWorkspaceBuffers]) {
        const Need all[kWorkspaceBuffers] = {
            {&h->payload, (size_t)point_bytes(mode) * pl.n_points},
            {&h->trialc, trial_bytes(mode) * (size_t)pl.n_trials},
            {&h->tau, coarse_mode(mode) ? 8 * (size_t)pl.n_points : 0},
            {&h->seg, sizeof(int) * nc * (j.cfg->n_mag_bins + 1)},
            {&h->order, sizeof(int) * nc},
            {&h->offsets, sizeof(long long) * (nc + 1)},
            {&h->band_stats, j.bands ? sizeof(double2) * nc * j.n_bands : 0},
            {&h->cand, topk ? 8 * lists * j.k : 0},
            {&h->stats, topk && j.rho ? sizeof(TileStats) * lists * pl.stats_per : 0},
            {&h->cand2, topk ? 8 * nc * pl.n_groups * j.k : 0},
            {&h->stats2, topk && j.rho ? sizeof(TileStats) * nc * pl.n_groups : 0},
            {&h->table, new_table ? 8 * (size_t)(pl.n_max + 1) : 0}};
        std::copy(all, all + kWorkspaceBuffers, need);
    };
    Need coarse[kWorkspaceBuffers], plain[kWorkspaceBuffers];
    const bool try_coarse = coarse_mode(pl.prep_mode);
    needs(pl.prep_mode, coarse);
    needs(try_coarse ? j.cfg->phase_mode : pl.prep_mode, plain);
    if (new_table) h->table_n = -1;  // (growing loses its contents)
    bool is_coarse = false;
    size_t most = 0;
    for (const Need &x : plain) most = std::max(most, x.bytes);
    st = growth_status(h, job_buffers(kDevMemory, try_coarse ? coarse : nullptr, plain,
                                      kWorkspaceBuffers, 3, &is_coarse, &h->ask_memory), most);
    if (st != GCE_OK) return st;
    if (try_coarse && !is_coarse) pl.prep_mode = j.cfg->phase_mode;
    const int mode = pl.prep_mode;
    if (new_table) {
        CUDA_TRY(h, launch_table((unsigned long long *)h->table.p, pl.n_max, s));
        ++h->launches;
        if (!captured) h->table_n = pl.n_max;  // (a captured launch has filled nothing yet)
    }

    // host staging (pinned): offsets and the longest-first curve order.  Every job's
    // first kernel reads them; a job whose offsets are those already staged leaves
    // the buffers alone and need not wait for the jobs before it.
    if (h->staged_n != j.n_curves ||
        std::memcmp(h->h_offsets, j.h_offsets, sizeof(long long) * (j.n_curves + 1)) != 0) {
        if (h->staged_pending) CUDA_TRY(h, cudaEventSynchronize(h->staged));
        h->staged_n = -1;
        if ((size_t)j.n_curves + 1 > h->h_cap) {
            if (h->h_order) cudaFreeHost(h->h_order);
            if (h->h_offsets) cudaFreeHost(h->h_offsets);
            h->h_order = nullptr;
            h->h_offsets = nullptr;
            h->h_cap = 0;
            size_t cap = (size_t)j.n_curves + 1;
            CUDA_TRY(h, cudaMallocHost((void **)&h->h_order, sizeof(int) * cap));
            CUDA_TRY(h, cudaMallocHost((void **)&h->h_offsets, sizeof(long long) * cap));
            h->h_cap = cap;
        }
        std::memcpy(h->h_offsets, j.h_offsets, sizeof(long long) * (j.n_curves + 1));
        std::iota(h->h_order, h->h_order + j.n_curves, 0);
        std::stable_sort(h->h_order, h->h_order + j.n_curves, [&](int a, int b) {
            return j.h_offsets[a + 1] - j.h_offsets[a] > j.h_offsets[b + 1] - j.h_offsets[b];
        });
        h->staged_n = j.n_curves;
    }

    const bool use_graph = !(j.cfg->flags & GCE_FLAG_NO_GRAPH) && s != nullptr &&
                           j.kind != JOB_SINGLE;
    h->timed = (j.cfg->flags & GCE_FLAG_TIME_KERNEL) != 0 && j.kind != JOB_COUNTS;
    if (!use_graph) {
        st = enqueue(h, j, pl, s, false, !captured);
        if (st != GCE_OK) {
            // the kernels before the one that failed may be on the stream
            if (!captured && cudaEventRecord(h->staged, s) == cudaSuccess) {
                h->staged_pending = true;
                h->last_stream = s;
                h->last_id = stream_id;
            }
            return st;
        }
    } else {
        GraphKey key{j.kind * 8 + (j.bands ? 4 : 0) + (j.rho ? 2 : 0) +
                         ((j.cfg->flags & GCE_FLAG_OVERLAP) ? 1 : 0),
                     mode, j.n_curves, j.n_periods, j.n_pdots, j.cfg->n_phase_bins,
                     j.cfg->n_mag_bins, j.k, pl.block, pl.tpt, pl.grid, pl.chunk, pl.table_smem,
                     pl.grab, pl.n_points};
        Fingerprint fp;
        const void *ptrs[] = {j.times, j.mags, j.periods, j.pdots, j.out, j.topk_H, j.topk_idx,
                              j.mean, j.std_dev, j.rho, j.cell_curve, j.cell_trial, j.counts,
                              j.bands, h->payload.p, h->seg.p, h->trialc.p, h->order.p,
                              h->offsets.p, h->cand.p, h->stats.p, h->cand2.p, h->stats2.p,
                              h->table.p, h->state.p, h->band_stats.p, h->h_order, h->h_offsets,
                              h->tau.p};
        for (const void *p : ptrs) fp.add(p);
        unsigned long long t0_bits;
        std::memcpy(&t0_bits, &j.cfg->t0, sizeof(t0_bits));
        fp.add_u(t0_bits);
        fp.add_u(j.cfg->flags);
        fp.add_u((unsigned long long)j.n_bands);
        fp.add_u((unsigned long long)j.n_cells);
        fp.add_u((unsigned long long)pl.n_long);
        fp.add_u((unsigned long long)pl.prep_mode);
        fp.add_u((unsigned long long)((pl.kmode * 8 + pl.kv) * 8 + pl.range));
        auto it = h->graphs.find(key);
        if (it != h->graphs.end() && it->second.fp == fp) {
            // same shape and the same arrays as the cached graph: replay it as it is
            h->launches += it->second.launches;
        } else {
            const int before = h->launches;
            cudaGraph_t graph = nullptr;
            CUDA_TRY(h, cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
            st = enqueue(h, j, pl, s, true, false);
            cudaError_t e = cudaStreamEndCapture(s, &graph);
            if (st != GCE_OK) {
                if (graph) cudaGraphDestroy(graph);
                return st;
            }
            if (e != cudaSuccess) return fail(h, GCE_ERR_CUDA, "graph capture: %s", cudaGetErrorString(e));
            bool ready = false;
            if (it != h->graphs.end()) {
                // same shape, other arrays: update the cached graph's parameters
                cudaGraphExecUpdateResultInfo info;
                if (cudaGraphExecUpdate(it->second.exec, graph, &info) == cudaSuccess) {
                    ready = true;
                } else {
                    cudaGetLastError();
                    if (h->staged_pending) cudaEventSynchronize(h->staged);
                    cudaGraphExecDestroy(it->second.exec);
                    h->graphs.erase(it);
                }
            }
            if (!ready) {
                cudaGraphExec_t exec = nullptr;
                e = cudaGraphInstantiate(&exec, graph, 0);
                if (e != cudaSuccess) {
                    cudaGraphDestroy(graph);
                    return fail(h, GCE_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
                }
                if (h->graphs.size() > 64) {
                    if (h->staged_pending) cudaEventSynchronize(h->staged);
                    for (auto &kv : h->graphs) cudaGraphExecDestroy(kv.second.exec);
                    h->graphs.clear();
                }
                h->graphs[key].exec = exec;
            }
            cudaGraphDestroy(graph);
            CachedGraph &cg = h->graphs[key];
            cg.fp = fp;
            cg.launches = h->launches - before;
        }
        CUDA_TRY(h, cudaGraphLaunch(h->graphs[key].exec, s));
    }
    if (captured) return GCE_OK;  // nothing has been submitted
    CUDA_TRY(h, cudaEventRecord(h->staged, s));
    h->staged_pending = true;
    h->last_stream = s;
    h->last_id = stream_id;
    return GCE_OK;
}

gce_status state_status(gce_handle h) {
    const unsigned int e = h->h_state->err;
    if (e & (ERR_TIME | ERR_PERIOD | ERR_PDOT | ERR_BAND))
        return fail(h, GCE_ERR_INVALID, "device check: %s%s%s%s",
                    (e & ERR_TIME) ? "non-finite time or magnitude; " : "",
                    (e & ERR_PERIOD) ? "non-finite or non-positive period; " : "",
                    (e & ERR_PDOT) ? "non-finite period derivative; " : "",
                    (e & ERR_BAND) ? "filter index >= n_bands; " : "");
    if (e & ERR_RANGE)
        return fail(h, GCE_ERR_UNSUPPORTED, "device check: trial range beyond the phase fold's range");
    if (e & ERR_SLOT)
        return fail(h, GCE_ERR_CUDA, "checked build: a counter slot outside the kept range");
    return GCE_OK;
}

}  // namespace

extern "C" gce_status gce_ce_grid(gce_handle h, const double *times, const double *mags,
                                  const int64_t *h_offsets, int32_t n_curves,
                                  const double *periods, int32_t n_periods, const double *pdots,
                                  int32_t n_pdots, const gce_config *cfg, float *out,
                                  void *stream) {
    Job j{};
    j.kind = JOB_GRID;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.out = out;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_topk(gce_handle h, const double *times, const double *mags,
                                  const int64_t *h_offsets, int32_t n_curves,
                                  const double *periods, int32_t n_periods, const double *pdots,
                                  int32_t n_pdots, const gce_config *cfg, int32_t k,
                                  float *topk_H, int64_t *topk_idx, void *stream) {
    Job j{};
    j.kind = JOB_TOPK;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.k = k; j.topk_H = topk_H; j.topk_idx = topk_idx;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_detect(gce_handle h, const double *times, const double *mags,
                                    const int64_t *h_offsets, int32_t n_curves,
                                    const double *periods, int32_t n_periods,
                                    const double *pdots, int32_t n_pdots, const gce_config *cfg,
                                    int32_t k, float *topk_H, int64_t *topk_idx, double *mean,
                                    double *std_dev, float *rho, void *stream) {
    if (!mean || !std_dev || !rho) return h ? fail(h, GCE_ERR_INVALID, "NULL moment output") : GCE_ERR_INVALID;
    Job j{};
    j.kind = JOB_TOPK;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.k = k; j.topk_H = topk_H; j.topk_idx = topk_idx;
    j.mean = mean; j.std_dev = std_dev; j.rho = rho;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_grid_bands(gce_handle h, const double *times, const double *mags,
                                        const uint8_t *bands, int32_t n_bands,
                                        const int64_t *h_offsets, int32_t n_curves,
                                        const double *periods, int32_t n_periods,
                                        const double *pdots, int32_t n_pdots,
                                        const gce_config *cfg, float *out, void *stream) {
    if (!bands) return h ? fail(h, GCE_ERR_INVALID, "NULL band array") : GCE_ERR_INVALID;
    Job j{};
    j.kind = JOB_GRID;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.out = out;
    j.bands = bands; j.n_bands = n_bands;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_detect_bands(gce_handle h, const double *times, const double *mags,
                                          const uint8_t *bands, int32_t n_bands,
                                          const int64_t *h_offsets, int32_t n_curves,
                                          const double *periods, int32_t n_periods,
                                          const double *pdots, int32_t n_pdots,
                                          const gce_config *cfg, int32_t k, float *topk_H,
                                          int64_t *topk_idx, double *mean, double *std_dev,
                                          float *rho, void *stream) {
    if (!bands) return h ? fail(h, GCE_ERR_INVALID, "NULL band array") : GCE_ERR_INVALID;
    Job j{};
    j.kind = JOB_TOPK;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.k = k; j.topk_H = topk_H; j.topk_idx = topk_idx;
    j.mean = mean; j.std_dev = std_dev; j.rho = rho;
    j.bands = bands; j.n_bands = n_bands;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_grid_single(gce_handle h, const double *times, const double *mags,
                                         const int64_t *h_offsets, int32_t n_curves,
                                         const double *periods, int32_t n_periods,
                                         const double *pdots, int32_t n_pdots,
                                         const gce_config *cfg, float *out, void *stream) {
    Job j{};
    j.kind = JOB_SINGLE;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.out = out;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_ce_counts(gce_handle h, const double *times, const double *mags,
                                    const int64_t *h_offsets, int32_t n_curves,
                                    const double *periods, int32_t n_periods,
                                    const double *pdots, int32_t n_pdots, const gce_config *cfg,
                                    int64_t n_cells, const int64_t *cell_curve,
                                    const int64_t *cell_trial, uint32_t *counts, void *stream) {
    if (n_cells < 0) return GCE_ERR_INVALID;
    Job j{};
    j.kind = JOB_COUNTS;
    j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = n_curves;
    j.periods = periods; j.n_periods = n_periods; j.pdots = pdots; j.n_pdots = n_pdots;
    j.cfg = cfg; j.n_cells = n_cells; j.cell_curve = cell_curve; j.cell_trial = cell_trial;
    j.counts = counts;
    return run_job(h, j, (cudaStream_t)stream);
}

extern "C" gce_status gce_stream_status(gce_handle h, void *stream) {
    if (!h) return GCE_ERR_INVALID;
    CUDA_TRY(h, cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    CUDA_TRY(h, cudaMemcpyAsync(h->h_state, h->state.p, sizeof(JobState), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(h, cudaStreamSynchronize(s));
    return state_status(h);
}

extern "C" gce_status gce_ce_topk_host(gce_handle h, const double *h_times, const double *h_mags,
                                       const int64_t *h_offsets, int32_t n_curves,
                                       const double *h_periods, int32_t n_periods,
                                       const double *h_pdots, int32_t n_pdots,
                                       const gce_config *cfg, int32_t k, float *h_topk_H,
                                       int64_t *h_topk_idx, void *stream) {
    if (!h) return GCE_ERR_INVALID;
    gce_status st = gce_check_job(h_offsets, n_curves, n_periods, n_pdots, cfg, k);
    if (st != GCE_OK) return fail(h, st, "argument check failed");
    if (k < 1) return fail(h, GCE_ERR_INVALID, "k must be >= 1");
    if (n_curves == 0) return GCE_OK;
    if (!h_times || !h_mags || !h_periods || !h_pdots || !h_topk_H || !h_topk_idx)
        return fail(h, GCE_ERR_INVALID, "NULL host array");
    CUDA_TRY(h, cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    const size_t np = (size_t)h_offsets[n_curves];
    if ((st = ensure(h, h->in_times, 8 * np)) != GCE_OK) return st;
    if ((st = ensure(h, h->in_mags, 8 * np)) != GCE_OK) return st;
    if ((st = ensure(h, h->in_periods, 8 * (size_t)n_periods)) != GCE_OK) return st;
    if ((st = ensure(h, h->in_pdots, 8 * (size_t)n_pdots)) != GCE_OK) return st;
    if ((st = ensure(h, h->out_H, 4 * (size_t)n_curves * k)) != GCE_OK) return st;
    if ((st = ensure(h, h->out_idx, 8 * (size_t)n_curves * k)) != GCE_OK) return st;
    CUDA_TRY(h, cudaMemcpyAsync(h->in_times.p, h_times, 8 * np, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaMemcpyAsync(h->in_mags.p, h_mags, 8 * np, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaMemcpyAsync(h->in_periods.p, h_periods, 8 * (size_t)n_periods,
                                cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaMemcpyAsync(h->in_pdots.p, h_pdots, 8 * (size_t)n_pdots,
                                cudaMemcpyHostToDevice, s));
    st = gce_ce_topk(h, (const double *)h->in_times.p, (const double *)h->in_mags.p, h_offsets,
                     n_curves, (const double *)h->in_periods.p, n_periods,
                     (const double *)h->in_pdots.p, n_pdots, cfg, k, (float *)h->out_H.p,
                     (int64_t *)h->out_idx.p, stream);
    if (st != GCE_OK) return st;
    CUDA_TRY(h, cudaMemcpyAsync(h_topk_H, h->out_H.p, 4 * (size_t)n_curves * k,
                                cudaMemcpyDeviceToHost, s));
    CUDA_TRY(h, cudaMemcpyAsync(h_topk_idx, h->out_idx.p, 8 * (size_t)n_curves * k,
                                cudaMemcpyDeviceToHost, s));
    return gce_stream_status(h, stream);
}

extern "C" gce_status gce_kernel_time(gce_handle h, float *ms) {
    if (!h || !ms) return GCE_ERR_INVALID;
    if (!h->timed) return fail(h, GCE_ERR_INVALID, "the last call was not made with GCE_FLAG_TIME_KERNEL");
    CUDA_TRY(h, cudaEventSynchronize(h->k1));
    CUDA_TRY(h, cudaEventElapsedTime(ms, h->k0, h->k1));
    return GCE_OK;
}

extern "C" gce_status gce_last_launches(gce_handle h, int32_t *n) {
    if (!h || !n) return GCE_ERR_INVALID;
    *n = h->launches;
    return GCE_OK;
}

// ------------------------------------------------------------------ tuning

extern "C" gce_status gce_get_tuning(gce_handle h, const gce_config *cfg, int32_t n_obs_hint,
                                     int32_t n_pdots_hint, gce_tuning *t) {
    if (!h || !cfg || !t || n_pdots_hint < 1) return GCE_ERR_INVALID;
    // a large job's shape, or a small one's where only that is cached
    bool tuned = false;
    *t = lookup_tuning(h, cfg, std::max(1, n_obs_hint), n_pdots_hint, false, &tuned);
    if (!tuned) *t = lookup_tuning(h, cfg, std::max(1, n_obs_hint), n_pdots_hint, true, &tuned);
    return GCE_OK;
}

extern "C" gce_status gce_set_tuning(gce_handle h, const gce_config *cfg, int32_t n_obs_hint,
                                     const gce_tuning *t) {
    if (!h || !cfg || !t || !tuning_ok(*t, cfg->phase_mode)) return GCE_ERR_INVALID;
    for (int pd_axis = 0; pd_axis < 2; ++pd_axis)
        for (bool small : {false, true})
            h->tune[tune_key(cfg, std::max(1, n_obs_hint), pd_axis, small)] = Tuned{*t, false};
    return GCE_OK;
}

// Candidate launch shapes of the autotuners (slot_range: the kept SPLIT32 slot
// range of every candidate).
static std::vector<gce_tuning> tune_candidates(int mode, int n_obs, int slot_range = 0) {
    const int blocks[] = {128, 256, 512};
    const int tpts[] = {1, 2, 4};
    const int chunks[] = {256, 512, 1024, 2048};
    std::vector<gce_tuning> cands;
    for (int b : blocks)
        for (int tp : tpts)
            for (int ch : chunks) {
                if (ch > 512 && ch >= 2 * n_obs) continue;  // same plan as a smaller chunk
                if (tp > most_tpt(mode)) continue;  // not built
                gce_tuning c{};
                c.block = b;
                c.tpt = tp;
                c.chunk = ch;
                c.slot_range = slot_range;
                cands.push_back(c);
            }
    return cands;
}

// Times every candidate on job j (one untimed run, then three timed ones), then
// times the three fastest again over six runs each and leaves the fastest of
// those in *best (a second look keeps close calls from being decided by one
// noisy measurement), or the job's own shape where that is faster still (it has
// forms that a gce_tuning has not: warps that share a trial set, four trials per
// thread for FP64); shapes that do not fit are skipped.  also_wide: each of
// the three is timed with the wide slot range too (the candidates keep the mid
// one, whose re-reduced warps can make it the slower on long baselines).
static gce_status time_candidates(gce_handle h, Job j, const std::vector<gce_tuning> &cands,
                                  cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1,
                                  Tuned *best, bool also_wide = false) {
    auto timed = [&](const gce_tuning *cand, int reps, float *ms) -> gce_status {
        j.force = cand;
        j.own = !cand;
        *ms = 1e30f;
        if (run_job(h, j, s) != GCE_OK) return GCE_OK;  // does not fit: stays 1e30
        cudaEventRecord(e0, s);
        for (int rep = 0; rep < reps; ++rep) run_job(h, j, s);
        cudaEventRecord(e1, s);
        if (cudaEventSynchronize(e1) != cudaSuccess)
            return fail(h, GCE_ERR_CUDA, "autotune: %s", cudaGetErrorString(cudaGetLastError()));
        cudaEventElapsedTime(ms, e0, e1);
        *ms /= (float)reps;
        return GCE_OK;
    };
    std::vector<std::pair<float, size_t>> first;
    for (size_t i = 0; i < cands.size(); ++i) {
        float ms;
        if (gce_status st = timed(&cands[i], 3, &ms)) return st;
        if (ms < 1e30f) first.emplace_back(ms, i);
    }
    if (first.empty()) return GCE_OK;
    std::sort(first.begin(), first.end());
    float best_ms = 1e30f;
    for (size_t r = 0; r < std::min<size_t>(3, first.size()); ++r) {
        for (int w = 0; w < (also_wide ? 2 : 1); ++w) {
            gce_tuning c = cands[first[r].second];
            if (w) c.slot_range = 0;
            float ms;
            if (gce_status st = timed(&c, 6, &ms)) return st;
            if (ms < best_ms) {
                best_ms = ms;
                *best = Tuned{c, false};
            }
        }
    }
    float ms;
    if (gce_status st = timed(nullptr, 6, &ms)) return st;
    if (ms < best_ms) best->own = true;
    return GCE_OK;
}

extern "C" gce_status gce_autotune_job(gce_handle h, const double *times, const double *mags,
                                       const int64_t *h_offsets, int32_t n_curves,
                                       const double *periods, int32_t n_periods,
                                       const double *pdots, int32_t n_pdots,
                                       const gce_config *cfg) {
    if (!h || !cfg) return GCE_ERR_INVALID;
    const gce_status chk = gce_check_job(h_offsets, n_curves, n_periods, n_pdots, cfg, 0);
    if (chk != GCE_OK) return fail(h, chk, "autotune: argument check failed");
    if (n_curves == 0) return GCE_OK;
    if (!times || !mags || !periods || !pdots) return fail(h, GCE_ERR_INVALID, "NULL input array");
    CUDA_TRY(h, cudaSetDevice(h->device));
    // the slice: up to 65536 periods and 8 Pdot values, each a strided subset that
    // spans the job's range, and a prefix of the curves with about 4e9 point-trials
    const int p_s = n_periods > 65536 ? (n_periods + 65535) / 65536 : 1;
    const int n_p2 = (n_periods + p_s - 1) / p_s;
    const int q_s = n_pdots > 8 ? (n_pdots + 7) / 8 : 1;
    const int n_q2 = (n_pdots + q_s - 1) / q_s;
    const long long trials = (long long)n_p2 * n_q2;
    int c2 = 0;
    long long pts = 0, nmax = 1;
    for (int c = 0; c < n_curves; ++c) nmax = std::max<long long>(nmax, h_offsets[c + 1] - h_offsets[c]);
    while (c2 < n_curves && pts * trials < 4000000000ll) {
        pts += h_offsets[c2 + 1] - h_offsets[c2];
        ++c2;
    }
    double *d_p = nullptr, *d_q = nullptr;
    float *d_H = nullptr;
    int64_t *d_I = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    gce_status result = GCE_OK;
    Tuned best{default_tuning(cfg, n_pdots), true};
    gce_config c2cfg = *cfg;
    c2cfg.flags = (c2cfg.flags | GCE_FLAG_NO_GRAPH) & ~GCE_FLAG_TIME_KERNEL;
    do {
        if (cudaMalloc(&d_p, 8 * (size_t)n_p2) || cudaMalloc(&d_q, 8 * (size_t)n_q2) ||
            cudaMalloc(&d_H, 4 * (size_t)c2) || cudaMalloc(&d_I, 8 * (size_t)c2) ||
            cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) || cudaEventCreate(&e0) ||
            cudaEventCreate(&e1)) {
            result = fail(h, GCE_ERR_NOMEM, "autotune: allocation failed");
            break;
        }
        // strided copies: one element every p_s (q_s) of the caller's arrays
        if (cudaMemcpy2DAsync(d_p, 8, periods, 8 * (size_t)p_s, 8, n_p2, cudaMemcpyDeviceToDevice, s) ||
            cudaMemcpy2DAsync(d_q, 8, pdots, 8 * (size_t)q_s, 8, n_q2, cudaMemcpyDeviceToDevice, s)) {
            result = fail(h, GCE_ERR_CUDA, "autotune: %s", cudaGetErrorString(cudaGetLastError()));
            break;
        }
        Job j{};
        j.kind = JOB_TOPK;
        j.times = times; j.mags = mags; j.h_offsets = h_offsets; j.n_curves = c2;
        j.periods = d_p; j.n_periods = n_p2; j.pdots = d_q; j.n_pdots = n_q2;
        j.cfg = &c2cfg; j.k = 1; j.topk_H = d_H; j.topk_idx = d_I;
        // SPLIT32 without a Pdot axis: candidates with the mid slot range, the
        // finalists with the wide one as well
        const bool mid = cfg->phase_mode == GCE_PHASE_SPLIT32 && n_pdots == 1;
        result = time_candidates(h, j, tune_candidates(cfg->phase_mode, (int)nmax, mid ? 1 : 0), s,
                                 e0, e1, &best, mid);
    } while (0);
    if (s) cudaStreamSynchronize(s);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (s) cudaStreamDestroy(s);
    cudaFree(d_p); cudaFree(d_q); cudaFree(d_H); cudaFree(d_I);
    if (result == GCE_OK)
        h->tune[tune_key(cfg, (int)nmax, n_pdots > 1 ? 1 : 0,
                         small_job(cfg->phase_mode, (long long)n_periods * n_pdots, n_curves, h->n_sm))] = best;
    return result;
}

extern "C" gce_status gce_autotune(gce_handle h, const gce_config *cfg, int32_t n_obs_hint,
                                   int64_t n_trials_hint) {
    if (!h || !cfg) return GCE_ERR_INVALID;
    const int n_obs = std::max(16, std::min<int>(n_obs_hint, GCE_MAX_CURVE_POINTS));
    const long long n_tr = std::max<long long>(4096, std::min<long long>(n_trials_hint, 1 << 22));
    // synthetic job of about 5e9 point-trials so that a candidate fills the GPU
    const int n_curves = (int)std::max<long long>(
        16, std::min<long long>(256, 5000000000ll / ((long long)n_obs * n_tr)));
    std::vector<int64_t> offs_v(n_curves + 1);
    for (int c = 0; c <= n_curves; ++c) offs_v[c] = (int64_t)c * n_obs;
    const int64_t *offs = offs_v.data();
    if (gce_check_job(offs, n_curves, (int32_t)n_tr, 1, cfg, 0) != GCE_OK)
        return fail(h, GCE_ERR_INVALID, "autotune: invalid config");
    CUDA_TRY(h, cudaSetDevice(h->device));
    // synthetic job: 3-year times, a square-ish signal, log-spaced periods
    const size_t np = (size_t)n_curves * n_obs;
    // the Pdot-axis pass: 8 Pdot values linear in [-1e-10, 0] over n_tr / 8 periods
    const int n_pd = 8;
    const long long n_trp = std::max<long long>(512, n_tr / n_pd);
    std::vector<double> t(np), m(np), per((size_t)n_tr), perp((size_t)n_trp), pd(n_pd);
    unsigned long long x = 0x9e3779b97f4a7c15ull;
    auto u01 = [&x]() {
        x ^= x << 13; x ^= x >> 7; x ^= x << 17;
        return (double)(x >> 11) * (1.0 / 9007199254740992.0);
    };
    for (size_t i = 0; i < np; ++i) {
        t[i] = u01() * 9.46e7;
        m[i] = 15.0 + (u01() < 0.1 ? 0.5 : 0.0) + 0.02 * u01();
    }
    for (long long p = 0; p < n_tr; ++p) per[p] = 300.0 * std::pow(288.0, (double)p / (double)(n_tr - 1));
    for (long long p = 0; p < n_trp; ++p)
        perp[p] = 300.0 * std::pow(288.0, (double)p / (double)(n_trp - 1));
    for (int q = 0; q < n_pd; ++q) pd[q] = -1e-10 * (double)q / (double)(n_pd - 1);
    double *d_t = nullptr, *d_m = nullptr, *d_p = nullptr, *d_pp = nullptr, *d_d = nullptr;
    float *d_out = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    gce_status result = GCE_OK;
    Tuned best[2] = {{default_tuning(cfg, 1), true}, {default_tuning(cfg, 8), true}};
    gce_config c2 = *cfg;
    c2.flags |= GCE_FLAG_NO_GRAPH;
    do {
        if (cudaMalloc(&d_t, 8 * np) || cudaMalloc(&d_m, 8 * np) || cudaMalloc(&d_p, 8 * n_tr) ||
            cudaMalloc(&d_pp, 8 * n_trp) || cudaMalloc(&d_d, 8 * n_pd) ||
            cudaMalloc(&d_out, 4 * (size_t)n_curves * std::max(n_tr, n_trp * n_pd)) ||
            cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) || cudaEventCreate(&e0) ||
            cudaEventCreate(&e1)) {
            result = fail(h, GCE_ERR_NOMEM, "autotune: allocation failed");
            break;
        }
        cudaMemcpy(d_t, t.data(), 8 * np, cudaMemcpyHostToDevice);
        cudaMemcpy(d_m, m.data(), 8 * np, cudaMemcpyHostToDevice);
        cudaMemcpy(d_p, per.data(), 8 * n_tr, cudaMemcpyHostToDevice);
        cudaMemcpy(d_pp, perp.data(), 8 * n_trp, cudaMemcpyHostToDevice);
        cudaMemcpy(d_d, pd.data(), 8 * n_pd, cudaMemcpyHostToDevice);
        const std::vector<gce_tuning> cands = tune_candidates(cfg->phase_mode, n_obs);
        // pass 0: one Pdot value (pd[0] = 0); pass 1: the Pdot axis
        for (int pass = 0; pass < 2 && result == GCE_OK; ++pass) {
            Job j{};
            j.kind = JOB_GRID;
            j.times = d_t; j.mags = d_m; j.h_offsets = offs; j.n_curves = n_curves;
            if (pass == 0) {
                j.periods = d_p; j.n_periods = (int)n_tr; j.pdots = d_d; j.n_pdots = 1;
            } else {
                j.periods = d_pp; j.n_periods = (int)n_trp; j.pdots = d_d; j.n_pdots = n_pd;
            }
            j.cfg = &c2; j.out = d_out;
            result = time_candidates(h, j, cands, s, e0, e1, &best[pass]);
        }
    } while (0);
    if (s) cudaStreamSynchronize(s);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (s) cudaStreamDestroy(s);
    cudaFree(d_t); cudaFree(d_m); cudaFree(d_p); cudaFree(d_pp); cudaFree(d_d); cudaFree(d_out);
    if (result == GCE_OK) {
        const int mode = cfg->phase_mode;
        h->tune[tune_key(cfg, n_obs, 0, small_job(mode, n_tr, n_curves, h->n_sm))] = best[0];
        h->tune[tune_key(cfg, n_obs, 1, small_job(mode, n_trp * n_pd, n_curves, h->n_sm))] = best[1];
    }
    return result;
}
