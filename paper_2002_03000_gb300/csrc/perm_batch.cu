// perm_batch.cu -- many independent flatPERM runs grown by one CUDA-graph launch,
// and the autotuner that picks each run's layout.
//
// A batch holds R runs (each a perm_handle with its own tables).  Their work --
// reset of the tables, growth, the tour counter clamp -- is captured once into a
// CUDA graph; replaying the graph grows every run again from empty tables.  Two
// forms:
//  * streams: one persistent growth kernel per run, on up to 64 streams, each
//    packed into the fewest CTAs that hold its walks, so that small runs fill
//    the device together instead of one after another;
//  * persistent: ONE persistent kernel on every SM grows all runs; each CTA
//    joins the run with the most tours left to start per CTA on it and moves
//    on when that run has no tours left to start (runs whose tours all started
//    are helped through their waiting copies once no run is open).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <tuple>
#include <vector>

#include <cuda_runtime.h>

#include "perm.h"
#include "perm_kernels.cuh"

struct perm_batch_s {
    int R = 0;
    std::vector<perm_handle> runs;
    std::vector<int64_t> tours;
    std::vector<cudaStream_t> streams;
    std::vector<cudaEvent_t> joins;
    cudaStream_t origin = nullptr;
    cudaEvent_t fork = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    // persistent form
    perm::RunDev *d_runs = nullptr;
    int *d_ctl = nullptr;
    bool persistent = false;
    int grid = 0, threads = 0;
    size_t smem = 0;
    long long max_ns = 0;
    std::vector<perm::RunDev> P0;   // the descriptors a replay grows (from empty tables)
    bool failed = false;            // a run of the last launch failed: it may have left tour sums behind
};

namespace {

bool all_plain(const std::vector<perm::RunDev> &P) {
    for (const perm::RunDev &p : P)
        if (!perm::plain_run(p)) return false;
    return true;
}

void batch_free(perm_batch_handle b) {
    if (!b) return;
    if (b->origin) cudaStreamSynchronize(b->origin);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (perm_handle h : b->runs) perm_destroy(h);
    for (cudaEvent_t e : b->joins) cudaEventDestroy(e);
    if (b->fork) cudaEventDestroy(b->fork);
    for (cudaStream_t s : b->streams) cudaStreamDestroy(s);
    if (b->origin) cudaStreamDestroy(b->origin);
    if (b->d_runs) cudaFree(b->d_runs);
    if (b->d_ctl) cudaFree(b->d_ctl);
    delete b;
}

}  // namespace

extern "C" {

int perm_batch_create(perm_batch_handle *out, const perm_config *cfgs, const int64_t *tours_per_seq,
                      int R, int n_streams) {
    if (!out || !cfgs || !tours_per_seq || R < 1) return PERM_EINVAL;
    *out = nullptr;
    for (int r = 0; r < R; ++r)
        if (tours_per_seq[r] < 0) return PERM_EINVAL;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PERM_EDEVICE;
    if (perm::set_smem_limits() != cudaSuccess) return PERM_EDEVICE;
    perm_batch_handle b = new (std::nothrow) perm_batch_s();
    if (!b) return PERM_ENOMEM;
    b->R = R;
    b->tours.assign(tours_per_seq, tours_per_seq + R);

    int S = n_streams > 0 ? n_streams : std::min(R, 64);
    S = std::min(S, R);
    int rc = PERM_OK;
    if (cudaStreamCreateWithFlags(&b->origin, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess)
        rc = PERM_EDEVICE;
    for (int s = 0; rc == PERM_OK && s < S; ++s) {
        cudaStream_t st;
        cudaEvent_t ev;
        if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) { rc = PERM_EDEVICE; break; }
        b->streams.push_back(st);
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) { rc = PERM_EDEVICE; break; }
        b->joins.push_back(ev);
    }
    for (int r = 0; rc == PERM_OK && r < R; ++r) {
        perm_config c = cfgs[r];
        // pack each run's walks into as few CTAs as shared memory allows, so that
        // the concurrent runs share the SMs
        if (c.max_ctas == 0) c.max_ctas = -1;
        perm_handle h = nullptr;
        rc = perm_create_ex(&h, &c);
        if (rc != PERM_OK) break;
        b->runs.push_back(h);
        rc = perm_set_stream(h, (void *)b->streams[r % S]);
    }
    // capture: fork to the run streams, reset + grow each run, join
    if (rc == PERM_OK && cudaStreamBeginCapture(b->origin, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        rc = PERM_EDEVICE;
    if (rc == PERM_OK) {
        cudaError_t e = cudaEventRecord(b->fork, b->origin);
        for (int s = 0; e == cudaSuccess && s < S; ++s) e = cudaStreamWaitEvent(b->streams[s], b->fork, 0);
        if (e != cudaSuccess) rc = PERM_EDEVICE;
        for (int r = 0; rc == PERM_OK && r < R; ++r) {
            rc = perm_reset(b->runs[r]);
            if (rc == PERM_OK) rc = perm_run(b->runs[r], b->tours[r]);
        }
        for (int s = 0; rc == PERM_OK && s < S; ++s) {
            if (cudaEventRecord(b->joins[s], b->streams[s]) != cudaSuccess ||
                cudaStreamWaitEvent(b->origin, b->joins[s], 0) != cudaSuccess)
                rc = PERM_EDEVICE;
        }
        cudaGraph_t g = nullptr;
        const cudaError_t ec = cudaStreamEndCapture(b->origin, &g);
        if (rc == PERM_OK && ec != cudaSuccess) rc = PERM_EDEVICE;
        b->graph = g;
        if (rc == PERM_OK && cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess) rc = PERM_EDEVICE;
    }
    if (rc != PERM_OK) {
        batch_free(b);
        return rc;
    }
    *out = b;
    return PERM_OK;
}

int perm_batch_create_persistent(perm_batch_handle *out, const perm_config *cfgs,
                                 const int64_t *tours_per_seq, int R) {
    if (!out || !cfgs || !tours_per_seq || R < 1) return PERM_EINVAL;
    *out = nullptr;
    for (int r = 0; r < R; ++r) {
        if (tours_per_seq[r] < 0) return PERM_EINVAL;
        if (cfgs[r].alg != PERM_ALG2 || cfgs[r].threshold != PERM_THRESH_SNAPSHOT) return PERM_EUNSUPPORTED;
    }
    size_t budget = 0;
    if (perm::set_smem_limits() != cudaSuccess || perm::batch_smem_budget(&budget) != cudaSuccess)
        return PERM_EDEVICE;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PERM_EDEVICE;
    perm_batch_handle b = new (std::nothrow) perm_batch_s();
    if (!b) return PERM_ENOMEM;
    b->R = R;
    b->tours.assign(tours_per_seq, tours_per_seq + R);
    int rc = PERM_OK;
    if (cudaStreamCreateWithFlags(&b->origin, cudaStreamNonBlocking) != cudaSuccess) rc = PERM_EDEVICE;
    // one CTA per SM: every run is laid out so that any CTA of the grid may join it
    const int grid = sms;
    std::vector<perm::RunDev> P(R);
    size_t smem = 0;
    int warps = 1;
    double max_s = 0.0;
    for (int r = 0; rc == PERM_OK && r < R; ++r) {
        perm_handle h = nullptr;
        rc = perm::member_create(&h, &cfgs[r], grid, budget);
        if (rc != PERM_OK) break;
        b->runs.push_back(h);
        rc = perm_set_stream(h, (void *)b->origin);
        size_t sm = 0;
        int w = 0;
        if (rc == PERM_OK) rc = perm::member_params(h, b->tours[r], r, &P[r], &sm, &w);
        smem = std::max(smem, sm);
        warps = std::max(warps, w);
        max_s = std::max(max_s, (double)P[r].max_ns * 1e-9);
    }
    const int threads = 32 * (warps + 1);
    b->persistent = true;
    b->grid = grid;
    b->threads = threads;
    b->smem = smem;
    b->max_ns = (long long)(max_s * 1e9);
    // every CTA of the grid must be resident at once: walks wait (boundedly) on
    // copies that other CTAs' walks hand over
    int resident = 0;
    if (rc == PERM_OK && (perm::batch_grid(threads, smem, &resident) != cudaSuccess || resident < grid))
        rc = PERM_EUNSUPPORTED;
    if (rc == PERM_OK && cudaMalloc((void **)&b->d_runs, sizeof(perm::RunDev) * R) != cudaSuccess) rc = PERM_ENOMEM;
    if (rc == PERM_OK && cudaMalloc((void **)&b->d_ctl, sizeof(int) * (3 * (size_t)R + 1 + (size_t)grid)) != cudaSuccess) rc = PERM_ENOMEM;
    if (rc == PERM_OK &&
        cudaMemcpy(b->d_runs, P.data(), sizeof(perm::RunDev) * R, cudaMemcpyHostToDevice) != cudaSuccess)
        rc = PERM_EDEVICE;
    perm::BatchDev B;
    B.runs = b->d_runs;
    B.R = R;
    B.active = b->d_ctl;
    B.granted = b->d_ctl + R;
    B.closed = b->d_ctl + 2 * R;
    B.runs_open = b->d_ctl + 3 * R;
    B.first = b->d_ctl + 3 * R + 1;
    B.ctas = grid;
    B.max_ns = (long long)(max_s * 1e9);
    B.plain = all_plain(P);
    // capture: reset every run, the batch kernel, clamp each run's tour counter
    if (rc == PERM_OK && cudaStreamBeginCapture(b->origin, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        rc = PERM_EDEVICE;
    if (rc == PERM_OK) {
        for (int r = 0; rc == PERM_OK && r < R; ++r) rc = perm::member_reset(b->runs[r]);
        if (rc == PERM_OK && perm::launch_batch(B, grid, threads, smem, b->origin) != cudaSuccess) rc = PERM_EDEVICE;
        for (int r = 0; rc == PERM_OK && r < R; ++r)
            if (perm::launch_finalize(P[r], b->origin) != cudaSuccess) rc = PERM_EDEVICE;
        cudaGraph_t g = nullptr;
        const cudaError_t ec = cudaStreamEndCapture(b->origin, &g);
        if (rc == PERM_OK && ec != cudaSuccess) rc = PERM_EDEVICE;
        b->graph = g;
        if (rc == PERM_OK && cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess) rc = PERM_EDEVICE;
    }
    // the resets above cleared the host-side tour counts; set them again
    for (int r = 0; rc == PERM_OK && r < R; ++r) rc = perm::member_params(b->runs[r], b->tours[r], r, &P[r], nullptr, nullptr);
    if (rc == PERM_OK) b->P0 = P;
    if (rc != PERM_OK) {
        batch_free(b);
        return rc;
    }
    *out = b;
    return PERM_OK;
}

int perm_batch_run(perm_batch_handle b) {
    if (!b || !b->exec) return PERM_EINVAL;
    if (b->failed) {
        for (perm_handle h : b->runs) {
            const int rc = perm::member_clear_sums(h);
            if (rc != PERM_OK) return rc;
        }
        for (cudaStream_t s : b->streams)
            if (cudaStreamSynchronize(s) != cudaSuccess) return PERM_EDEVICE;
        b->failed = false;
    }
    // a replay grows every run from empty tables by its creation-time tours, also
    // after perm_batch_continue moved the descriptors and tour counts on
    if (b->persistent && cudaMemcpyAsync(b->d_runs, b->P0.data(), sizeof(perm::RunDev) * b->R,
                                         cudaMemcpyHostToDevice, b->origin) != cudaSuccess)
        return PERM_EDEVICE;
    if (cudaGraphLaunch(b->exec, b->origin) != cudaSuccess) return PERM_EDEVICE;
    if (cudaStreamSynchronize(b->origin) != cudaSuccess) return PERM_EDEVICE;
    for (int r = 0; r < b->R; ++r) {
        perm::RunDev P;
        const int rc = perm::member_params(b->runs[r], b->tours[r], r, &P, nullptr, nullptr);
        if (rc != PERM_OK) return rc;
    }
    for (perm_handle h : b->runs) {
        perm_stats_t st;
        const int rc = perm_stats(h, &st);
        if (rc != PERM_OK || st.status != PERM_OK) {
            b->failed = true;
            return rc != PERM_OK ? rc : st.status;
        }
    }
    return PERM_OK;
}

int perm_batch_continue(perm_batch_handle b, const int64_t *extra_tours_per_seq) {
    if (!b || !extra_tours_per_seq) return PERM_EINVAL;
    for (int r = 0; r < b->R; ++r)
        if (extra_tours_per_seq[r] < 0) return PERM_EINVAL;
    if (!b->persistent) {
        // each run's own kernel on its stream, cumulative on its tables
        for (int r = 0; r < b->R; ++r) {
            if (extra_tours_per_seq[r] == 0) continue;
            const int rc = perm_run(b->runs[r], extra_tours_per_seq[r]);
            if (rc != PERM_OK) return rc;
        }
        for (cudaStream_t s : b->streams)
            if (cudaStreamSynchronize(s) != cudaSuccess) return PERM_EDEVICE;
    } else {
        // one persistent launch over the runs with tours to grow; the others keep
        // their tables (every CTA skips a run with no tours left to start)
        std::vector<perm::RunDev> P(b->R);
        for (int r = 0; r < b->R; ++r) {
            const int rc = perm::member_extend(b->runs[r], extra_tours_per_seq[r], r, &P[r]);
            if (rc != PERM_OK) return rc;
        }
        if (cudaMemcpyAsync(b->d_runs, P.data(), sizeof(perm::RunDev) * b->R, cudaMemcpyHostToDevice,
                            b->origin) != cudaSuccess)
            return PERM_EDEVICE;
        perm::BatchDev B;
        B.runs = b->d_runs;
        B.R = b->R;
        B.active = b->d_ctl;
        B.granted = b->d_ctl + b->R;
        B.closed = b->d_ctl + 2 * b->R;
        B.runs_open = b->d_ctl + 3 * b->R;
        B.first = b->d_ctl + 3 * b->R + 1;
        B.ctas = b->grid;
        B.max_ns = b->max_ns;
        B.plain = all_plain(P);
        if (perm::launch_batch(B, b->grid, b->threads, b->smem, b->origin) != cudaSuccess) return PERM_EDEVICE;
        for (int r = 0; r < b->R; ++r)
            if (perm::launch_finalize(P[r], b->origin) != cudaSuccess) return PERM_EDEVICE;
        if (cudaStreamSynchronize(b->origin) != cudaSuccess) return PERM_EDEVICE;
    }
    for (perm_handle h : b->runs) {
        perm_stats_t st;
        const int rc = perm_stats(h, &st);
        if (rc != PERM_OK || st.status != PERM_OK) {
            b->failed = true;
            return rc != PERM_OK ? rc : st.status;
        }
    }
    return PERM_OK;
}

int perm_batch_size(perm_batch_handle b) { return b ? b->R : PERM_EINVAL; }

int perm_batch_estimates(perm_batch_handle b, int r, double *log_cn, double *S_n, double *relvar_n) {
    if (!b || r < 0 || r >= b->R) return PERM_EINVAL;
    return perm_estimates(b->runs[r], log_cn, S_n, relvar_n);
}

int perm_batch_stats(perm_batch_handle b, int r, perm_stats_t *out) {
    if (!b || r < 0 || r >= b->R) return PERM_EINVAL;
    return perm_stats(b->runs[r], out);
}

void perm_batch_destroy(perm_batch_handle b) { batch_free(b); }

// ---------------------------------------------------------------------------
// Autotuner: short calibration runs over walks per warp, hash size and the
// shared-memory stack ring ("spill tile").  Choices that come to a layout already timed
// are left out (a warp holds at most 8 walks, 4 on the cubic lattice, and hash_scale 0
// doubles the hash where it fits: about half of the choices repeat another).  Each trial times a complete run of
// probe_tours tours per sequence from empty tables (twice, the faster counts),
// so the trials compare equal work, start-up included.  The default layout is
// timed first and stays unless a choice beats it by 3% and then again on runs
// of four times the tours.  The choice is written back and cached per (d,
// n_max, n_seq, max_ctas, alg, threshold).
// ---------------------------------------------------------------------------
namespace {
struct TuneChoice { int lanes, hash_scale, ring; };
std::mutex g_tune_mutex;
std::map<std::tuple<int, int, int, int, int, int>, TuneChoice> g_tune_cache;
}  // namespace

int perm_autotune(perm_config *cfg, int64_t probe_tours) {
    if (!cfg || probe_tours < 1) return PERM_EINVAL;
    const auto key = std::make_tuple(cfg->d, cfg->n_max, cfg->n_seq, cfg->max_ctas, cfg->alg, cfg->threshold);
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            cfg->lanes_per_warp = it->second.lanes;
            cfg->hash_scale = it->second.hash_scale;
            cfg->stack_ring = it->second.ring;
            return PERM_OK;
        }
    }
    const int lanes_c[] = {0, 2, 4, 8};
    const int hash_c[] = {0, 1};
    const int ring_c[] = {16, 64};
    // the layouts timed so far: warps, walks a warp, CTAs, hash slots, ring
    std::set<std::tuple<int, int, int, int, int>> timed;
    // a complete run of `tours` from empty tables with the layout of `t`, `reps`
    // times (start-up included: it is part of every run); the fastest counts.  once: not if
    // the layout has been timed
    auto time_layout = [&](const TuneChoice &t, int64_t tours, int reps, bool once) {
        perm_config c = *cfg;
        c.lanes_per_warp = t.lanes;
        c.hash_scale = t.hash_scale;
        c.stack_ring = t.ring;
        perm_handle h = nullptr;
        if (perm_create_ex(&h, &c) != PERM_OK) return -1.0;
        double sec = -1.0;
        perm_stats_t st;
        int rc = perm_stats(h, &st);
        if (rc == PERM_OK && once &&
            !timed.insert(std::make_tuple(st.warps_per_cta, st.lanes_per_warp, st.ctas, st.hash_slots, t.ring)).second) {
            perm_destroy(h);
            return -1.0;
        }
        for (int rep = 0; rep < reps && rc == PERM_OK; ++rep) {
            rc = perm_reset(h);
            const auto t0 = std::chrono::steady_clock::now();
            if (rc == PERM_OK) rc = perm_run_sync(h, tours);
            const auto t1 = std::chrono::steady_clock::now();
            const double s1 = std::chrono::duration<double>(t1 - t0).count();
            if (rc == PERM_OK && (sec < 0.0 || s1 < sec)) sec = s1;
        }
        perm_destroy(h);
        return rc == PERM_OK ? sec : -1.0;
    };
    const TuneChoice dflt{0, 0, 16};
    const double dflt_s = time_layout(dflt, probe_tours, 2, true);
    double best_s = dflt_s;
    TuneChoice best = dflt;
    for (int ring : ring_c) {
        for (int hs : hash_c) {
            for (int lw : lanes_c) {
                const TuneChoice t{lw, hs, ring};
                if (lw == 0 && hs == 0 && ring == 16) continue;
                const double sec = time_layout(t, probe_tours, 2, true);
                // a choice other than the default has to beat it by 3% (the spread
                // of repeated complete runs), else the default stays
                if (sec >= 0.0 && (best_s < 0.0 || sec < best_s * (best.lanes == 0 && best.hash_scale == 0 &&
                                                                     best.ring == 16 ? 0.97 : 1.0))) {
                    best_s = sec;
                    best = t;
                }
            }
        }
    }
    // the pick is validated against the default on runs four times as long,
    // alternating the two three times (the node count of a complete run varies by
    // 10-30 % from run to run), and kept only if its fastest run beats the
    // default's by 3 %
    if (best_s >= 0.0 && !(best.lanes == 0 && best.hash_scale == 0 && best.ring == 16)) {
        double b4 = -1.0, d4 = -1.0;
        for (int k = 0; k < 3; ++k) {
            const double b = time_layout(best, 4 * probe_tours, 1, false),
                         d = time_layout(dflt, 4 * probe_tours, 1, false);
            if (b >= 0.0 && (b4 < 0.0 || b < b4)) b4 = b;
            if (d >= 0.0 && (d4 < 0.0 || d < d4)) d4 = d;
        }
        if (b4 < 0.0 || (d4 >= 0.0 && b4 >= d4 * 0.97)) { best = dflt; best_s = dflt_s; }
    }
    if (best_s < 0.0) return PERM_EUNSUPPORTED;
    cfg->lanes_per_warp = best.lanes;
    cfg->hash_scale = best.hash_scale;
    cfg->stack_ring = best.ring;
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    g_tune_cache[key] = best;
    return PERM_OK;
}

}  // extern "C"
