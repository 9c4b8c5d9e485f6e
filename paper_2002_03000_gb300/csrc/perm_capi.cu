// perm_capi.cu -- C ABI of libperm.so (declared in include/perm.h).
//
// Host side of the interacting flatPERM run: argument checks, the layout of
// walks on the device (slots per warp, warps per CTA, CTAs), device memory,
// launches, and the estimates of Sec. 1, eq. (4) (Alg. 1: eq. (7)) computed
// from the tables the kernels fill.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "perm.h"
#include "perm_kernels.cuh"

using perm::RunDev;

struct perm_run_s {
    perm_config cfg;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0, num_sms = 0;
    bool key64 = false;
    int thresh = perm::kSnapshot;
    int log2h = 0, slots = 0, ctas = 0, worker_warps = 0, lanes = 0, stack_cache = 16;
    size_t smem = 0;
    int arena_mode = 0;            // perm::ArenaMode
    long long arena_cta_bytes = 0;
    unsigned char *arena = nullptr;
    int ntab = 1;
    int xrows = 0;                 // tour-sum rows: one per walk, two with shared copies
    int tour_slots = 0;            // walks that start tours; the other slots are helpers
    // what a reset zeroes, in one buffer: the counters (a 256-byte line each: the kernels' walks
    // meet on several of them), the tables and the rings' stamps
    unsigned char *block = nullptr;
    size_t zero_bytes = 0;
    // device buffers (those of the block point into it)
    int parts = 1;                 // copies of W_n and Q_n that the CTAs add to
    double *Wp = nullptr, *Qp = nullptr;
    double *Wn = nullptr, *Qn = nullptr, *X = nullptr, *gstk_w = nullptr, *Rn = nullptr;
    unsigned long long *Sn = nullptr, *tickets = nullptr, *seq_M = nullptr;
    unsigned long long *steps = nullptr, *max_stack = nullptr, *copies = nullptr, *refreshes = nullptr, *trace_count = nullptr;
    unsigned long long *iterations = nullptr, *finished = nullptr, *exact_steps = nullptr;
    long long *admit = nullptr;    // admission of new tours (two counts)
    uint32_t *gstk_meta = nullptr;
    int *status = nullptr;
    // shared copies
    bool share = false;
    int share_cap = 0;
    int dq_log2cap = 0, dq_cell_bytes = 0;
    unsigned char *dq_cells = nullptr;
    unsigned long long *dq_head = nullptr, *dq_tail = nullptr;
    unsigned int *dq_ready = nullptr, *dq_free = nullptr, *outst = nullptr, *tmaxn = nullptr;
    int *hungry = nullptr, *queued = nullptr, *dq_used = nullptr;
    double2 *cut = nullptr;        // original PERM's cut-offs (nullptr: flatPERM)
    int cut_copies = 1;
    double cut_q = 1.0;
    perm_trace_record *trace = nullptr;
    int32_t *trace_coords = nullptr;
    int trace_cap = 0;
    long long trace_every = 0, trace_tour_every = 1;
    // host bookkeeping
    long long tour_limit = 0;      // Alg. 2 tickets handed out so far (cumulative)
    long long seq_target = 0;      // Alg. 1 tours per sequence (cumulative)
    long long device_bytes = 0;
    bool own_limit = false;        // the caller gave an admission limit (ramp_c0 or ramp_gamma)
    int last_status = PERM_OK;
    bool unread = false;           // launches queued since their status was last read
};

namespace {

// The counters of a handle's block, a line each.
constexpr size_t kLine = 256;
// Few lengths and many walks: the walks' additions to W_n and Q_n meet on a few lines.  With
// tables of a kilobyte or two in one slice of L2 the steady rate was 1.7e9 steps/s at
// n = 16, 2.4e9 at 64, 2.9e9 at 128 and 5.0e9 at 256; with four copies 3.6, 4.9, 5.2 and 5.3e9
// (square, 8192 sequences; 8 or 16 copies the same; at n = 512 they gain nothing).
constexpr int kParts = 4, kPartsLengths = 400, kPartsWalks = 512;
constexpr size_t kPartStride = 544;      // doubles: 4352 bytes apart
constexpr size_t kOneCopy = 1 << 20;   // tables up to this size come back in one copy
enum Counter { kTickets, kSteps, kMaxStack, kCopies, kRefreshes, kIterations, kFinished, kExact, kStatus, kAdmit, kHead, kTail,
               kHungry, kQueued, kUsed, kCounters };

int to_code(cudaError_t e) {
    if (e == cudaSuccess) return PERM_OK;
    if (e == cudaErrorMemoryAllocation) return PERM_ENOMEM;
    return PERM_EDEVICE;
}

template <typename T>
int dalloc(perm_handle h, T **p, size_t count) {
    const size_t bytes = count * sizeof(T);
    if (bytes == 0) { *p = nullptr; return PERM_OK; }
    cudaError_t e = cudaMalloc((void **)p, bytes);
    if (e != cudaSuccess) { *p = nullptr; return to_code(e); }
    h->device_bytes += (long long)bytes;
    e = cudaMemsetAsync(*p, 0, bytes, h->stream);
    return to_code(e);
}

void free_all(perm_handle h) {
    void *ptrs[] = {h->block, h->X, h->gstk_w, h->gstk_meta, h->trace_count, h->trace, h->trace_coords, h->dq_cells,
                    h->outst, h->cut, h->arena};
    for (void *p : ptrs) if (p) cudaFree(p);
}

// Parts of one tour that may grow on other walks at once (shared copies), and the
// larger bound used once no tour of the run has finished for kStallNs.  GB300, ms per
// complete run at 5 / 2 / 0.7 / 0.3 ms: square n = 512, 4096 x 256 215 / 210 / 208 / 208;
// cubic n = 512, 8192 x 128 173 / 168 / 166 / 165; square n = 256, 1000 x 64 32 / 28 / 26 / 25;
// cubic n = 945, 2142 x 4 86 / 38 / 33 / 33; square n = 1725, 422 x 4 250 / 205 / 184 / 470.
constexpr int kAutoWalks = 32;          // walks per CTA of the automatic layout, in the arena
constexpr int kBatchWalks = 48;         // and about as many of a persistent batch's members: each has
                                        // scratch for a grid of such CTAs (24 runs of n = 64..256:
                                        // 0.66, 0.76 and 0.99 GB, 15.1, 15.4 and 15.6 ms at 40, 48
                                        // and 88; whole warps of them, 10 x 5 where they fit)
constexpr int kDefaultShareCap = 4;
constexpr int kRampC0 = 2;              // the default admission limit
constexpr double kRampGamma = 0.25;
constexpr int kBoostShareCap = 1024;
constexpr long long kStallNs = 700000;

// S_n is kept on the device as its differences along n, row by row of L entries.
// (out may be the differences' own memory.)
template <typename T>
void counts_from_differences(const void *differences, size_t cnt, size_t L, T *out) {
    const unsigned char *s = static_cast<const unsigned char *>(differences);
    for (size_t row = 0; row < cnt; row += L) {
        unsigned long long sum = 0ull, d;
        for (size_t i = row; i < row + L; ++i) {
            std::memcpy(&d, s + 8 * i, 8);
            out[i] = (T)(sum += d);
        }
    }
}
void differences_from_counts(unsigned char *s, size_t cnt, size_t L) {
    for (size_t row = 0; row < cnt; row += L) {
        unsigned long long before = 0ull, c;
        for (size_t i = row; i < row + L; ++i) {
            std::memcpy(&c, s + 8 * i, 8);
            const unsigned long long d = c - before;
            std::memcpy(s + 8 * i, &d, 8);
            before = c;
        }
    }
}

// A length's cut-offs as the kernel compares them, by their bit patterns: no NaN (which no
// weight is above or below) and no -0.0.
double2 clean_cutoffs(double hi, double lo) {
    if (std::isnan(hi)) hi = INFINITY;
    if (std::isnan(lo)) lo = 0.0;
    return make_double2(hi == 0.0 ? 0.0 : hi, lo == 0.0 ? 0.0 : lo);
}

int scale_exp_host(int d, int n) { return d == 2 ? (11 * n) >> 3 : (9 * n) >> 2; }

int max_n_for(int d, bool key64) {
    if (d == 2) return 32766;
    return key64 ? (1 << 20) - 2 : 512;
}

}  // namespace

extern "C" {

void perm_config_init(perm_config *cfg, int d, int n_max, int n_seq, uint64_t seed) {
    if (!cfg) return;
    std::memset(cfg, 0, sizeof(*cfg));
    cfg->d = d;
    cfg->n_max = n_max;
    cfg->n_seq = n_seq;
    cfg->seed = seed;
    cfg->run_id = 0u;
    cfg->alg = PERM_ALG2;
    cfg->threshold = PERM_THRESH_SNAPSHOT;
    cfg->slots = 0;
    cfg->lanes_per_warp = 0;
    cfg->refresh_ns = 0;
    cfg->max_seconds = 0.0;
    cfg->ramp_c0 = 0;
    cfg->ramp_gamma = 0.0;
    cfg->max_ctas = 0;
    cfg->hash_scale = 0;
    cfg->share_copies = 0;
    cfg->stack_ring = 0;
    cfg->observables = 0;
    cfg->walk_memory = 0;
    cfg->helper_walks = 0;
}

const char *perm_strerror(int code) {
    switch (code) {
        case PERM_OK: return "ok";
        case PERM_EINVAL: return "invalid argument";
        case PERM_ENOMEM: return "out of memory";
        case PERM_EOVERFLOW: return "stack or hash bound exceeded in a kernel";
        case PERM_EDEVICE: return "CUDA device error";
        case PERM_ETIMEOUT: return "bounded device wait ran out";
        case PERM_EUNSUPPORTED: return "configuration not supported";
        case PERM_ESCRATCH: return "requested walks need more scratch than the static buffer holds";
        default: return "unknown error";
    }
}

}  // extern "C"

namespace {

// A layout forced by a batch launch: `ctas` CTAs (the batch grid) within
// smem_budget bytes of shared memory each.
struct ForcedLayout {
    int ctas;
    size_t smem_budget;
};

int create_impl(perm_handle *out, const perm_config *cfg, const ForcedLayout *force) {
    if (!out || !cfg) return PERM_EINVAL;
    *out = nullptr;
    const int d = cfg->d, n_max = cfg->n_max, n_seq = cfg->n_seq;
    if ((d != 2 && d != 3) || n_max < 1 || n_seq < 1) return PERM_EINVAL;
    if (cfg->alg != PERM_ALG1 && cfg->alg != PERM_ALG2) return PERM_EINVAL;
    if (cfg->threshold != PERM_THRESH_SNAPSHOT && cfg->threshold != PERM_THRESH_FRESH) return PERM_EINVAL;
    if (cfg->slots < 0 || cfg->refresh_ns < 0 || !(cfg->max_seconds >= 0.0)) return PERM_EINVAL;
    if (!(cfg->ramp_gamma >= 0.0) || cfg->ramp_gamma > 1e6) return PERM_EINVAL;
    if (cfg->max_ctas < -1 || cfg->hash_scale < 0 || cfg->hash_scale > 2) return PERM_EINVAL;
    if (cfg->share_copies < -1 || cfg->share_copies > 1024) return PERM_EINVAL;
    if (cfg->observables != 0 && cfg->observables != 1) return PERM_EINVAL;
    if (cfg->walk_memory < 0 || cfg->walk_memory > 2) return PERM_EINVAL;
    // helper walks take waiting copies only: they need shared copies
    if (cfg->helper_walks < -1 || cfg->helper_walks > (1 << 20)) return PERM_EINVAL;
    if (cfg->helper_walks > 0 && !(cfg->share_copies >= 0 && cfg->alg == PERM_ALG2 &&
                                   cfg->threshold == PERM_THRESH_SNAPSHOT))
        return PERM_EINVAL;
    if (cfg->stack_ring != 0 && cfg->stack_ring != 16 && cfg->stack_ring != 32 &&
        cfg->stack_ring != 64 && cfg->stack_ring != 128) return PERM_EINVAL;
    const int lpw = cfg->lanes_per_warp;
    if (lpw != 0 && (lpw < 1 || lpw > 32)) return PERM_EINVAL;
    const bool key64 = (d == 3 && n_max > 512);
    if (n_max > max_n_for(d, key64)) return PERM_EUNSUPPORTED;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PERM_EDEVICE;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return PERM_EDEVICE;

    perm_handle h = new (std::nothrow) perm_run_s();
    if (!h) return PERM_ENOMEM;
    h->cfg = *cfg;
    if (cfg->stack_ring) h->stack_cache = cfg->stack_ring;
    if (h->cfg.refresh_ns == 0) h->cfg.refresh_ns = 8000;
    if (h->cfg.refresh_ns > 1000000) h->cfg.refresh_ns = 1000000;
    if (h->cfg.max_seconds == 0.0) h->cfg.max_seconds = 600.0;
    h->own_limit = cfg->ramp_c0 != 0 || cfg->ramp_gamma != 0.0;
    if (h->cfg.ramp_c0 == 0) h->cfg.ramp_c0 = kRampC0;
    if (h->cfg.ramp_gamma == 0.0) h->cfg.ramp_gamma = kRampGamma;
    h->device = dev;
    h->num_sms = prop.multiProcessorCount;
    if (cfg->max_ctas > 0 && cfg->max_ctas < h->num_sms) h->num_sms = cfg->max_ctas;
    h->key64 = key64;
    // Algorithm 1 reads its private rows directly (no snapshot needed)
    h->thresh = (cfg->alg == PERM_ALG1) ? perm::kFresh
              : (cfg->threshold == PERM_THRESH_FRESH ? perm::kFresh : perm::kSnapshot);
    int log2h = 4;
    while ((1 << log2h) < 2 * n_max) ++log2h;
    log2h += cfg->hash_scale;
    if (log2h > 16) log2h = 16;                 // site slots are 16-bit
    h->log2h = log2h;
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete h;
        return PERM_EDEVICE;
    }
    h->own_stream = true;

    // layout: walks per warp (lanes), walk warps per CTA, CTAs.  A group of lanes grows
    // one walk; the walks of an SM are spread over up to 11 warps (8 with 64-bit
    // keys), so that every scheduler has several walks' dependent chains to issue from.
    const bool snap = (h->thresh == perm::kSnapshot);
    const size_t budget = force ? force->smem_budget : prop.sharedMemPerBlockOptin;
    const int max_l = perm::walks_per_warp_max(d), max_w = perm::walk_warps_max(key64);
    size_t walk_b = perm::walk_bytes(key64, n_max, log2h, h->stack_cache);
    // where the walks' hashes, site lists and stack rings live: shared memory, or a
    // global arena when asked for or when not one walk per CTA fits beside the head
    const size_t head_b = perm::cta_head_bytes(n_max, snap);
    auto arena_for = [&](int wm) {
        if (wm != 2) return (int)perm::kArenaNone;
        return head_b <= budget ? (int)perm::kArenaWalks : (int)perm::kArenaAll;
    };
    int arena_mode = arena_for(force ? 1 : cfg->walk_memory);
    if (!force && cfg->walk_memory == 0 &&
        head_b + walk_b > budget)
        arena_mode = arena_for(2);
    auto smem_for = [&](int walks) {
        if (arena_mode == perm::kArenaWalks) return head_b;
        if (arena_mode == perm::kArenaAll) return (size_t)0;
        return head_b + walk_b * (size_t)walks;
    };
    int warps = 0, lanes = 0;
    // walks of a CTA over its warps: over as many of them as there are walks
    auto spread = [&](int t) {
        lanes = (t + max_w - 1) / max_w;
        warps = (t + lanes - 1) / lanes;
    };
    // automatic: of the layouts that fill the shared memory, the one whose walks times
    // warps are the most.  A warp's iteration takes hardly longer for more walks, and an
    // SM's iterations take hardly longer for more warps.  GB300, 16384 sequences, ms:
    // n = 400, 8 tours continued, 484 (11 warps x 4 walks) 12.0, 363 (11 x 3) 13.3, 320
    // (8 x 5) 13.5, 294 (7 x 6) 14.2, 252 (6 x 7) 15.1, 200 (5 x 8) 16.5; n = 512, 400
    // (10 x 4) 18.5, 363 18.6, 294 20.6, 242 (11 x 2) 20.8, 200 24.5; n = 128, 32 tours,
    // where all fit, 11 x 4 / 5 / 6 / 7 / 8 11.1 / 9.7 / 8.8 / 8.2 / 7.8, from empty tables
    // 17.3 / 16.5 / 15.8 / 15.6 / 15.4 (the walks go before twice the hash: n = 256, 16
    // tours, 44 with it 12.4 and 23.0, 80 without 11.3 and 23.5)
    int auto_walks = kAutoWalks, full_l = 0;
    if (arena_mode == perm::kArenaNone) {
        const long long room = (long long)((budget - head_b) / walk_b);
        long long best = 0;
        for (int l = 1; l <= max_l; ++l) {
            const long long w = std::min<long long>(max_w, room / l);
            if (w * w * l > best) { best = w * w * l; full_l = l; auto_walks = (int)(w * l); }
        }
    }
    // a CTA's layout for t walks, or for the most below that fit; the walks that it holds (0:
    // none fits).  most: what the largest CTA is asked for
    const long long most = lpw ? max_w * std::min(lpw, max_l) : auto_walks;
    auto lay_out = [&](long long t) {
        for (warps = 0; t >= 1 && !warps; --t) {
            if (lpw) {
                lanes = (int)std::min<long long>(t, std::min(lpw, max_l));
                warps = (int)((t + lanes - 1) / lanes);
            } else if (t == auto_walks && full_l) {
                lanes = full_l;
                warps = auto_walks / full_l;
            } else {
                spread((int)t);
            }
            if (smem_for(warps * lanes) > budget) warps = 0;
        }
        return warps * lanes;
    };
    if (!force && cfg->max_ctas == -1) {
        // dense packing: the fewest CTAs that hold one walk per sequence, so that runs
        // sharing the device take few SMs each (24 runs of n = 64..256 on streams: 33.8 ms at 4
        // full warps a CTA, 25.4 at 8, 22.6 at 11).  A CTA holds what its layout does, which may be
        // fewer walks than the shared memory
        const long long per_cta = lay_out(most);
        if (per_cta > 0) {
            const long long need = ((long long)n_seq + per_cta - 1) / per_cta;
            h->num_sms = (int)std::max(1LL, std::min((long long)h->num_sms, need));
        }
    }
    long long tslots = cfg->slots ? cfg->slots : (long long)n_seq;   // walks that grow tours
    if (tslots > n_seq) tslots = n_seq;
    // and helper walks: as asked (none by default), or (-1) the walks the automatic
    // layout has room for beyond the tour walks, up to 32 per SM, when shared copies
    // are on
    const bool can_help = cfg->share_copies >= 0 && cfg->alg == PERM_ALG2 &&
                          cfg->threshold == PERM_THRESH_SNAPSHOT && !force;
    long long helpers = cfg->helper_walks;
    if (helpers < 0) helpers = can_help && !lpw ? std::max(0LL, (long long)h->num_sms * 32 - tslots) : 0;
    long long slots = tslots + helpers;
    if (force) {
        // every CTA of the batch grid may join this run: the most walks up to the automatic
        // layout's bound that fit the shared memory
        for (int t = std::min(auto_walks, kBatchWalks); t >= 1 && !warps; --t) {
            spread(t);
            if (smem_for(warps * lanes) > budget) warps = 0;
        }
        slots = (long long)force->ctas * warps * lanes;
        if (!warps || slots > (1LL << 30)) { cudaStreamDestroy(h->stream); delete h; return PERM_EUNSUPPORTED; }
        h->num_sms = force->ctas;
    }
    // the walks that the SMs share, or the most of them that fit
    if (!force) lay_out(std::min((slots + h->num_sms - 1) / h->num_sms, most));
    if (!warps) { cudaStreamDestroy(h->stream); delete h; return PERM_EUNSUPPORTED; }
    const long long per_cta_eff = (long long)warps * lanes;
    // (sequences beyond the layout wait at tour boundaries)
    if (!force) slots = std::min(slots, (long long)h->num_sms * per_cta_eff);
    h->ctas = (int)((slots + per_cta_eff - 1) / per_cta_eff);
    // helpers are the walks beyond the tour walks (fewer when not all fit).  A batch
    // member is laid out for the whole grid and its walks are granted per sequence by
    // the batch kernel, so none of its walks is a helper by position
    h->tour_slots = force ? (int)slots : (int)std::min(tslots, slots);
    h->worker_warps = warps;
    h->lanes = lanes;
    // twice the hash where the CTA's walks then still fit: a bucket that is full sends its
    // probe, and the warp, to another (n = 255, 4096 sequences, 64 tours: square 18.0 ->
    // 16.8 ms, cubic 16.7 -> 15.6)
    if (cfg->hash_scale == 0 && arena_mode == perm::kArenaNone && log2h < 16) {
        const size_t twice = perm::walk_bytes(key64, n_max, log2h + 1, h->stack_cache);
        if (head_b + twice * (size_t)(warps * lanes) <= budget) {
            walk_b = twice;
            h->log2h = ++log2h;
        }
    }
    h->slots = (int)slots;
    h->smem = smem_for(warps * lanes);
    // the batch kernel grows its members with the shared-memory body only
    if (force && arena_mode != perm::kArenaNone) { cudaStreamDestroy(h->stream); delete h; return PERM_EUNSUPPORTED; }
    h->arena_mode = arena_mode;
    if (arena_mode != perm::kArenaNone) {
        h->arena_cta_bytes = (long long)(walk_b * (size_t)(warps * lanes) + (arena_mode == perm::kArenaAll ? head_b : 0));
        h->arena_cta_bytes = (h->arena_cta_bytes + 255) & ~255LL;
        // at most 64 GB of walk state
        if ((double)h->arena_cta_bytes * h->ctas > 64e9) { cudaStreamDestroy(h->stream); delete h; return PERM_ENOMEM; }
    }

    const size_t L = (size_t)n_max + 1;
    h->ntab = (cfg->alg == PERM_ALG1) ? n_seq : 1;
    int rc = PERM_OK;
    h->share = cfg->share_copies >= 0 && cfg->alg == PERM_ALG2 && h->thresh == perm::kSnapshot;
    h->xrows = h->slots * (h->share ? 2 : 1);
    // shared copies: a ring of cells, each one waiting copy record plus the keys of the
    // walk up to its branch point (header, the keys of sites 0..n_max, their hash slots)
    h->share_cap = cfg->share_copies > 0 ? cfg->share_copies : kDefaultShareCap;
    size_t cells = 0;
    if (h->share) {
        int lc = 6;
        while ((1 << lc) < h->slots && lc < 12) ++lc;
        h->dq_log2cap = lc;
        h->dq_cell_bytes = (int)(32 + ((((size_t)n_max + 1) * (key64 ? 8 : 4) + 15) & ~(size_t)15) +
                                 ((((size_t)n_max + 1) * 2 + 15) & ~(size_t)15));
        cells = (size_t)1 << lc;
    }
    // the block a reset zeroes
    const size_t cnt = L * (size_t)h->ntab;
    size_t off = 0;
    auto place = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + kLine - 1) / kLine * kLine;
        return at;
    };
    const size_t o_counters = place(kCounters * kLine), o_W = place(cnt * 8), o_Q = place(cnt * 8), o_S = place(cnt * 8);
    const size_t o_R = cfg->observables ? place(cnt * 8) : 0, o_M = place((size_t)n_seq * 8);
    if (h->thresh == perm::kSnapshot && n_max <= kPartsLengths && h->slots >= kPartsWalks) h->parts = kParts;
    const size_t o_Wp = place((size_t)(h->parts - 1) * kPartStride * 8), o_Qp = place((size_t)(h->parts - 1) * kPartStride * 8);
    const size_t o_ready = place(cells * 4), o_free = place(cells * 4), o_tmax = place(h->share ? (size_t)h->xrows * 4 : 0);
    h->zero_bytes = off;
    rc = dalloc(h, &h->block, off);
    if (rc == PERM_OK) {
        unsigned char *B = h->block;
        auto counter = [&](int i) { return reinterpret_cast<unsigned long long *>(B + o_counters + (size_t)i * kLine); };
        h->Wn = reinterpret_cast<double *>(B + o_W);
        h->Qn = reinterpret_cast<double *>(B + o_Q);
        h->Sn = reinterpret_cast<unsigned long long *>(B + o_S);
        if (h->parts > 1) {
            h->Wp = reinterpret_cast<double *>(B + o_Wp);
            h->Qp = reinterpret_cast<double *>(B + o_Qp);
        }
        if (cfg->observables) h->Rn = reinterpret_cast<double *>(B + o_R);
        h->seq_M = reinterpret_cast<unsigned long long *>(B + o_M);
        h->tickets = counter(kTickets);
        h->steps = counter(kSteps);
        h->max_stack = counter(kMaxStack);
        h->copies = counter(kCopies);
        h->refreshes = counter(kRefreshes);
        h->iterations = counter(kIterations);
        h->finished = counter(kFinished);
        h->exact_steps = counter(kExact);
        h->status = reinterpret_cast<int *>(counter(kStatus));
        h->admit = reinterpret_cast<long long *>(counter(kAdmit));
        if (h->share) {
            h->dq_head = counter(kHead);
            h->dq_tail = counter(kTail);
            h->hungry = reinterpret_cast<int *>(counter(kHungry));
            h->queued = reinterpret_cast<int *>(counter(kQueued));
            h->dq_used = reinterpret_cast<int *>(counter(kUsed));
            h->dq_ready = reinterpret_cast<unsigned int *>(B + o_ready);
            h->dq_free = reinterpret_cast<unsigned int *>(B + o_free);
            h->tmaxn = reinterpret_cast<unsigned int *>(B + o_tmax);
        }
    }
    if (rc == PERM_OK) rc = dalloc(h, &h->X, L * (size_t)h->xrows);
    if (rc == PERM_OK) rc = dalloc(h, &h->gstk_meta, (size_t)n_max * h->slots);
    if (rc == PERM_OK) rc = dalloc(h, &h->gstk_w, (size_t)n_max * h->slots);
    if (rc == PERM_OK && h->arena_mode != perm::kArenaNone)
        rc = dalloc(h, &h->arena, (size_t)h->arena_cta_bytes * (size_t)h->ctas);
    if (rc == PERM_OK) rc = dalloc(h, &h->trace_count, 1);
    if (rc == PERM_OK && h->share) {
        rc = dalloc(h, &h->dq_cells, cells * (size_t)h->dq_cell_bytes);
        if (rc == PERM_OK) rc = dalloc(h, &h->outst, (size_t)h->xrows);
        if (rc == PERM_OK) rc = to_code(cudaMemsetAsync(h->outst, 0xFF, sizeof(unsigned int) * h->xrows, h->stream));
    }
    if (rc == PERM_OK) rc = to_code(cudaStreamSynchronize(h->stream));
    if (rc != PERM_OK) {
        free_all(h);
        cudaStreamDestroy(h->stream);
        delete h;
        return rc;
    }
    *out = h;
    return PERM_OK;
}

}  // namespace

extern "C" {

int perm_create_ex(perm_handle *out, const perm_config *cfg) { return create_impl(out, cfg, nullptr); }

int perm_create(perm_handle *out, int d, int n_max, int n_seq, uint64_t seed) {
    perm_config cfg;
    perm_config_init(&cfg, d, n_max, n_seq, seed);
    return perm_create_ex(out, &cfg);
}

int perm_set_stream(perm_handle h, void *stream) {
    if (!h) return PERM_EINVAL;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return PERM_EDEVICE;
    if (h->own_stream) cudaStreamDestroy(h->stream);
    h->stream = (cudaStream_t)stream;
    h->own_stream = false;
    return PERM_OK;
}

static RunDev make_params(perm_handle h) {
    RunDev P;
    std::memset(&P, 0, sizeof(P));
    P.d = h->cfg.d; P.n_max = h->cfg.n_max; P.n_seq = h->cfg.n_seq; P.alg = h->cfg.alg;
    P.log2h = h->log2h; P.S = h->lanes;
    P.worker_warps = h->worker_warps; P.slots = h->slots; P.tour_slots = h->tour_slots;
    P.stack_cache = h->stack_cache;
    P.arena_mode = h->arena_mode; P.arena = h->arena; P.arena_cta_bytes = h->arena_cta_bytes;
    P.key0 = (uint32_t)h->cfg.seed ^ h->cfg.run_id;
    P.key1 = (uint32_t)(h->cfg.seed >> 32);
    P.tour_limit = h->tour_limit;
    P.seq_target = h->seq_target;
    P.refresh_ns = h->cfg.refresh_ns;
    P.max_ns = (long long)(h->cfg.max_seconds * 1e9);
    // original PERM keeps one table, so that its tables agree with a sequential sum of the same
    // weights (within 5e-15; with four copies within 3.5e-14).  That is agreement, not accuracy: its
    // weights repeat, equal terms round the same way each time, and both then are 3.4e-14 from the
    // exact sum (four copies 1.1e-14; square, n = 257, 16000 tours)
    P.parts = h->cut ? 1 : h->parts; P.part_stride = kPartStride; P.Wp = h->Wp; P.Qp = h->Qp;
    P.Wn = h->Wn; P.Sn = h->Sn; P.Qn = h->Qn; P.Rn = h->Rn; P.tickets = h->tickets; P.seq_M = h->seq_M;
    P.X = h->X; P.gstk_meta = h->gstk_meta; P.gstk_w = h->gstk_w;
    P.steps = h->steps; P.max_stack = h->max_stack; P.copies = h->copies; P.refreshes = h->refreshes; P.iterations = h->iterations;
    P.exact_steps = h->exact_steps;
    P.finished = h->finished;
    P.admit = h->admit;
    // cut-offs read no table, so tours need not wait for samples of others: unless the caller
    // gave a limit they all start at once (cubic chains, n_max 10000, 608 sequences, 4 tours each, from
    // an empty run: 97.8 -> 26.1 ms; square, n = 257, 2000 sequences, 8 tours: 10.8 -> 9.2)
    const bool no_limit = h->cut != nullptr && !h->own_limit;
    P.ramp_c0 = h->cfg.ramp_c0 < 0 || no_limit ? -1 : (long long)h->cfg.ramp_c0;
    P.ramp_gamma_q16 = (unsigned long long)(h->cfg.ramp_gamma * 65536.0);
    P.share = h->share ? h->share_cap : 0;
    P.share_boost = h->share ? std::max(h->share_cap, kBoostShareCap) : 0;
    P.stall_ns = kStallNs;
    P.dq_log2cap = h->dq_log2cap; P.dq_cell_bytes = h->dq_cell_bytes; P.dq_cells = h->dq_cells;
    P.dq_head = h->dq_head; P.dq_tail = h->dq_tail; P.dq_ready = h->dq_ready; P.dq_free = h->dq_free;
    P.outst = h->outst; P.tmaxn = h->tmaxn; P.hungry = h->hungry; P.queued = h->queued; P.dq_used = h->dq_used;
    P.status = h->status;
    P.cut = h->cut;
    P.cut_copies = h->cut_copies;
    P.cut_q = h->cut_q;
    P.cut_inv_q = 1.0 / h->cut_q;
    // survive iff u0 < 1/q, i.e. w0 < 2^32 fl(1/q), i.e. w0 < ceil(2^32 fl(1/q)) (w0 integer)
    P.cut_K = (unsigned long long)std::ceil(P.cut_inv_q * 4294967296.0);
    P.trace = (h->trace_every > 0) ? h->trace : nullptr;
    P.trace_coords = h->trace_coords; P.trace_count = h->trace_count; P.trace_cap = h->trace_cap;
    P.trace_every = h->trace_every > 0 ? h->trace_every : 1;
    P.trace_tour_every = h->trace_tour_every > 0 ? h->trace_tour_every : 1;
    return P;
}

int perm_set_cutoffs(perm_handle h, const double *T_hi, const double *t_lo, int copies, double q) {
    if (!h) return PERM_EINVAL;
    if (!T_hi && !t_lo) {                                   // back to flatPERM
        if (h->cut) {
            if (cudaStreamSynchronize(h->stream) != cudaSuccess) return PERM_EDEVICE;
            cudaFree(h->cut);
            h->device_bytes -= (long long)(sizeof(double2) * ((size_t)h->cfg.n_max + 1));
        }
        h->cut = nullptr;
        return PERM_OK;
    }
    if (!T_hi || !t_lo || copies < 1 || copies > 2 * h->cfg.d || !(q >= 1.0) || q > 4294967296.0)
        return PERM_EINVAL;
    const size_t L = (size_t)h->cfg.n_max + 1;
    std::vector<double2> host(L);
    for (size_t k = 0; k < L; ++k) host[k] = clean_cutoffs(T_hi[k], t_lo[k]);
    if (!h->cut) {
        const int rc = dalloc(h, &h->cut, L);
        if (rc != PERM_OK) return rc;
    }
    // the copy is ordered on the handle's stream, after any launch already queued
    cudaError_t e = cudaMemcpyAsync(h->cut, host.data(), sizeof(double2) * L, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return to_code(e);
    h->cut_copies = copies;
    h->cut_q = q;
    return PERM_OK;
}

int perm_run(perm_handle h, int64_t tours_per_seq) {
    if (!h || tours_per_seq < 0) return PERM_EINVAL;
    if (tours_per_seq == 0) return PERM_OK;
    cudaError_t e;
    if (h->cfg.alg == PERM_ALG2) {
        h->tour_limit += tours_per_seq * (long long)h->cfg.n_seq;
    } else {
        h->seq_target += tours_per_seq;
        e = cudaMemsetAsync(h->tickets, 0, sizeof(unsigned long long), h->stream);
        if (e != cudaSuccess) return to_code(e);
    }
    h->unread = true;
    const RunDev P = make_params(h);
    e = perm::launch_grow(P, h->thresh, h->key64, h->ctas, h->stream);
    if (e != cudaSuccess) return to_code(e);
    if (h->cfg.alg == PERM_ALG2) {
        e = perm::launch_finalize(P, h->stream);
        if (e != cudaSuccess) return to_code(e);
    }
    return PERM_OK;
}

// Copy device -> host on the handle's own stream and wait for that stream only
// (other streams, e.g. other runs served concurrently, keep running).
static cudaError_t copy_out(perm_handle h, void *dst, const void *src, size_t bytes) {
    cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    return e;
}

// The status of everything queued so far, as it came back.
static void took_status(perm_handle h, int st) {
    h->last_status = st;
    h->unread = false;
}

// Wait for the stream; the run's status (one copy: it orders after the run and reports
// its failure).
static int sync_status(perm_handle h) {
    int st = 0;
    const cudaError_t e = copy_out(h, &st, h->status, sizeof(int));
    if (e != cudaSuccess) return to_code(e);
    took_status(h, st);
    return st;
}

int perm_run_sync(perm_handle h, int64_t tours_per_seq) {
    int rc = perm_run(h, tours_per_seq);
    if (rc != PERM_OK) return rc;
    return sync_status(h);
}

int perm_tables(perm_handle h, double *W_n, double *S_n, double *Q_n, int64_t *M) {
    if (!h) return PERM_EINVAL;
    const size_t L = (size_t)h->cfg.n_max + 1, cnt = L * h->ntab;
    const unsigned char *from = h->block;
    const size_t o_W = (size_t)(reinterpret_cast<unsigned char *>(h->Wn) - from), o_Q = (size_t)(reinterpret_cast<unsigned char *>(h->Qn) - from),
                 o_S = (size_t)(reinterpret_cast<unsigned char *>(h->Sn) - from), upto = o_S + cnt * 8;
    cudaError_t e = cudaSuccess;
    int st;
    if (upto <= kOneCopy) {
        // the counters and the tables in one copy (each costs about 10 us of host time)
        std::vector<unsigned char> buf(upto);
        e = copy_out(h, buf.data(), from, upto);
        if (e != cudaSuccess) return to_code(e);
        std::memcpy(&st, buf.data() + kStatus * kLine, sizeof(int));
        took_status(h, st);
        if (st < 0 && st != PERM_EOVERFLOW && st != PERM_ETIMEOUT) return st;
        if (W_n) std::memcpy(W_n, buf.data() + o_W, cnt * 8);
        if (Q_n) std::memcpy(Q_n, buf.data() + o_Q, cnt * 8);
        if (S_n) counts_from_differences(buf.data() + o_S, cnt, L, S_n);
    } else {
        st = sync_status(h);
        if (st < 0 && st != PERM_EOVERFLOW && st != PERM_ETIMEOUT) return st;
        if (W_n) e = copy_out(h, W_n, h->Wn, cnt * sizeof(double));
        if (e == cudaSuccess && Q_n) e = copy_out(h, Q_n, h->Qn, cnt * sizeof(double));
        if (e == cudaSuccess && S_n) {
            e = copy_out(h, S_n, h->Sn, cnt * sizeof(unsigned long long));
            if (e == cudaSuccess) counts_from_differences(S_n, cnt, L, S_n);
        }
    }
    if (e == cudaSuccess && M) {
        if (h->cfg.alg == PERM_ALG2) {
            M[0] = h->tour_limit;
        } else {
            std::vector<unsigned long long> m(h->cfg.n_seq);
            e = copy_out(h, m.data(), h->seq_M, m.size() * sizeof(unsigned long long));
            for (size_t i = 0; i < m.size(); ++i) M[i] = (int64_t)m[i];
        }
    }
    if (e != cudaSuccess) return to_code(e);
    return st;
}

int perm_reset(perm_handle h) {
    if (!h) return PERM_EINVAL;
    const size_t L = (size_t)h->cfg.n_max + 1;
    cudaError_t e = cudaMemsetAsync(h->block, 0, h->zero_bytes, h->stream);
    // a stopped run may leave tour sums behind, and one that is not known to have completed
    if (e == cudaSuccess && (h->last_status != PERM_OK || h->unread))
        e = cudaMemsetAsync(h->X, 0, L * (size_t)h->xrows * sizeof(double), h->stream);
    if (e == cudaSuccess && h->share)
        e = cudaMemsetAsync(h->outst, 0xFF, sizeof(unsigned int) * h->xrows, h->stream);
    if (e != cudaSuccess) return to_code(e);
    h->tour_limit = 0;
    h->seq_target = 0;
    took_status(h, PERM_OK);
    return PERM_OK;
}

int perm_estimates_from_tables(int d, int n_max, int rows, const double *W_n, const double *Q_n,
                               const int64_t *M, int combine, double *log_cn, double *relvar_n) {
    if ((d != 2 && d != 3) || n_max < 0 || rows < 1 || !W_n || !M) return PERM_EINVAL;
    if (combine != PERM_COMBINE_MEAN && combine != PERM_COMBINE_GEOMETRIC) return PERM_EINVAL;
    const size_t L = (size_t)n_max + 1;
    const double log2 = std::log(2.0);
    for (size_t n = 0; n < L; ++n) {
        // per row: the sample average c = W_n / M (eq. 4, any M >= 1) and the
        // per-tour variance of it, (Q_n / M - c^2) / (M - 1) (M >= 2)
        double mean = 0.0, mlog = 0.0, var = 0.0, rvar = 0.0;
        bool ok = Q_n != nullptr, any_zero = false;
        for (int t = 0; t < rows; ++t) {
            const int64_t m = M[t];
            if (m < 1) return PERM_EINVAL;
            const double c = W_n[(size_t)t * L + n] / (double)m;
            mean += c;
            if (c > 0.0) mlog += std::log(c); else any_zero = true;
            if (m < 2 || !Q_n) { ok = false; continue; }
            double v = (Q_n[(size_t)t * L + n] / (double)m - c * c) / (double)(m - 1);
            if (v < 0.0) v = 0.0;
            var += v;
            if (c > 0.0) rvar += v / (c * c);
        }
        const double R = (double)rows;
        const double shift = scale_exp_host(d, (int)n) * log2;
        double lc, rv;
        if (combine == PERM_COMBINE_MEAN) {
            // the average of the rows' sample averages (Sec. 3; one row: eq. 4)
            mean /= R;
            lc = mean > 0.0 ? std::log(mean) + shift : -INFINITY;
            rv = (ok && mean > 0.0) ? (var / (R * R)) / (mean * mean) : INFINITY;
        } else {
            // the mean of the rows' log sample averages (the geometric combination of
            // Sec. 4); its variance to first order is the mean relative variance / rows
            lc = any_zero ? -INFINITY : mlog / R + shift;
            rv = (ok && !any_zero) ? rvar / (R * R) : INFINITY;
        }
        if (log_cn) log_cn[n] = lc;
        if (relvar_n) relvar_n[n] = rv;
    }
    return PERM_OK;
}

int perm_estimates(perm_handle h, double *log_cn, double *S_n, double *relvar_n) {
    if (!h) return PERM_EINVAL;
    const size_t L = (size_t)h->cfg.n_max + 1, cnt = L * h->ntab;
    std::vector<double> W(cnt), S(cnt), Q(cnt);
    std::vector<int64_t> M(h->ntab);
    int rc = perm_tables(h, W.data(), S.data(), Q.data(), M.data());
    if (rc != PERM_OK) return rc;
    for (int t = 0; t < h->ntab; ++t) {
        if (M[t] < 1) {                          // no tour yet: nothing estimated
            for (size_t n = 0; n < L; ++n) {
                if (log_cn) log_cn[n] = -INFINITY;
                if (relvar_n) relvar_n[n] = INFINITY;
                if (S_n) S_n[n] = 0.0;
            }
            return PERM_OK;
        }
    }
    rc = perm_estimates_from_tables(h->cfg.d, h->cfg.n_max, h->ntab, W.data(), Q.data(), M.data(),
                                    PERM_COMBINE_MEAN, log_cn, relvar_n);
    if (rc != PERM_OK) return rc;
    if (S_n) {
        for (size_t n = 0; n < L; ++n) {
            double s = 0.0;
            for (int t = 0; t < h->ntab; ++t) s += S[(size_t)t * L + n];
            S_n[n] = s;
        }
    }
    return PERM_OK;
}

int perm_observable_r2(perm_handle h, double *mean_r2, double *R_n) {
    if (!h || !mean_r2 || !h->Rn) return PERM_EINVAL;
    const size_t L = (size_t)h->cfg.n_max + 1, cnt = L * h->ntab;
    std::vector<double> W(cnt), R(cnt);
    std::vector<int64_t> M(h->ntab);
    int rc = perm_tables(h, W.data(), nullptr, nullptr, M.data());
    if (rc != PERM_OK) return rc;
    if (copy_out(h, R.data(), h->Rn, cnt * sizeof(double)) != cudaSuccess) return PERM_EDEVICE;
    for (size_t n = 0; n < L; ++n) {
        double num = 0.0, den = 0.0;
        for (int t = 0; t < h->ntab; ++t) {
            if (M[t] < 1) continue;
            num += R[(size_t)t * L + n] / (double)M[t];
            den += W[(size_t)t * L + n] / (double)M[t];
        }
        mean_r2[n] = den > 0.0 ? num / den : NAN;
    }
    if (R_n) for (size_t i = 0; i < cnt; ++i) R_n[i] = R[i];
    return PERM_OK;
}

int perm_stats(perm_handle h, perm_stats_t *out) {
    if (!h || !out) return PERM_EINVAL;
    unsigned char buf[kCounters * kLine];
    const cudaError_t e = copy_out(h, buf, h->block, sizeof(buf));
    if (e != cudaSuccess) return to_code(e);
    int st = 0;
    std::memcpy(&st, buf + kStatus * kLine, sizeof(int));
    took_status(h, st);
    if (st < 0 && st != PERM_EOVERFLOW && st != PERM_ETIMEOUT) return st;
    auto value = [&](int i) {
        unsigned long long v;
        std::memcpy(&v, buf + (size_t)i * kLine, 8);
        return v;
    };
    const unsigned long long steps = value(kSteps), ms = value(kMaxStack), cp = value(kCopies), rf = value(kRefreshes),
                             it = value(kIterations), fin = value(kFinished), ex = value(kExact), shr = value(kTail);
    out->steps = (int64_t)steps;
    out->tours = h->cfg.alg == PERM_ALG2 ? h->tour_limit : h->seq_target * h->cfg.n_seq;
    out->max_stack = (int64_t)ms;
    out->copies = (int64_t)cp;
    out->refreshes = (int64_t)rf;
    out->iterations = (int64_t)it;
    out->slots = h->slots;
    out->ctas = h->ctas;
    out->lanes_per_warp = h->lanes;
    out->warps_per_cta = h->worker_warps;
    out->hash_slots = 1 << h->log2h;
    out->status = st;
    out->device_bytes = h->device_bytes;
    out->tours_finished = (int64_t)fin;
    out->shared = (int64_t)shr;
    out->exact_steps = (int64_t)ex;
    out->walk_memory = h->arena_mode == perm::kArenaNone ? 1 : 2;
    out->pad = 0;
    return PERM_OK;
}

int perm_trace_enable(perm_handle h, int64_t every, int64_t tour_every, int capacity) {
    if (!h || every < 0 || tour_every < 0 || capacity < 0) return PERM_EINVAL;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return PERM_EDEVICE;
    if (h->trace) { cudaFree(h->trace); h->trace = nullptr; }
    if (h->trace_coords) { cudaFree(h->trace_coords); h->trace_coords = nullptr; }
    h->trace_every = every;
    h->trace_tour_every = tour_every > 0 ? tour_every : 1;
    h->trace_cap = 0;
    if (every == 0 || capacity == 0) { h->trace_every = 0; return PERM_OK; }
    const size_t L = (size_t)h->cfg.n_max + 1;
    if (cudaMalloc((void **)&h->trace, sizeof(perm_trace_record) * (size_t)capacity) != cudaSuccess ||
        cudaMalloc((void **)&h->trace_coords, sizeof(int32_t) * (size_t)capacity * L * h->cfg.d) != cudaSuccess) {
        h->trace_every = 0;
        return PERM_ENOMEM;
    }
    h->trace_cap = capacity;
    if (cudaMemset(h->trace_count, 0, 8) != cudaSuccess) return PERM_EDEVICE;
    return PERM_OK;
}

int perm_trace_read(perm_handle h, int64_t *count, perm_trace_record *recs, int32_t *coords) {
    if (!h) return PERM_EINVAL;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return PERM_EDEVICE;
    unsigned long long c = 0;
    if (cudaMemcpy(&c, h->trace_count, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return PERM_EDEVICE;
    if (count) *count = (int64_t)c;
    const size_t kept = c < (unsigned long long)h->trace_cap ? (size_t)c : (size_t)h->trace_cap;
    const size_t L = (size_t)h->cfg.n_max + 1;
    if (recs && kept && cudaMemcpy(recs, h->trace, kept * sizeof(perm_trace_record), cudaMemcpyDeviceToHost) != cudaSuccess)
        return PERM_EDEVICE;
    if (coords && kept && cudaMemcpy(coords, h->trace_coords, kept * L * h->cfg.d * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
        return PERM_EDEVICE;
    return PERM_OK;
}

void perm_destroy(perm_handle h) {
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    free_all(h);
    if (h->own_stream) cudaStreamDestroy(h->stream);
    delete h;
}

static int debug_step(int d, int n_max, int B, const int32_t *coords, const int32_t *len,
                      const double *W, const double *Wsum, const uint64_t *M,
                      const uint64_t *ordinal, const uint32_t *seq, const uint32_t *tour,
                      uint64_t seed, uint32_t run_id, bool snapshot, int force_exact, int32_t *out_i,
                      double *out_r, double *out_w, void *stream) {
    if ((d != 2 && d != 3) || n_max < 1 || n_max > 512 || B < 0) return PERM_EINVAL;
    if (force_exact != 0 && force_exact != 1) return PERM_EINVAL;
    if (B > 0 && (!coords || !len || !W || !Wsum || !M || !ordinal || !seq || !tour || !out_i ||
                  !out_r || !out_w))
        return PERM_EINVAL;
    cudaError_t e = perm::launch_debug_step(d, n_max, B, coords, len, W, Wsum, M, ordinal, seq, tour,
                                            (uint32_t)seed ^ run_id, (uint32_t)(seed >> 32), snapshot, force_exact,
                                            out_i, out_r, out_w, (cudaStream_t)stream);
    return to_code(e);
}

int perm_debug_step(int d, int n_max, int B, const int32_t *coords, const int32_t *len,
                    const double *W, const double *Wsum, const uint64_t *M,
                    const uint64_t *ordinal, const uint32_t *seq, const uint32_t *tour,
                    uint64_t seed, uint32_t run_id, int force_exact, int32_t *out_i,
                    double *out_r, double *out_w, void *stream) {
    return debug_step(d, n_max, B, coords, len, W, Wsum, M, ordinal, seq, tour, seed, run_id, false, force_exact,
                      out_i, out_r, out_w, stream);
}

int perm_debug_step_snapshot(int d, int n_max, int B, const int32_t *coords, const int32_t *len,
                             const double *W, const double *Wsum, const uint64_t *M,
                             const uint64_t *ordinal, const uint32_t *seq, const uint32_t *tour,
                             uint64_t seed, uint32_t run_id, int force_exact, int32_t *out_i,
                             double *out_r, double *out_w, void *stream) {
    return debug_step(d, n_max, B, coords, len, W, Wsum, M, ordinal, seq, tour, seed, run_id, true, force_exact,
                      out_i, out_r, out_w, stream);
}

int perm_debug_philox(int B, const uint32_t *ctr, const uint32_t *key, uint32_t *out) {
    if (B < 0 || (B > 0 && (!ctr || !key || !out))) return PERM_EINVAL;
    cudaError_t e = perm::launch_debug_philox(B, ctr, key[0], key[1], out, nullptr);
    if (e != cudaSuccess) return to_code(e);
    return to_code(cudaDeviceSynchronize());
}

}  // extern "C"

namespace perm {

int member_create(perm_handle *out, const perm_config *cfg, int ctas, size_t smem_budget) {
    if (!cfg || ctas < 1) return PERM_EINVAL;
    if (cfg->alg != PERM_ALG2 || cfg->threshold != PERM_THRESH_SNAPSHOT) return PERM_EUNSUPPORTED;
    const ForcedLayout f{ctas, smem_budget};
    return create_impl(out, cfg, &f);
}

int member_params(perm_handle h, int64_t tours_per_seq, int run_index, RunDev *P, size_t *smem,
                  int *worker_warps) {
    if (!h || !P || tours_per_seq < 0) return PERM_EINVAL;
    h->tour_limit = tours_per_seq * (long long)h->cfg.n_seq;
    *P = make_params(h);
    P->run_index = run_index;
    if (smem) *smem = h->smem;
    if (worker_warps) *worker_warps = h->worker_warps;
    return PERM_OK;
}

int member_extend(perm_handle h, int64_t extra_tours_per_seq, int run_index, RunDev *P) {
    if (!h || !P || extra_tours_per_seq < 0) return PERM_EINVAL;
    h->tour_limit += extra_tours_per_seq * (long long)h->cfg.n_seq;
    *P = make_params(h);
    P->run_index = run_index;
    return PERM_OK;
}

int member_reset(perm_handle h) { return perm_reset(h); }

int member_clear_sums(perm_handle h) {
    const size_t L = (size_t)h->cfg.n_max + 1;
    return to_code(cudaMemsetAsync(h->X, 0, L * (size_t)h->xrows * sizeof(double), h->stream));
}

}  // namespace perm

// ---------------------------------------------------------------------------
// Checkpoint and resume at a tour boundary.  Between launches every tour of the
// handle has ended: the per-walk tour sums are zero, the stacks are empty and
// no copy waits in the donation ring, so the run's state is its tables, its
// tour counters and its statistics.  The random streams are counter-based
// (sequence, tour, node), so a resumed run draws what the uninterrupted run
// would have drawn.
// ---------------------------------------------------------------------------
namespace {

constexpr char kCkptMagic[8] = {'P', 'E', 'R', 'M', 'C', 'K', 'P', '1'};
constexpr uint32_t kCkptVersion = 3;

struct CkptHeader {
    char magic[8];
    uint32_t version;
    uint32_t header_bytes;
    perm_config cfg;               // as the handle holds it (defaults filled in, but for the admission limit)
    int64_t tour_limit, seq_target;
    int32_t ntab, has_rn, has_cut, cut_copies;
    double cut_q;
    uint64_t steps, max_stack, copies, refreshes, iterations, finished, exact_steps;
};

// Bytes of the arrays after the header, or 0 when the sizes make no sense.
uint64_t ckpt_payload(const CkptHeader &hd) {
    const uint64_t L = (uint64_t)hd.cfg.n_max + 1;
    if (hd.cfg.n_max < 1 || hd.cfg.n_seq < 1 || hd.cfg.n_max > (1 << 20)) return 0;
    const uint64_t ntab = hd.cfg.alg == PERM_ALG1 ? (uint64_t)hd.cfg.n_seq : 1;
    if ((uint64_t)hd.ntab != ntab || L * ntab > (1ull << 34)) return 0;
    const uint64_t cnt = L * ntab;
    return cnt * 8 * (3 + (hd.has_rn ? 1 : 0)) + (uint64_t)hd.cfg.n_seq * 8 + (hd.has_cut ? L * 16 : 0);
}

}  // namespace

extern "C" {

int perm_save(perm_handle h, const char *path) {
    if (!h || !path) return PERM_EINVAL;
    const int st = sync_status(h);
    if (st != PERM_OK) return st < 0 ? st : PERM_EINVAL;     // a failed run is not saved
    CkptHeader hd;
    std::memset(&hd, 0, sizeof(hd));
    std::memcpy(hd.magic, kCkptMagic, 8);
    hd.version = kCkptVersion;
    hd.header_bytes = (uint32_t)sizeof(CkptHeader);
    hd.cfg = h->cfg;
    if (!h->own_limit) { hd.cfg.ramp_c0 = 0; hd.cfg.ramp_gamma = 0.0; }    // the default again when loaded
    hd.tour_limit = h->tour_limit;
    hd.seq_target = h->seq_target;
    hd.ntab = h->ntab;
    hd.has_rn = h->Rn != nullptr;
    hd.has_cut = h->cut != nullptr;
    hd.cut_copies = h->cut_copies;
    hd.cut_q = h->cut_q;
    const size_t L = (size_t)h->cfg.n_max + 1, cnt = L * h->ntab;
    std::vector<double> W(cnt), Q(cnt), R(hd.has_rn ? cnt : 0);
    std::vector<unsigned long long> S(cnt), sM(h->cfg.n_seq);
    std::vector<double2> cut(hd.has_cut ? L : 0);
    cudaError_t e = copy_out(h, W.data(), h->Wn, cnt * 8);
    if (e == cudaSuccess) e = copy_out(h, Q.data(), h->Qn, cnt * 8);
    if (e == cudaSuccess) e = copy_out(h, S.data(), h->Sn, cnt * 8);
    counts_from_differences(S.data(), cnt, L, S.data());    // a checkpoint holds counts
    if (e == cudaSuccess && hd.has_rn) e = copy_out(h, R.data(), h->Rn, cnt * 8);
    if (e == cudaSuccess) e = copy_out(h, sM.data(), h->seq_M, sM.size() * 8);
    if (e == cudaSuccess && hd.has_cut) e = copy_out(h, cut.data(), h->cut, L * sizeof(double2));
    unsigned long long *cnts[7] = {h->steps, h->max_stack, h->copies, h->refreshes, h->iterations, h->finished,
                                   h->exact_steps};
    uint64_t *dst[7] = {&hd.steps, &hd.max_stack, &hd.copies, &hd.refreshes, &hd.iterations, &hd.finished,
                        &hd.exact_steps};
    for (int i = 0; e == cudaSuccess && i < 7; ++i) e = copy_out(h, dst[i], cnts[i], 8);
    if (e != cudaSuccess) return to_code(e);
    // write beside the target, then rename: a crash never leaves half a checkpoint
    const std::string tmp = std::string(path) + ".tmp";
    FILE *f = std::fopen(tmp.c_str(), "wb");
    if (!f) return PERM_EINVAL;
    bool ok = std::fwrite(&hd, sizeof(hd), 1, f) == 1;
    ok = ok && std::fwrite(W.data(), 8, cnt, f) == cnt;
    ok = ok && std::fwrite(Q.data(), 8, cnt, f) == cnt;
    ok = ok && std::fwrite(S.data(), 8, cnt, f) == cnt;
    if (hd.has_rn) ok = ok && std::fwrite(R.data(), 8, cnt, f) == cnt;
    ok = ok && std::fwrite(sM.data(), 8, sM.size(), f) == sM.size();
    if (hd.has_cut) ok = ok && std::fwrite(cut.data(), sizeof(double2), L, f) == L;
    ok = (std::fclose(f) == 0) && ok;
    if (!ok || std::rename(tmp.c_str(), path) != 0) {
        std::remove(tmp.c_str());
        return PERM_EINVAL;
    }
    return PERM_OK;
}

int perm_get_config(perm_handle h, perm_config *out) {
    if (!h || !out) return PERM_EINVAL;
    *out = h->cfg;
    return PERM_OK;
}

int perm_load(perm_handle *out, const char *path) {
    if (!out || !path) return PERM_EINVAL;
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) return PERM_EINVAL;
    CkptHeader hd;
    bool ok = std::fread(&hd, sizeof(hd), 1, f) == 1 && std::memcmp(hd.magic, kCkptMagic, 8) == 0 &&
              hd.version == kCkptVersion && hd.header_bytes == (uint32_t)sizeof(CkptHeader);
    const uint64_t payload = ok ? ckpt_payload(hd) : 0;
    ok = ok && payload > 0;
    // (not cleared: the file fills it)
    std::unique_ptr<unsigned char[]> body(ok ? new (std::nothrow) unsigned char[(size_t)payload] : nullptr);
    const bool room = !ok || body != nullptr;
    ok = ok && room && std::fread(body.get(), 1, (size_t)payload, f) == (size_t)payload;
    ok = ok && std::fgetc(f) == EOF;                        // nothing after the arrays
    std::fclose(f);
    if (!ok) return room ? PERM_EINVAL : PERM_ENOMEM;
    perm_handle h = nullptr;
    int rc = perm_create_ex(&h, &hd.cfg);
    if (rc != PERM_OK) return rc;
    if (hd.has_rn != (h->Rn != nullptr)) { perm_destroy(h); return PERM_EINVAL; }
    const size_t L = (size_t)hd.cfg.n_max + 1, cnt = L * (size_t)hd.ntab;
    unsigned char *p = body.get();
    auto put = [&](void *dev, size_t bytes) {
        cudaError_t e = cudaMemcpyAsync(dev, p, bytes, cudaMemcpyHostToDevice, h->stream);
        p += bytes;
        return e;
    };
    cudaError_t e = put(h->Wn, cnt * 8);
    if (e == cudaSuccess) e = put(h->Qn, cnt * 8);
    if (e == cudaSuccess) {
        differences_from_counts(p, cnt, L);
        e = put(h->Sn, cnt * 8);
    }
    if (e == cudaSuccess && hd.has_rn) e = put(h->Rn, cnt * 8);
    if (e == cudaSuccess) e = put(h->seq_M, (size_t)hd.cfg.n_seq * 8);
    if (e == cudaSuccess && hd.has_cut) {
        rc = dalloc(h, &h->cut, L);
        if (rc != PERM_OK) { perm_destroy(h); return rc; }
        std::vector<double2> cut(L);
        std::memcpy(cut.data(), p, L * sizeof(double2));
        for (double2 &c : cut) c = clean_cutoffs(c.x, c.y);
        p += L * sizeof(double2);
        e = cudaMemcpyAsync(h->cut, cut.data(), L * sizeof(double2), cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        h->cut_copies = hd.cut_copies;
        h->cut_q = hd.cut_q;
    }
    // the tour counter: Alg. 2 hands out tickets from the tours started so far
    const unsigned long long tickets = hd.cfg.alg == PERM_ALG2 ? (unsigned long long)hd.tour_limit : 0ull;
    const uint64_t vals[8] = {hd.steps, hd.max_stack, hd.copies, hd.refreshes, hd.iterations, hd.finished,
                              hd.exact_steps, tickets};
    unsigned long long *dev[8] = {h->steps, h->max_stack, h->copies, h->refreshes, h->iterations, h->finished,
                                  h->exact_steps, h->tickets};
    for (int i = 0; e == cudaSuccess && i < 8; ++i)
        e = cudaMemcpyAsync(dev[i], &vals[i], 8, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess && hd.cfg.alg == PERM_ALG2) {
        // every saved tour has finished: the admission count as a launch leaves it
        h->tour_limit = hd.tour_limit;
        e = perm::launch_finalize(make_params(h), h->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) { perm_destroy(h); return to_code(e); }
    h->tour_limit = hd.tour_limit;
    h->seq_target = hd.seq_target;
    *out = h;
    return PERM_OK;
}

}  // extern "C"
