// perm_kernels.cu -- the batch kernel (many runs in one persistent launch), the
// snapshot-state kernel of the tests, and the choice of a launch's kernel.
#include "perm_grow.cuh"

namespace perm {

namespace {

// ---------------------------------------------------------------------------
// Batch launch: R runs grown by one persistent grid.  Each CTA picks the open
// run (tours left to start, walks left to grant) with the most tours left to
// start per CTA already on it, weighted by n_max + 1, copies its descriptor to
// shared memory, lays its shared memory out for that run and grows it until
// the run is complete, or until its walks have no tickets left while another
// run is open; then it picks again.  A run's tour-growing walks (at most one per
// sequence, as in a single launch) are granted to the CTAs that join it.  With
// no run open, a CTA joins an unfinished run (a stalled one first) as a helper
// whose walks take waiting copies only.
// ---------------------------------------------------------------------------
// Takes walks of run r for this CTA (one walk per sequence over all CTAs); 0: none left.
__device__ int grant_walks(const BatchDev &B, int r) {
    const RunDev &Q = B.runs[r];
    const int cap = Q.worker_warps * Q.S;
    for (int attempt = 0; attempt < 64; ++attempt) {
        const int g = *(volatile int *)(B.granted + r);
        const int k = Q.n_seq - g < cap ? Q.n_seq - g : cap;
        if (k <= 0) break;
        if (atomicCAS(B.granted + r, g, g + k) == g) {
            if (g + k >= Q.n_seq && (atomicOr(B.closed + r, 2) & 3) == 0) atomicSub(B.runs_open, 1);
            return k;
        }
    }
    return 0;
}

// Returns the run to join (walks: how many of the CTA's walks grow tours), -1
// when no run can take the CTA now, -2 when every run has finished or failed.
__device__ int pick_run(const BatchDev &B, int &walks, bool &helper) {
    walks = 0;
    helper = false;
    for (int attempt = 0; attempt < 4; ++attempt) {
        int best = -1, stall = -1, seen = 0;
        double best_s = -1.0, stall_s = -1.0, next_s = -1.0, best_w = 0.0;
        bool best_open = false, unfinished = false;
        for (int r = 0; r < B.R; ++r) {
            const RunDev &Q = B.runs[r];
            if (*(volatile int *)Q.status != 0) continue;
            const long long lim = Q.tour_limit;
            const long long f = (long long)*(volatile unsigned long long *)Q.finished;
            if (f >= lim) continue;
            unfinished = true;
            const long long t = (long long)*(volatile unsigned long long *)Q.tickets;
            const int a = *(volatile int *)(B.active + r);
            const int g = *(volatile int *)(B.granted + r);
            const double len = (double)(Q.n_max + 1);
            // a run stalled on a large tour is the batch's critical path: among runs
            // that take helpers it comes first, up to the CTAs its parts can use
            const int fl = *(volatile int *)(B.closed + r);
            if ((fl & kStalledBit) && Q.share && a * Q.worker_warps * Q.S < Q.share_boost) {
                const double sc = (double)(lim - f) * len / (double)(a + 1);
                if (sc > stall_s) { stall = r; stall_s = sc; }
            }
            const bool open = t < lim;
            if (open ? g >= Q.n_seq : (best_open || !Q.share)) continue;
            const double w = (double)(open ? lim - t : lim - f) * len, sc = w / (double)(a + 1);
            if (open && !best_open) { best_s = next_s = -1.0; best_open = true; }
            if (sc > best_s) { next_s = best_s; best = r; best_s = sc; best_w = w; seen = a; }
            else if (sc > next_s) next_s = sc;
        }
        if (stall >= 0 && !best_open) { best = stall; next_s = -1.0; }
        if (best < 0) return unfinished ? -1 : -2;
        // CTAs that look at the same moment see the same best run: one that finds others have
        // joined it since looks again while another run now comes before it
        const int now = atomicAdd(B.active + best, 1);
        if (attempt < 3 && now > seen && best_w / (double)(now + 1) < next_s) {
            atomicSub(B.active + best, 1);
            continue;
        }
        if (best_open) {
            walks = grant_walks(B, best);
            if (walks == 0) {
                atomicSub(B.active + best, 1);
                return -1;
            }
        } else {
            walks = B.runs[best].worker_warps * B.runs[best].S;
            helper = true;
        }
        return best;
    }
    return -1;
}

template <int MODE, int FORM>
__global__ void __launch_bounds__(32 * (walk_warps_max(false) + 1), 1) batch_kernel(const BatchDev B) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RunDev Ps;
    __shared__ int cur, walks, helping;
    const long long t0 = global_ns();
    for (bool at_start = true;; at_start = false) {
        if (threadIdx.x == 0) {
            int w = 0;
            bool hp = false;
            int r = -1;
            if (at_start) {
                // (the launch's first runs were shared out by batch_init_kernel)
                r = B.first[blockIdx.x];
                if (r >= 0) {
                    w = grant_walks(B, r);
                    if (w > 0) atomicAdd(B.active + r, 1);
                    else r = -1;
                }
            }
            if (r < 0) r = pick_run(B, w, hp);
            helping = hp ? 1 : 0;
            if (r == -1 && global_ns() - t0 > B.max_ns) {
                // the batch's time is up: every run not finished fails
                for (int q = 0; q < B.R; ++q) {
                    const RunDev &Q = B.runs[q];
                    if ((long long)*(volatile unsigned long long *)Q.finished < Q.tour_limit)
                        set_status(Q.status, PERM_ETIMEOUT);
                }
                r = -2;
            }
            cur = r;
            walks = w;
        }
        __syncthreads();
        const int r = cur;
        if (r == -2) break;
        if (r == -1) {
            __nanosleep(8000);
            __syncthreads();
            continue;
        }
        const uint32_t *src = reinterpret_cast<const uint32_t *>(B.runs + r);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&Ps);
        for (int i = threadIdx.x; i < (int)(sizeof(RunDev) / 4); i += blockDim.x) dst[i] = __ldcg(src + i);
        __syncthreads();
        const BatchLeave bl{B.runs_open, B.closed, B.active + r, helping != 0};
        const int cw = walks;
        // a batch member's walks are laid out in shared memory (never the arena)
        if (Ps.d == 2) grow_run<2, uint32_t, MODE, true, FORM>(Ps, smem, &bl, cw);
        else if (Ps.n_max > 512) grow_run<3, unsigned long long, MODE, true, FORM>(Ps, smem, &bl, cw);
        else grow_run<3, uint32_t, MODE, true, FORM>(Ps, smem, &bl, cw);
        __syncthreads();
        if (threadIdx.x == 0) atomicSub(B.active + r, 1);
        __syncthreads();
    }
}

// Scheduling counters of a batch launch: nothing granted, no CTA on a run; a run
// with no tours left to start counts as closed.  And each CTA's first run: the CTAs go
// one by one to the run with the most work per CTA already given (at most the CTAs that
// hold one walk per sequence).  When every CTA chose for itself at the launch's start,
// they all saw the same empty counts, filled the largest runs and left the others, with
// their start-up, for later (24 runs of n = 64..256, 8 tours: 21.1 ms, so 15.5).
// One block of 256 threads; past kSharedOut runs every CTA chooses for itself.
constexpr int kSharedOut = 512;
__global__ void batch_init_kernel(const BatchDev B) {
    __shared__ int open;
    __shared__ float work[kSharedOut];     // 0: takes no CTA
    __shared__ int given[kSharedOut], most[kSharedOut];
    if (threadIdx.x == 0) open = 0;
    __syncthreads();
    for (int r = threadIdx.x; r < B.R; r += blockDim.x) {
        // a run grows in this launch if it has tours left to start (a continued
        // batch leaves retired runs with none)
        const RunDev &Q = B.runs[r];
        const long long left = Q.tour_limit - (long long)*(volatile unsigned long long *)Q.tickets;
        const bool grows = left > 0;
        B.active[r] = 0;
        B.granted[r] = 0;
        B.closed[r] = grows ? 0 : 3;
        if (grows) atomicAdd(&open, 1);
        if (r < kSharedOut) {
            const int cap = Q.worker_warps * Q.S;
            work[r] = grows ? (float)left * (float)(Q.n_max + 1) : 0.0f;
            given[r] = 0;
            most[r] = (Q.n_seq + cap - 1) / cap;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *B.runs_open = open;
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x, R = B.R <= kSharedOut ? B.R : 0;
    for (int b = 0; b < B.ctas; ++b) {
        float best_s = 0.0f;
        int best = -1;
        for (int r = lane; r < R; r += 32) {
            const float sc = given[r] < most[r] ? work[r] / (float)(given[r] + 1) : 0.0f;
            if (sc > best_s) { best_s = sc; best = r; }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float os = __shfl_xor_sync(kFull, best_s, off);
            const int ob = __shfl_xor_sync(kFull, best, off);
            if (os > best_s || (os == best_s && ob > best)) { best_s = os; best = ob; }
        }
        if (lane == 0) {
            B.first[b] = best;
            if (best >= 0) given[best] += 1;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Growth step on caller-given snapshot states (one group of lanes per state, one
// warp per block, as the persistent kernel's node).  REFINE: the fresh form's decision,
// else the snapshot form's.
// ---------------------------------------------------------------------------
template <int D, typename Key, bool REFINE>
__global__ void __launch_bounds__(32) debug_step_kernel(int n_max, int log2h, int B,
        const int32_t *coords, const int32_t *len, const double *Wv, const double *Wsv,
        const uint64_t *Mv, const uint64_t *ordv, const uint32_t *seqv, const uint32_t *tourv,
        uint32_t k0, uint32_t k1, int force_exact, int32_t *out_i, double *out_r, double *out_w) {
    constexpr int G = kGroupLanes<D>, kPer = 32 / G;
    extern __shared__ __align__(16) unsigned char smem[];
    double *aoc = reinterpret_cast<double *>(smem);
    const uint32_t *lists = reinterpret_cast<const uint32_t *>(aoc + kFactors);
    const int lane = threadIdx.x, grp = lane / G, j = lane % G, lead = lane - j;
    const int H = 1 << log2h, log2b = log2h - Buckets<Key>::kLog2;
    Key *all = reinterpret_cast<Key *>(smem + 1024);
    Key *hash = all + (size_t)H * grp;
    fill_constants(aoc, D, lane, 32);
    for (int s = lane; s < H * kPer; s += 32) all[s] = (Key)0;
    __syncwarp();
    const int b = blockIdx.x * kPer + grp;
    const bool have = b < B;
    const int n = have ? len[b] : -1;
    const bool good = n >= 0 && n <= n_max;
    if (have && !good && j == 0) out_i[(size_t)b * 11] = -1;
    const int32_t *cb = coords + (size_t)(good ? b : 0) * (n_max + 1) * D;
    // the walk's sites in order (the one at depth n_max is never inserted)
    bool ovf = false;
    const int last = good ? (n < n_max - 1 ? n : n_max - 1) : -1;
    for (int k = 0; __any_sync(kFull, k <= last); ++k) {
        Key key = KeyCodec<D, Key>::encode(0, 0, 0);
        if (k <= last) key = KeyCodec<D, Key>::encode(cb[k * D], cb[k * D + 1], D == 3 ? cb[k * D + 2] : 0);
        int slot = 0;
        bool o = false;
        const bool absent = probe<Key>(hash, log2b, key, k <= last, slot, o);
        ovf = ovf || (k <= last && !absent);
        __syncwarp();
        if (j == 0 && absent) hash[slot] = key;
        __syncwarp();
    }
    Key cur = KeyCodec<D, Key>::encode(0, 0, 0);
    if (good) cur = KeyCodec<D, Key>::encode(cb[n * D], cb[n * D + 1], D == 3 ? cb[n * D + 2] : 0);
    const double W = good ? Wv[b] : 1.0, Wsum = good ? Wsv[b] : 1.0;
    const unsigned long long M = good ? Mv[b] : 1ull, ordinal = good ? ordv[b] : 0ull;
    const Philox4 w = philox4x32_10((uint32_t)ordinal, (uint32_t)(ordinal >> 32), good ? tourv[b] : 0u,
                                    good ? seqv[b] : 0u, k0, k1);
    int slot = 0;
    const bool grows_on = good && n < n_max;
    const bool free_j = probe<Key>(hash, log2b, cur + step_key<D, Key>(j < 2 * D ? j : 0), grows_on && j < 2 * D, slot, ovf);
    const int fm = (int)((__ballot_sync(kFull, free_j) >> lead) & ((1u << G) - 1u));
    ovf = ((__ballot_sync(kFull, ovf) >> lead) & ((1u << G) - 1u)) != 0u;
    const int a = __popc(fm);
    const bool decides = grows_on && a > 0;
    Tours t;
    set_tours<true>(t, M);
    const double sum = __dadd_rn(Wsum, W);
    const Decision o = decide_node<D>(good ? n : 0, a > 0 ? a : 1, W, sum, guess(W, Wsum, t.Mf, w.x), t,
                                      REFINE, false, w.x, aoc, decides, decides && force_exact != 0);
    if (!good || j != 0) return;
    const int c = decides ? o.c : 0;
    uint32_t dirs = lists[fm], xw = w.y;
    for (int i = 0; i < c; ++i) choose_step(i, a, dirs, xw);
    int32_t *oi = out_i + (size_t)b * 11;
    oi[0] = ovf ? -2 : (!grows_on ? kLeafNmax : (a == 0 ? kTrapped : (c == 0 ? kPruned : kChildren)));
    oi[1] = a;
    oi[2] = fm;
    oi[3] = c;
    for (int i = 0; i < 6; ++i) oi[4 + i] = (i < c) ? (int)((dirs >> (3 * i)) & 7u) : -1;
    oi[10] = decides && o.exact ? 1 : 0;
    out_r[b] = decision_r(o, n, false);
    out_w[b] = c > 0 ? o.child_w : 0.0;
}

__global__ void philox_kernel(int B, const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const Philox4 w = philox4x32_10(ctr[4 * b], ctr[4 * b + 1], ctr[4 * b + 2], ctr[4 * b + 3], k0, k1);
    out[4 * b] = w.x; out[4 * b + 1] = w.y; out[4 * b + 2] = w.z; out[4 * b + 3] = w.w;
}

__global__ void finalize_kernel(const RunDev P) {
    if (threadIdx.x == 0) {
        const long long limit = P.tour_limit;
        if ((long long)*P.tickets > limit) *P.tickets = (unsigned long long)limit;
        // every tour has finished: what the admission rule leaves beyond them
        const long long extra = (long long)(((unsigned long long)limit * P.ramp_gamma_q16) >> 16);
        P.admit[0] = extra;
        P.admit[1] = limit + extra;
    }
    // the tables' further copies into the first
    if (P.parts > 1) {
        for (int k = threadIdx.x; k <= P.n_max; k += blockDim.x) {
            double w = P.Wn[k], q = P.Qn[k];
            for (int r = 0; r + 1 < P.parts; ++r) {
                const size_t at = (size_t)r * (size_t)P.part_stride + (size_t)k;
                w = __dadd_rn(w, P.Wp[at]);
                q = __dadd_rn(q, P.Qp[at]);
                P.Wp[at] = 0.0;
                P.Qp[at] = 0.0;
            }
            P.Wn[k] = w;
            P.Qn[k] = q;
        }
    }
}

// An inclusive sum of L entries in place, by one block: each thread a run of entries.
__global__ void __launch_bounds__(1024) counts_kernel(unsigned long long *S, int L) {
    __shared__ unsigned long long part[1024];
    const int per = (L + (int)blockDim.x - 1) / (int)blockDim.x;
    const int lo = min(L, (int)threadIdx.x * per), hi = min(L, lo + per);
    unsigned long long sum = 0ull;
    for (int i = lo; i < hi; ++i) sum += S[i];
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
        const unsigned long long v = (int)threadIdx.x >= off ? part[threadIdx.x - off] : 0ull;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned long long run = part[threadIdx.x] - sum;
    for (int i = lo; i < hi; ++i) { run += S[i]; S[i] = run; }
}

}  // namespace

bool plain_run(const RunDev &P) {
    return P.cut == nullptr && P.Rn == nullptr && P.trace == nullptr && P.arena_mode == kArenaNone;
}

size_t cta_head_bytes(int n_max, bool snapshot) { return head_region_bytes(n_max, snapshot); }

size_t walk_bytes(bool key64, int n_max, int log2h, int stack_cache) {
    return walk_region_bytes(n_max, log2h, stack_cache, key64 ? 8 : 4);
}

int walks_per_warp_max(int d) { return 32 / (d == 2 ? kGroupLanes<2> : kGroupLanes<3>); }

cudaError_t batch_smem_budget(size_t *dynamic_max) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa, fg;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, batch_kernel<kSnapshot, kPlain>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fg, batch_kernel<kSnapshot, kWatched>);
    if (e != cudaSuccess) return e;
    const long long held = (long long)(fa.sharedSizeBytes > fg.sharedSizeBytes ? fa.sharedSizeBytes : fg.sharedSizeBytes);
    const long long dyn = (long long)optin - held;
    if (dyn <= 0) return cudaErrorInvalidValue;
    *dynamic_max = (size_t)dyn;
    e = cudaFuncSetAttribute(batch_kernel<kSnapshot, kPlain>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_kernel<kSnapshot, kWatched>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    return e;
}

cudaError_t batch_grid(int threads, size_t smem, int *ctas) {
    int dev = 0, sms = 0, per_sm = 0, per_sm_g = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<kSnapshot, kPlain>, threads, smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_g, batch_kernel<kSnapshot, kWatched>, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm_g < per_sm) per_sm = per_sm_g;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *ctas = sms * per_sm;
    return cudaSuccess;
}

cudaError_t launch_batch(const BatchDev &B, int ctas, int threads, size_t smem, cudaStream_t stream) {
    batch_init_kernel<<<1, 256, 0, stream>>>(B);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (B.plain) batch_kernel<kSnapshot, kPlain><<<ctas, threads, smem, stream>>>(B);
    else batch_kernel<kSnapshot, kWatched><<<ctas, threads, smem, stream>>>(B);
    return cudaGetLastError();
}

cudaError_t set_smem_limits() {
    cudaError_t e = allow_square();
    if (e == cudaSuccess) e = allow_cubic();
    if (e == cudaSuccess) e = allow_cubic_long();
    return e;
}

cudaError_t launch_grow(const RunDev &P, int thresh_mode, bool key64, int ctas, cudaStream_t stream) {
    if (P.d == 2) return launch_square(P, thresh_mode, ctas, stream);
    return key64 ? launch_cubic_long(P, thresh_mode, ctas, stream) : launch_cubic(P, thresh_mode, ctas, stream);
}

cudaError_t launch_counts(unsigned long long *Sn, int L, cudaStream_t stream) {
    counts_kernel<<<1, 1024, 0, stream>>>(Sn, L);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const RunDev &P, cudaStream_t stream) {
    finalize_kernel<<<1, P.parts > 1 ? 256 : 32, 0, stream>>>(P);
    return cudaGetLastError();
}

template <int D, bool REFINE>
static cudaError_t debug_step_form(int n_max, int B, const int32_t *coords, const int32_t *len, const double *W,
                                   const double *Wsum, const uint64_t *M, const uint64_t *ordinal,
                                   const uint32_t *seq, const uint32_t *tour, uint32_t key0, uint32_t key1,
                                   int force_exact, int32_t *out_i, double *out_r, double *out_w, cudaStream_t stream) {
    int log2h = 4;
    while ((1 << log2h) < 2 * n_max) ++log2h;
    const int per = walks_per_warp_max(D);               // states per block of one warp
    const int blocks = (B + per - 1) / per;
    const size_t smem = 1024 + walk_hash_bytes(log2h, 4) * (size_t)per;
    const cudaError_t e = cudaFuncSetAttribute(debug_step_kernel<D, uint32_t, REFINE>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    debug_step_kernel<D, uint32_t, REFINE><<<blocks, 32, smem, stream>>>(n_max, log2h, B, coords, len, W, Wsum,
            M, ordinal, seq, tour, key0, key1, force_exact, out_i, out_r, out_w);
    return cudaGetLastError();
}

cudaError_t launch_debug_step(int d, int n_max, int B, const int32_t *coords, const int32_t *len,
                              const double *W, const double *Wsum, const uint64_t *M,
                              const uint64_t *ordinal, const uint32_t *seq, const uint32_t *tour,
                              uint32_t key0, uint32_t key1, bool snapshot, int force_exact, int32_t *out_i,
                              double *out_r, double *out_w, cudaStream_t stream) {
    if (B <= 0) return cudaSuccess;
    const auto form = d == 2 ? (snapshot ? debug_step_form<2, false> : debug_step_form<2, true>)
                             : (snapshot ? debug_step_form<3, false> : debug_step_form<3, true>);
    return form(n_max, B, coords, len, W, Wsum, M, ordinal, seq, tour, key0, key1, force_exact, out_i, out_r,
                out_w, stream);
}

cudaError_t launch_debug_philox(int B, const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out,
                                cudaStream_t stream) {
    if (B <= 0) return cudaSuccess;
    philox_kernel<<<(B + 127) / 128, 128, 0, stream>>>(B, ctr, k0, k1, out);
    return cudaGetLastError();
}

}  // namespace perm
