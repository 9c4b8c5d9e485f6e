// perm_grow.cuh -- persistent flatPERM growth kernel (Algorithms 1 and 2 of
// Campbell and Janse van Rensburg, "Parallel PERM", Sec. 3) for sm_103a.
//
// A group of lanes grows one walk ("slot"): 4 lanes on the square lattice, 8 on the
// cubic one, so a warp holds up to 8 or 4 walks.  Every lane of a group carries the
// walk's state; lane j probes neighbour j, deletes every 4th (8th) site of a
// backtrack, and issues one of the node's table updates.  Per walk, shared memory
// holds the occupancy hash (buckets of 4 keys, keys deleted in LIFO order on
// backtrack), the hash slot of every site, and the top of the stack of waiting
// copies (the rest spills to global memory).  Each walk runs the tours handed to
// it one after another; a tour is a depth-first traversal of the tree of copies
// made by enrichment (Sec. 2).
//
// What bounds it: the walks are few (one per sequence; an SM's shared memory and
// registers hold at most 88), so the dependent instruction streams of 9 to 11 warps set
// the rate (an SM issues on 39 % of its cycles at 9 warps), not memory or arithmetic.  On
// this part a lone warp pays 25 cycles or more for a branch, 45 for a vote and a branch on
// it, 20-60 for a reduction, 33 for a shared-memory load, 64 for every double-precision
// instruction whatever its active lanes (measured, one warp).  One lane per walk ran all
// four (six) probes, the table updates and a dozen branches of a node one after another,
// 7 walks to a warp; a group of lanes does them side by side, and the node is one straight
// line.  GB300, one lane per walk -> the first form of a group -> now: 12 walks to n = 16,
// 24 000 tours 48.5 -> 31.5 -> 22.9 ms; square n = 512, 4096 sequences, 96 tours each of a
// continued run 193 -> 126 -> 49.5 ms, 256 tours from empty tables 561 -> 302 -> 164 ms;
// cubic n = 512, 8192 sequences, 128 tours 491 -> 253 -> 119 ms.
//
// Threshold sources for Algorithm 2 (one shared table W, Fig. 1):
//  - snapshot: every node adds its weight to the global table with a
//    reduction that returns nothing (S_n, the nodes of length n, is kept as its
//    differences along n: +1 where a walk started or resumed, -1 past its leaf,
//    one reduction a leaf); one extra warp per CTA reloads a
//    shared-memory copy of W_n and M every refresh period.  The nodes read
//    that copy (a stale but fixed threshold keeps the estimator unbiased:
//    enrichment and pruning conserve the expected weight for any r).  Walks
//    with no tour to start grow waiting copies of other walks' tours (shared
//    copies).
//  - fresh: every node adds its weight to the global table with an atomic that
//    returns the previous sum, and uses it at once (sequential flatPERM exactly
//    when one walk runs).
// Algorithm 1 (private tables) always uses the fresh form on its own rows.  The
// per-tour sums X_n go to a global row per walk and, squared, into Q_n when the
// tour ends.  With cut-offs set (original PERM, Sec. 2) r comes from the
// cut-offs instead of the table.  perm_kernels.cu holds the batch kernel, which
// grows many runs in one persistent launch with the same per-run body; perm_grow_*.cu the
// instances of the growth kernel, a file each so that they compile side by side.
#pragma once

#include <cstdio>

#include "perm_device.cuh"
#include "perm_kernels.cuh"
#include "perm_parts.h"

namespace perm {

namespace {

constexpr int kUnwind = 4;         // hash deletions per lane per iteration (16 or 32 per walk)
// Extra tour tickets fetched per warp.  M counts them as started, so few where a thousand
// warps hold them; a few walks (12 walks to n = 16: 24.1 -> 23.0 ms) fetch more at a time, as far
// as the tours left go round (tickets_ahead; 12 sequences to n = 512, 4 tours each without shared
// copies: square 0.38 -> 0.33 us a node, cubic 0.31 -> 0.26; bounding the many walks' two as
// well took 4096 sequences, 1 tour each, from 2.44 to 2.59 ms).
constexpr int kPoolExtra = 2, kPoolExtraFew = 8, kFewWalks = 64;
constexpr int kChunk = 8;          // stack records moved per spill or fill (ring >= 2 kChunk)
constexpr int kReloadBatch = 8;    // snapshot entries a refresher lane loads before storing them
constexpr unsigned kRowFree = 0xFFFFFFFFu;   // outst: the walk's tour-sum row is unused
constexpr int kMinShareGap = 8;    // share a waiting copy only if it may still grow this many steps
constexpr int kCellSpin = 1 << 20; // bounded wait for a donation cell being written
constexpr unsigned kFull = 0xFFFFFFFFu;

enum LaneState { kNeed = 0, kNode = 1, kUnwindState = 2, kFlush = 3, kDone = 4 };
// What a run asks of the growth kernel besides flatPERM.
enum Form { kPlain = 0, kWatched = 1, kCutoffs = 2 };
enum Outcome { kLeafNmax = 0, kTrapped = 1, kPruned = 2, kChildren = 3 };

struct CtaHead {
    unsigned long long Ms;   // tours started, as of the last snapshot
    int done_warps;
    int want_don;            // copies this CTA may still hand to idle walks this period
    int queued;              // shared copies waiting in the ring, as of the last snapshot
    int status;              // run status, as of the last snapshot
    unsigned long long fin;  // tours finished, as of the last snapshot
    int cap;                 // parts of one tour that may grow at once (shared copies)
    int may_leave;           // batch launch: another run still has tours to start
    int stalled;             // no tour of the run has finished for stall_ns
    int pad[5];
};
static_assert(sizeof(CtaHead) == 64, "header size");

__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// A load of a table entry that other SMs update with atomics: an aligned 8-byte
// load is single-copy atomic; relaxed at GPU scope, so the loads of one batch
// stay in flight together.
__device__ __forceinline__ double ld_relaxed(const double *p) {
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ void set_status(int *status, int code) {
    atomicCAS(status, 0, code);
}

__device__ __forceinline__ size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

// A walk's region: hash, site list, stack ring (records, then their weights).
__host__ __device__ __forceinline__ size_t walk_hash_bytes(int log2h, size_t key_bytes) {
    return ((size_t)1 << log2h) * key_bytes;              // a multiple of 16: 2^4 slots or more
}
__host__ __device__ __forceinline__ size_t walk_sites_bytes(int n_max) { return ((size_t)n_max * 2 + 15) & ~(size_t)15; }
__host__ __device__ __forceinline__ size_t walk_region_bytes(int n_max, int log2h, int K, size_t key_bytes) {
    return walk_hash_bytes(log2h, key_bytes) + walk_sites_bytes(n_max) + (size_t)K * 12;
}

__host__ __device__ __forceinline__ size_t head_region_bytes(int n_max, bool snapshot) {
    const size_t L = (size_t)n_max + 1;
    size_t b = 64 + 1024;         // header + constants (fill_constants)
    if (snapshot) b += 8 * L;     // the snapshot of W_n
    return (b + 15) & ~(size_t)15;
}

// The constants of a CTA's head region: weight factors for the two scale steps dE of
// the lattice (t: dE = dE_lo + t), [t*48 + (a-1)*8 + c] = (a/c) 2^-dE for c >= 1
// (enrichment), c = 0: a 2^-dE (exact); and after the 96 factors the free list of
// every free mask (directions in order, 3 bits each).
constexpr int kFactors = 96;
__device__ void fill_constants(double *aoc, int d, int tid, int nthreads) {
    const int dE_lo = (d == 2) ? 1 : 2;
    for (int i = tid; i < kFactors; i += nthreads) {
        const int t = i / 48, a = (i % 48) / 8 + 1, c = i & 7;
        const double s = __longlong_as_double((long long)((unsigned long long)(1023 - dE_lo - t) << 52));
        aoc[i] = c >= 1 ? __dmul_rn(__ddiv_rn((double)a, (double)c), s) : __dmul_rn((double)a, s);
    }
    uint32_t *lists = reinterpret_cast<uint32_t *>(aoc + kFactors);
    for (int m = tid; m < 64; m += nthreads) {
        uint32_t list = 0u;
        int cnt = 0;
        for (int j = 0; j < 6; ++j)
            if (m >> j & 1) { list |= (uint32_t)j << (3 * cnt); ++cnt; }
        lists[m] = list;
    }
}

// E(n+1) - E(n) - dE_lo: which of the lattice's two scale steps length n takes.
template <int D>
__device__ __forceinline__ int scale_row(int n) {
    return D == 2 ? (((3 * n) & 7) + 3) >> 3 : ((n & 3) + 1) >> 2;
}

// Original PERM's cut-offs (Sec. 2) as a node reads them: per length (T_n, t_n)
// at the stored scale, the copies made above T_n, and below t_n the survival
// threshold K (survive iff w0 < K, i.e. u0 < 1/q) and the factor q.
struct Cutoffs {
    const longlong2 *cut;      // bit patterns
    int copies;
    double q, inv_q;
    unsigned long long K;
};

// What the nodes of a walk compute from M, the tours started: once per tour and
// snapshot (a double-precision division takes as long as a node).
struct Tours {
    unsigned long long M;
    double Md;                 // M rounded to double
    float Mf;                  // tours_float(M)
    double inv1, inv3, inv5;   // 1/M rounded to double, and 3 and 5 times that
};
template <bool RATIOS>         // (with cut-offs a node needs M for its trace only)
__device__ __forceinline__ void set_tours(Tours &t, unsigned long long M) {
    t.M = M;
    if (!RATIOS) return;
    t.Md = __ull2double_rn(M);
    t.Mf = tours_float(M);
    t.inv1 = __drcp_rn(t.Md);
    t.inv3 = __dmul_rn(3.0, t.inv1);
    t.inv5 = __dmul_rn(5.0, t.inv1);
}

// The running average sum / M, correctly rounded: q = sum (1/M) and one correction by its
// remainder with the correctly rounded 1/M (P. Markstein, "Computation of elementary functions
// on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34 (1990) 111-119), where M is
// below 2^32 and the sum far from the range's ends; else the division itself.  (q is within
// 1.5 units in the last place, so the remainder sum - q M, a multiple of q's last place below
// 2^33 of them, is exact; the corrected value is then within 2^-52 units of the quotient,
// which lies 2^-33 units or more from a midpoint between two doubles.)
__device__ __forceinline__ double average(double sum, const Tours &t) {
    const double q = __dmul_rn(sum, t.inv1);
    double avg = __fma_rn(__fma_rn(-q, t.Md, sum), t.inv1, q);
    const int es = __double2hiint(sum) >> 20;
    if (t.Mf < 0.0f || es < 128 || es > 1920) avg = __ddiv_rn(sum, t.Md);
    return avg;
}

struct Decision {
    int c;               // copies (0: pruned)
    bool exact;          // the decision was taken on r in double precision
    float x;             // the estimate of r, and r itself where it was evaluated
    double r;            // (cut-offs: in both forms what the cut-off stands for)
    double child_w;
};
// r as the decision used it.
__device__ __forceinline__ double decision_r(const Decision &o, int n, bool cutoffs) {
    return o.exact || cutoffs ? o.r : (n == 0 ? 1.0 : widen(o.x));
}

// r exactly as defined and the decision on it.  avg: the running average (Wsum + W)/M,
// correctly rounded.
__device__ __forceinline__ Decision decide_on_average(int a, double W, double avg, uint32_t w0, double a_sc) {
    Decision o;
    bool surv = false;
    o.exact = true;
    o.x = 0.0f;
    if (avg == W && W > 0.0) {
        // r = 1 exactly (of a lone sequence at every n <= 3, where every weight is the same)
        o.r = 1.0;
        o.c = 1;
        o.child_w = __dmul_rn(W, a_sc);
        return o;
    }
    o.r = __ddiv_rn(W, avg);
    o.c = decide_exact(o.r, a, w0, surv);
    if (surv) o.child_w = __dmul_rn(__dmul_rn(W, __ddiv_rn(1.0, o.r)), a_sc);
    else o.child_w = o.c > 1 ? __dmul_rn(__ddiv_rn(W, (double)o.c), a_sc) : __dmul_rn(W, a_sc);
    return o;
}
// Snapshot form: one node in 10^4 or fewer, out of line (inline it costs the other nodes
// 5 %, by their registers).
__device__ __noinline__ Decision decide_node_exact(int a, double W, double sum, unsigned long long M, uint32_t w0,
                                                   double a_sc) {
    return decide_on_average(a, W, __ddiv_rn(sum, __ull2double_rn(M)), w0, a_sc);
}

// A survivor's weight where M is its tour's own number: the quotient by M correctly rounded.
__device__ __noinline__ double divided_survivor(double sum, unsigned long long M, double a_sc) {
    return __dmul_rn(__ddiv_rn(sum, __ull2double_rn(M)), a_sc);
}

// The decision at a node with a >= 1 free neighbours (Sec. 2): r, the copies, the
// children's weight.  sum: the weights recorded at length n up to this node, gs: what
// the estimate of r says; refine: round the survivor's quotient by M correctly (one correction
// by its remainder); divide: the snapshot form's M is not the snapshot's, and a survivor's quotient is
// divided out (a tour's first nodes, until the snapshot counts it).  valid: the lane has a node to decide (the others' results are not used);
// force_exact: decide on the double-precision r.  Shared by the persistent kernel
// and the snapshot-state kernel; every lane of a walk's group takes the same decision.
// One straight line with selects but for the exact path: a branch costs a lone warp
// 25 cycles or more, a double-precision instruction 64 whatever its active lanes.
template <int D>
__device__ __forceinline__ Decision decide_node(int n, int a, double W, double sum, const Guess &gs, const Tours &t,
                                                bool refine, bool divide, uint32_t w0, const double *aoc, bool valid, bool force_exact) {
    Decision o;
    o.exact = false;
    o.x = gs.x;
    o.r = 0.0;
    const int dE = scale_row<D>(n) + (D == 2 ? 1 : 2);
    const double *row = aoc + 48 * (dE - (D == 2 ? 1 : 2)) + 8 * (a - 1);
    const bool surv = !gs.up && gs.c > 0 && n != 0;
    const int c = n == 0 ? 1 : (gs.c < a ? gs.c : a);    // r = 1 at the empty walk
    const bool exact = valid && n != 0 && (gs.open || (gs.near_k && gs.k <= a) || force_exact);
    // a survivor carries W/r = [W_n]^sample = (Wsum + W)/M, a child of an enrichment
    // (W/c) a_+ 2^-dE: one double-precision product for both, on the critical path
    // alone.  The survivor's factor (1/M) a_+ 2^-dE (a node past the empty walk has
    // a_+ <= 5) is one of three products kept per M, its exponent shifted (exact: 1/M
    // is far from the subnormals); the weight is within 2^-51 of the quotient.  That holds for the
    // snapshot's M; with the tour's own number the quotient is divided out below, beside the exact
    // path (in one branch with it: under 1 %)
    double base = W, fac = row[c];
    if (refine) {
        // the quotient as average() forms it (past M = 2^32 it may be a unit in the last place
        // off).  (Under a branch: three dependent operations of 62 cycles, which ran no faster
        // beside the probes)
        if (surv) {
            const double q = __dmul_rn(sum, t.inv1);
            base = __fma_rn(__fma_rn(-q, t.Md, sum), t.inv1, q);
            fac = row[0];
        }
    } else {
        const double f0 = a == 3 ? t.inv3 : (D == 3 && a == 5 ? t.inv5 : t.inv1);
        const int sh = (a == 2 ? 1 : (a == 4 ? 2 : 0)) - dE;
        const double fs = __hiloint2double(__double2hiint(f0) + (sh << 20), __double2loint(f0));
        base = surv ? sum : W;
        fac = surv ? fs : fac;
    }
    o.child_w = __dmul_rn(base, fac);
    o.c = c;
    // the estimate cannot settle a comparison: r exactly as defined
    if (exact && refine) {
        o = decide_on_average(a, W, average(sum, t), w0, row[0]);
    } else if (!refine && (exact || (valid && surv && divide))) {
        if (exact) o = decide_node_exact(a, W, sum, t.M, w0, row[0]);
        else o.child_w = divided_survivor(sum, t.M, row[0]);
    }
    return o;
}

// Original PERM's decision (Sec. 2, cut-offs T_n, t_n): copies above T_n, survival with
// probability 1/q (weight times q) below t_n, one copy between them and at the empty
// walk.
template <int D>
__device__ __forceinline__ Decision decide_cutoffs(int n, int a, double W, longlong2 tc, uint32_t w0,
                                                   const double *aoc, const Cutoffs &cuts) {
    Decision o;
    const double *row = aoc + 48 * scale_row<D>(n) + 8 * (a - 1);
    o.exact = false;
    o.x = 0.0f;
    // the cut-offs' bit patterns: a weight is not negative and the library keeps no NaN and
    // no -0.0 among them, so the patterns compare as the numbers do (a double-precision
    // comparison takes 50 cycles)
    const long long wb = __double_as_longlong(W);
    const bool above = wb > tc.x && n > 0, below = wb < tc.y && n > 0;      // the empty walk: one copy
    o.c = above ? (cuts.copies < a ? cuts.copies : a) : (below && !((unsigned long long)w0 < cuts.K) ? 0 : 1);
    o.r = above ? (double)cuts.copies : (below ? cuts.inv_q : 1.0);
    o.child_w = __dmul_rn(below && !above ? __dmul_rn(W, cuts.q) : W, row[above ? o.c : 0]);
    return o;
}

// A reduction into global memory by the lanes that take part, without a branch around it
// (the compiler's costs a lone warp 40 cycles, the predicated instruction 20).
__device__ __forceinline__ void red_add(double *p, double v, bool take) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %2, 0;\n@q red.relaxed.gpu.global.add.f64 [%0], %1;\n}"
                 :: "l"(p), "d"(v), "r"((int)take) : "memory");
}
__device__ __forceinline__ void red_count(unsigned long long *p, long long v, bool take) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %2, 0;\n@q red.relaxed.gpu.global.add.u64 [%0], %1;\n}"
                 :: "l"(p), "l"(v), "r"((int)take) : "memory");
}

// A tour-sum row as its parts' ends see it (end_part).
struct PartsRow {
    unsigned int *tmaxn, *outst;
    __device__ __forceinline__ void deepen(unsigned n) { atomicMax(tmaxn, n); }
    __device__ __forceinline__ unsigned leave() { return atomicSub(outst, 1u); }
    __device__ __forceinline__ unsigned depth() { return *(volatile unsigned int *)tmaxn; }
    __device__ __forceinline__ void fence() { __threadfence(); }
};

// The whole warp copies a donor's sites 0..bdp (key and hash slot) into a cell.
template <typename Key>
__device__ __noinline__ void copy_sites_to_cell(const Key *hash, const uint16_t *sites, int bdp, Key *ck, uint16_t *cs,
                                                int lane) {
    for (int k = lane; k <= bdp; k += 32) {
        const uint16_t sl = sites[k];
        ck[k] = hash[sl];
        cs[k] = sl;
    }
}

// The whole warp places a taker's sites 0..dp from a cell at their hash slots.
template <typename Key>
__device__ __noinline__ void place_sites_from_cell(Key *hash, uint16_t *sites, int dp, const Key *ck, const uint16_t *cs,
                                                   int lane) {
    for (int k = lane; k <= dp; k += 32) {
        const uint16_t sl = __ldcg(cs + k);
        hash[sl] = __ldcg(ck + k);
        sites[k] = sl;
    }
}

// ---------------------------------------------------------------------------
// The persistent growth kernel.
// ---------------------------------------------------------------------------
// What lets a CTA leave a run before every tour of the run has finished: in a
// batch launch, another run still has walks to grant and tours to start
// (runs_open > 0).  The first walk to find a run's tickets exhausted marks it
// closed (bit 0 of its flag; bit 1: all its walks granted); the first of those two
// marks takes the run off runs_open.  Bit 2 of the flag says that no tour of the run has
// finished for a while (its CTAs' refreshers set and clear it): such a run
// draws helper CTAs before other unfinished runs do.
struct BatchLeave {
    int *runs_open;
    int *closed;
    const int *ctas_on_run;   // CTAs growing this run now
    bool helper;              // this CTA's walks take waiting copies only
};
constexpr int kStalledBit = 4;

// The growth of one run by one CTA (Secs. 1-3): the refresher warp and the walk
// warps.  A single-run launch calls it once (bl == nullptr: the CTA stays until
// the run is complete); a batch launch calls it for each run a CTA joins.
// SHARED: every region is in shared memory (no arena), known at compile time, so
// that the walks' hashes, site lists and stacks are reached by shared-memory
// instructions rather than generic ones (a generic load that lands in shared
// memory waits longer, and in the long-scoreboard queue).
// Admission (Algorithm 2): tours in flight stay at most c0 + gamma * finished, i.e.
// tickets at most c0 + f + gamma f.  admit[0] counts the admitted tours not yet taken
// (c0 apart), admit[1] is the f + gamma f that went into it.  A warp takes what it
// wants from the count and gives back what was not there; one that comes short brings
// the count up to date with f.  `again`: the warp asks for walks that waited already,
// so the count may be short: it looks before it takes (a thousand idle warps taking and
// giving back would hide the few admitted tours from each other).  No retries: with a
// compare-and-swap on the tickets a thousand warps got 3 grants per microsecond
// together, and short tours waited for them (square n = 16, 4096 sequences, 40 tours
// each: 27 ms, now 3.4).
__device__ unsigned long long admitted(const RunDev &P, unsigned long long want, bool again) {
    unsigned long long *left = reinterpret_cast<unsigned long long *>(P.admit);
    for (int attempt = 0; attempt < 2; ++attempt) {
        const long long k = (long long)want;
        if (!again || (long long)*(volatile unsigned long long *)left + P.ramp_c0 > 0) {
            const long long had = (long long)atomicAdd(left, 0ull - want) + P.ramp_c0;
            const long long got = had < 0 ? 0 : (had < k ? had : k);
            if (got < k) atomicAdd(left, (unsigned long long)(k - got));
            if (got > 0) return (unsigned long long)got;
        }
        if (attempt > 0) break;
        const unsigned long long f = *(volatile unsigned long long *)P.finished;
        const unsigned long long now = f + ((f * P.ramp_gamma_q16) >> 16);
        const unsigned long long was = atomicMax(left + 1, now);
        if (now <= was) break;
        atomicAdd(left, now - was);
    }
    return 0ull;
}

template <int D> constexpr int kGroupLanes = D == 2 ? 4 : 8;   // lanes that hold one walk

// FORM: flatPERM alone (kPlain), flatPERM with observables or a trace (kWatched: the
// node is 4-6 % slower for their registers and the length of the loop), or the original
// PERM's cut-offs, with either (kCutoffs: no ratio, and no M).
template <int D, typename Key, int MODE, bool SHARED, int FORM>
__device__ __forceinline__ void grow_run(const RunDev &P, unsigned char *smem, const BatchLeave *bl,
                                         int cta_walks) {
    constexpr int G = kGroupLanes<D>;
    const int L = P.n_max + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool snapshot = (MODE == kSnapshot);
    const int K = P.stack_cache;

    // The CTA's state: the head region (header, constant tables, snapshot of W_n)
    // and one region per walk (occupancy hash, site list, stack ring).  Both sit in
    // shared memory, or, for walks too long for it, the walk regions (and, if even
    // the head does not fit, the head too) in this CTA's slice of a global arena,
    // served through L1 and L2.  A walk's data is touched by its own warp only, and
    // the lanes of the warp order their accesses by __syncwarp(), so the same code
    // runs on either.
    const size_t hbytes = head_region_bytes(P.n_max, snapshot);
    const size_t wbytes = walk_region_bytes(P.n_max, P.log2h, K, sizeof(Key));
    unsigned char *hbase = smem, *wbase = smem + hbytes;
    if (!SHARED && P.arena_mode != kArenaNone) {
        unsigned char *a = P.arena + (size_t)blockIdx.x * (size_t)P.arena_cta_bytes;
        if (P.arena_mode == kArenaAll) { hbase = a; wbase = a + hbytes; }
        else wbase = a;
    }
    CtaHead *head = reinterpret_cast<CtaHead *>(hbase);
    double *aoc = reinterpret_cast<double *>(hbase + 64);
    const uint32_t *lists = reinterpret_cast<const uint32_t *>(aoc + kFactors);
    double *Wsnap = snapshot ? reinterpret_cast<double *>(hbase + 64 + 1024) : nullptr;

    // zero everything (empty hashes, empty stacks), then the constant tables
    for (size_t i = threadIdx.x; i < hbytes / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(hbase)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = threadIdx.x; i < wbytes * (size_t)(P.S * P.worker_warps) / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(wbase)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (P.arena_mode != kArenaNone) __threadfence_block();
    __syncthreads();
    fill_constants(aoc, D, threadIdx.x, blockDim.x);
    const long long limit = P.tour_limit;
    if (snapshot) {
        for (int k = threadIdx.x; k < L; k += blockDim.x) {
            double v = *(volatile double *)(P.Wn + k);
            for (int q = 1; q < P.parts; ++q)
                v = __dadd_rn(v, *(volatile double *)(P.Wp + (size_t)(q - 1) * (size_t)P.part_stride + k));
            Wsnap[k] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long Ms = *(volatile unsigned long long *)P.tickets;     // after the sums, as below
            if ((long long)Ms > limit) Ms = (unsigned long long)limit;
            head->Ms = Ms;
        }
    }
    __syncthreads();

    // ----------------------------------------------------------------------
    // refresher warp (snapshot form): reload the snapshot of W_n and M
    // ----------------------------------------------------------------------
    if (snapshot && warp == P.worker_warps) {
        const long long t0 = global_ns();
        unsigned long long last_fin = *(volatile unsigned long long *)P.finished;
        long long t_change = t0;
        bool boosted = false;
        if (lane == 0) *(volatile int *)&head->cap = P.share;
        for (long long it = 0;; ++it) {
            const long long c_it = clock64();
            const int done = __shfl_sync(kFull, *(volatile int *)&head->done_warps, 0);
            __threadfence_block();
            if (done >= P.worker_warps) {
                if (lane == 0) atomicAdd(P.refreshes, (unsigned long long)it);
                break;
            }
            unsigned long long Ms = 0ull;
            for (int k0 = 0; k0 < L; k0 += 32 * kReloadBatch) {
                double v[kReloadBatch];
#pragma unroll
                for (int j = 0; j < kReloadBatch; ++j) {
                    const int k = k0 + j * 32 + lane;
                    v[j] = k < L ? ld_relaxed(P.Wn + k) : 0.0;
                }
                for (int q = 1; q < P.parts; ++q) {
                    const double *Wq = P.Wp + (size_t)(q - 1) * (size_t)P.part_stride;
                    double u[kReloadBatch];
#pragma unroll
                    for (int j = 0; j < kReloadBatch; ++j) {
                        const int k = k0 + j * 32 + lane;
                        u[j] = k < L ? ld_relaxed(Wq + k) : 0.0;
                    }
#pragma unroll
                    for (int j = 0; j < kReloadBatch; ++j) v[j] = __dadd_rn(v[j], u[j]);
                }
                if (k0 == 0) {
                    // M read after the sums of the shortest lengths and published before them, so
                    // that M counts every tour whose weights a node finds in them: with M older
                    // than the sums r falls below 1 at n = 1, where every tour has the same
                    // weight, and prunes some (the only way that c_2 can get an error at all)
                    __threadfence();
                    Ms = *(volatile unsigned long long *)P.tickets;
                    if ((long long)Ms > limit) Ms = (unsigned long long)limit;
                    Ms = __shfl_sync(kFull, Ms, 0);
                    if (lane == 0) *(volatile unsigned long long *)&head->Ms = Ms;
                    __threadfence_block();
                    __syncwarp();
                }
#pragma unroll
                for (int j = 0; j < kReloadBatch; ++j) {
                    const int k = k0 + j * 32 + lane;
                    if (k < L) *(volatile double *)&Wsnap[k] = v[j];
                }
            }
            if (P.share && lane == 0) {
                // idle walks not yet served by a queued copy, split over the CTAs
                const long long hg = *(volatile int *)P.hungry;
                long long q = (long long)(*(volatile unsigned long long *)P.dq_tail -
                                          *(volatile unsigned long long *)P.dq_head);
                q = q < 0 ? 0 : (q > (1 << 30) ? (1 << 30) : q);
                const long long want = hg - q;
                const long long nct = bl != nullptr ? (long long)max(1, *(volatile const int *)bl->ctas_on_run)
                                                    : (long long)gridDim.x;
                const long long per = want > 0 ? (want + nct - 1) / nct : 0;
                *(volatile int *)&head->want_don = (int)(per < (1 << 20) ? per : (1 << 20));
                *(volatile int *)&head->queued = (int)q;
                *(volatile int *)&head->status = *(volatile int *)P.status;
                *(volatile int *)&head->may_leave = (bl != nullptr && *(volatile int *)bl->runs_open > 0) ? 1 : 0;
                const unsigned long long fin_now = *(volatile unsigned long long *)P.finished;
                *(volatile unsigned long long *)&head->fin = fin_now;
                // a run whose tours stop finishing is growing a start-up tree far
                // larger than its walks can grow a few parts at a time: let its
                // tours spread over every idle walk from then on
                const long long now = global_ns();
                if (fin_now != last_fin) { last_fin = fin_now; t_change = now; }
                // and so does a run's end: no tour is left to start, and at most one in eight of
                // the run's tours is not finished, so the table has samples at the lengths that
                // the parts reach, and spreading makes no larger trees
                const bool tail = (long long)Ms >= limit && (long long)fin_now >= limit - limit / 8;
                if (now - t_change > P.stall_ns) boosted = true;
                *(volatile int *)&head->cap = boosted || tail ? P.share_boost : P.share;
                const int st_now = (now - t_change > P.stall_ns) ? 1 : 0;
                if (st_now != *(volatile int *)&head->stalled) {
                    *(volatile int *)&head->stalled = st_now;
                    if (bl != nullptr) {
                        if (st_now) atomicOr(bl->closed + P.run_index, kStalledBit);
                        else atomicAnd(bl->closed + P.run_index, ~kStalledBit);
                    }
                }
            }
            __syncwarp();
            // one reload per refresh period, paced on the SM's cycle counter at two
            // cycles per ns (the 2 GHz SM clock): one __nanosleep may end well before
            // or after the time it is given
            for (int nap = 0; nap < 256; ++nap) {
                const long long left = __shfl_sync(kFull, (c_it + 2ll * P.refresh_ns - clock64()) >> 1, 0);
                if (left <= 0) break;
                __nanosleep((unsigned)(left < 1000 ? left : 1000));
            }
            const bool late = (it & 15) == 0 && global_ns() - t0 > P.max_ns;
            if (__any_sync(kFull, late)) {
                if (lane == 0) set_status(P.status, PERM_ETIMEOUT);
                break;
            }
        }
    } else if (warp < P.worker_warps) {

    // ----------------------------------------------------------------------
    // worker warps
    // ----------------------------------------------------------------------
    const int grp = lane / G, j = lane % G, lead = lane - j;   // group, direction, the group's first lane
    const bool first = j == 0;
    const unsigned lt_mask = (1u << lead) - 1u;
    const int gwarp = blockIdx.x * P.worker_warps + warp;
    const int slot = gwarp * P.S + grp;
    const bool active = grp < P.S && slot < P.slots && warp * P.S + grp < cta_walks;
    const int sidx = active ? slot : 0;
    const size_t hash_b = walk_hash_bytes(P.log2h, sizeof(Key)), sites_b = walk_sites_bytes(P.n_max);
    // (the lanes of a group without a walk read the warp's first one and write nothing)
    unsigned char *warp_base = wbase + wbytes * (size_t)(warp * P.S);
    unsigned char *wb = warp_base + wbytes * (size_t)(grp < P.S ? grp : 0);
    Key *hash = reinterpret_cast<Key *>(wb);
    uint16_t *sites = reinterpret_cast<uint16_t *>(wb + hash_b);
    uint32_t *smeta = reinterpret_cast<uint32_t *>(wb + hash_b + sites_b);
    double *sw = reinterpret_cast<double *>(wb + hash_b + sites_b + (size_t)K * 4);
    const int log2b = P.log2h - Buckets<Key>::kLog2;
    const Key origin = KeyCodec<D, Key>::encode(0, 0, 0);
    const Key dkey = step_key<D, Key>(j < 2 * D ? j : 0);

    uint32_t *gmeta = P.gstk_meta + (size_t)sidx * P.n_max;
    double *gwt = P.gstk_w + (size_t)sidx * P.n_max;
    const Cutoffs cuts{reinterpret_cast<const longlong2 *>(P.cut), P.cut_copies, P.cut_q, P.cut_inv_q, P.cut_K};
    constexpr bool cutoffs = FORM == kCutoffs;

    // the walk's state: the same in every lane of its group
    int state = active ? kNeed : kDone;
    int n = 0, maxn = 0;
    int seg = 0;               // length at which the walk started or last resumed
    Key cur = origin;          // key of the end-point
    double W = 1.0;
    uint32_t ord = 0u;         // nodes of this part so far; a node's 64-bit ordinal is did 2^32 + ord
    unsigned long long g = 0ull;
    // the random blocks of the G nodes from ordinal pbase on: lane j holds the first two
    // words of node pbase + j's (a block a pass for every lane would be G times the work)
    uint32_t pbase = (uint32_t)-G, pw0 = 0u, pw1 = 0u;
    uint32_t seq = 0u, tour = 0u;
    int top = 0, sbase = 0;
    int un_lo = 0, un_hi = -1, pend_dir = 0, pend_depth = 0;
    double pend_w = 0.0;
    unsigned long long my_steps = 0ull, my_copies = 0ull, my_exact = 0ull;
    int my_max_stack = 0;
    int cur_seq = -1;
    long long seq_t = 0;
    unsigned long long pool_lo = 0ull, pool_hi = 0ull;
    bool waiting = false;
    // tour-sum rows: with shared copies a walk has two, so that it can start its
    // next tour while parts of its last one still grow on other walks
    const int rows_per_walk = P.share ? 2 : 1;
    int myrow = sidx * rows_per_walk;
    // shared copies: the walk grows either its own tour or a part of another
    // walk's tour (own = that tour's row, did = the part's donation id)
    int own = myrow, bot = 0;
    uint32_t did = 0u;
    bool donated = false;      // a part of this walk's own tour went to another walk
    bool xbusy = false;        // every tour-sum row of this walk is still used by such parts
    // no tour tickets left; a helper (of a batch, or a walk beyond the run's tour walks)
    // takes none and grows waiting copies only
    bool exhausted = (bl != nullptr && bl->helper) || sidx >= P.tour_slots;
    int my_hungry = 0;         // this warp's share of P.hungry
    unsigned idle_ns = 500u;   // back-off of a warp with nothing to grow
    const uint32_t dq_mask = (1u << P.dq_log2cap) - 1u;
    // a donation cell: 32-byte header, the keys of sites 0..n_max, then their slots
    const size_t cell_key_bytes = align16(((size_t)P.n_max + 1) * sizeof(Key));
    unsigned long long my_iters = 0ull;
    Tours tours;               // tours started as this walk's nodes see them
    set_tours<!cutoffs>(tours, 1ull);
    uint32_t ms_low = 0u;      // the low word of the snapshot's M as last taken
    bool fresh_need = true;    // the walk has ended its tour since it last looked for work
    // this CTA's copies of the tables (parts: a table of a kilobyte sits in one slice of L2,
    // which adds 2.9e9 doubles a second whoever sends them)
    const int part = snapshot && P.parts > 1 ? (int)(blockIdx.x % (unsigned)P.parts) : 0;
    double *Wrow = part > 0 ? P.Wp + (size_t)(part - 1) * (size_t)P.part_stride : P.Wn;
    double *Qtab = part > 0 ? P.Qp + (size_t)(part - 1) * (size_t)P.part_stride : P.Qn;
    unsigned long long *Srow = P.Sn;
    double *Rrow = P.Rn;
    double *acc = Wrow;        // the row this lane adds a node's weight to (lane 0: W_n, lane 1: the tour's sums)

    const bool extras = FORM != kPlain && (P.Rn != nullptr || P.trace != nullptr);
    // fresh form: this walk alone reads and writes the table row of its tours (Algorithm 1:
    // one row per sequence, one walk per sequence at a time; else a run of one walk, whose
    // tickets it alone takes, so that M is its own tour's number)
    const bool own_rows = !snapshot && (P.alg == PERM_ALG1 || P.slots == 1);
    // start tour g at the empty walk (Sec. 1: W(empty) = 1); the walk's hash is empty, so
    // the origin takes the first place of its home bucket
    auto start_tour = [&]() {
        if (P.alg == PERM_ALG1) {
            seq = (uint32_t)cur_seq;
            tour = (uint32_t)g;
        } else if ((g >> 32) == 0ull) {            // (a 64-bit division takes three times as long)
            tour = (uint32_t)g / (uint32_t)P.n_seq;
            seq = (uint32_t)g - tour * (uint32_t)P.n_seq;
        } else {
            seq = (uint32_t)(g % (unsigned long long)P.n_seq);
            tour = (uint32_t)(g / (unsigned long long)P.n_seq);
        }
        n = 0; cur = origin; maxn = 0; W = 1.0; ord = 0u; pbase = (uint32_t)-G;
        top = 0; sbase = 0; bot = 0;
        own = myrow; did = 0u; donated = false;
        acc = first ? Wrow : P.X + (size_t)own * L;
        if (first) {
            const uint32_t s0 = hash_home(origin, log2b) * (uint32_t)Buckets<Key>::kKeys;
            hash[s0] = origin;
            sites[0] = (uint16_t)s0;
        }
        state = kNode;
        seg = 0;
    };
    const long long t_start = global_ns();
    for (uint32_t iter = 0u;; ++iter) {
        // ---------------- everything but the nodes ----------------
        // Walks that ended their tour are looked after at once, the rest every eighth
        // iteration: one vote and one branch on the node's way.
        const bool eighth = (iter & 7u) == 0u;
        if (eighth || __any_sync(kFull, state == kFlush || (state == kNeed && fresh_need))) {
        __syncwarp();                           // the walks' regions as the last node left them
        if ((iter & 255u) == 0u) {
            const bool late = global_ns() - t_start > P.max_ns;
            if (__any_sync(kFull, late)) {
                if (lane == 0) set_status(P.status, PERM_ETIMEOUT);
                break;
            }
            // in a batch launch a failed run stops at once, so that its CTAs move on
            // (the whole warp leaves together: one lane's read decides)
            if (bl != nullptr && __shfl_sync(kFull, *(volatile int *)P.status, 0) != 0) break;
        }
        // ---------------- hand-overs: waiting copies for idle walks ----------------
        // A walk with two waiting records or more hands its oldest one to an idle walk:
        // that subtree grows there, and its weights still go to this tour's row `own`.
        // Its first lane decides and writes the cell's header; the whole warp copies the
        // sites 0..bdp with the slot that an in-order rebuild would give each, so the
        // taker places them without probing.
        // (the warp's donors reserve their cells together:
        // a few round trips to L2 and one fence whatever their number)
        if (snapshot && P.share && eighth && __shfl_sync(kFull, *(volatile int *)&head->want_don, 0) > 0) {
            // at most `cap` parts of one tour grow at once (a soft cap: the parts of a tour
            // stay few, so each still sees its siblings' samples)
            const bool part = did != 0u || donated;       // the tour has parts elsewhere already
            uint32_t bm = 0u;
            double bw = 0.0;
            bool can = first && state == kNode && top - bot >= 2;
            if (can) {
                const int bi = bot & (K - 1);
                bm = bot < sbase ? __ldcg(gmeta + bot) : smeta[bi];
                bw = bot < sbase ? __ldcg(gwt + bot) : sw[bi];
                can = P.n_max - (int)(bm & 0xFFFFu) >= kMinShareGap;
                if (can && part) can = *(volatile unsigned int *)(P.outst + own) < (unsigned)*(volatile int *)&head->cap;
            }
            const unsigned dm = __ballot_sync(kFull, can);
            if (dm) {
                const int cnt = __popc(dm), rk = __popc(dm & lt_mask);
                int k = 0;
                unsigned long long t0 = 0ull;
                if (lane == 0) {
                    // this CTA's quota first, then room in the ring (a count, as on the takers'
                    // side), then the next cells: no retries
                    const int quota = atomicSub(&head->want_don, cnt);
                    k = quota < 0 ? 0 : (quota < cnt ? quota : cnt);
                    if (k > 0) {
                        const int room = (1 << P.dq_log2cap) - atomicAdd(P.dq_used, k);
                        const int fit = room < 0 ? 0 : (room < k ? room : k);
                        if (fit < k) atomicSub(P.dq_used, k - fit);
                        k = fit;
                        if (k > 0) t0 = atomicAdd(P.dq_tail, (unsigned long long)k);
                    }
                    if (k < cnt) atomicAdd(&head->want_don, cnt - k);
                }
                k = __shfl_sync(kFull, k, 0);
                t0 = __shfl_sync(kFull, t0, 0);
                const unsigned long long pos = t0 + (unsigned long long)rk;
                const uint32_t cell = (uint32_t)pos & dq_mask, round = (uint32_t)(pos >> P.dq_log2cap);
                const bool gives = can && rk < k;
                unsigned char *cb = P.dq_cells + (size_t)cell * (size_t)P.dq_cell_bytes;
                if (gives) {
                    // (the taker of the cell's last round may still be copying it)
                    bool ok = false;
                    for (int spin = 0; spin < kCellSpin; ++spin) {
                        if (*(volatile unsigned int *)(P.dq_free + cell) == round) { ok = true; break; }
                        __nanosleep(32);
                    }
                    if (!ok) set_status(P.status, PERM_ETIMEOUT);
                    __threadfence();
                    if (part) atomicAdd(P.outst + own, 1u);
                    else P.outst[own] = 2u;
                    *reinterpret_cast<uint4 *>(cb) = make_uint4((uint32_t)own, seq, tour, bm & 0xFFFFu);
                    *reinterpret_cast<uint2 *>(cb + 16) = make_uint2(bm, 0u);
                    *reinterpret_cast<double *>(cb + 24) = bw;
                }
                const unsigned gm = __ballot_sync(kFull, gives);
                for (unsigned cm = gm; cm; cm &= cm - 1u) {
                    const int src = __ffs(cm) - 1;
                    unsigned char *db = P.dq_cells + (size_t)__shfl_sync(kFull, cell, src) * (size_t)P.dq_cell_bytes;
                    unsigned char *sb = warp_base + wbytes * (size_t)(src / G);
                    copy_sites_to_cell<Key>(reinterpret_cast<const Key *>(sb),
                                            reinterpret_cast<const uint16_t *>(sb + hash_b),
                                            (int)(__shfl_sync(kFull, bm, src) & 0xFFFFu), reinterpret_cast<Key *>(db + 32),
                                            reinterpret_cast<uint16_t *>(db + 32 + cell_key_bytes), lane);
                }
                if (gm) {
                    __threadfence();
                    __syncwarp();
                    if (gives) *(volatile unsigned int *)(P.dq_ready + cell) = round + 1u;
                    if (lane == 0) atomicAdd(P.queued, __popc(gm));
                    if (gm >> lead & 1u) {
                        if (did == 0u) donated = true;
                        bot += 1;
                        if (sbase < bot) sbase = bot;
                    }
                }
            }
        }
        // ---------------- end of a tour (part): per-tour sums into Q (whole warp) ----------------
        if (__any_sync(kFull, state == kFlush)) {
            const bool fl = state == kFlush, whole = did == 0u && !donated;
            bool last = fl;                     // with this part the tour has ended
            int row_max = maxn;                 // the row's deepest length
            if (__any_sync(kFull, fl && !whole)) {
                // parts of a tour grew on several walks: this part's sums must be in the row
                // before the count of its parts says so (a tour that stayed on its walk needs
                // the warp's own order only), and the last part to end flushes the row
                __threadfence();
                __syncwarp();
                unsigned depth = 0u;
                bool ends = false;
                if (fl && !whole && first) {
                    PartsRow row{P.tmaxn + own, P.outst + own};
                    ends = end_part(row, (unsigned)maxn, depth);
                }
                __syncwarp();
                depth = __shfl_sync(kFull, depth, lead);
                ends = __shfl_sync(kFull, (int)ends, lead) != 0;
                bool other_row = false;
                if (fl && !whole) {
                    last = ends;
                    row_max = (int)depth;
                    // the row stays with the parts still growing: the next tour takes the
                    // walk's other row, if that one is free
                    other_row = !last && did == 0u;
                    if (other_row) myrow ^= rows_per_walk - 1;
                }
                unsigned row_use = kRowFree;
                if (other_row && first) row_use = *(volatile unsigned int *)(P.outst + myrow);
                row_use = __shfl_sync(kFull, row_use, lead);
                if (other_row) xbusy = row_use != kRowFree;
            }
            // the whole warp, one ended walk at a time: the row's sums squared into Q, the
            // hash emptied (every bucket, or, of a short walk, its sites' slots)
            unsigned em = __ballot_sync(kFull, fl && first);
            while (em) {
                const int src = __ffs(em) - 1;
                em &= em - 1u;
                const int hi = __shfl_sync(kFull, un_hi, src);
                const int s_row = __shfl_sync(kFull, own, src);
                const int s_max = __shfl_sync(kFull, last ? row_max : -1, src);
                const int s_seq = P.alg == PERM_ALG1 ? __shfl_sync(kFull, cur_seq, src) : 0;
                double *Xr = P.X + (size_t)s_row * L, *Qr = Qtab + (size_t)s_seq * L;
                // eight loads in flight per lane, the first of them while the hash is emptied
                double x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = u * 32 + lane <= s_max ? __ldcg(Xr + u * 32 + lane) : 0.0;
                unsigned char *hb = warp_base + wbytes * (size_t)(src / G);
                const int vecs = (int)(hash_b / 16);
                if (vecs <= 2 * (hi + 1)) {
                    for (int i = lane; i < vecs; i += 32) reinterpret_cast<uint4 *>(hb)[i] = make_uint4(0u, 0u, 0u, 0u);
                } else {
                    const uint16_t *st = reinterpret_cast<const uint16_t *>(hb + hash_b);
                    for (int i = lane; i <= hi; i += 32) reinterpret_cast<Key *>(hb)[st[i]] = (Key)0;
                }
                for (int k0 = 0; k0 <= s_max;) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (k0 + u * 32 > s_max) break;
                        const int k = k0 + u * 32 + lane;
                        const bool take = __double_as_longlong(x[u]) != 0ll;     // (an integer test: no -0.0 here)
                        red_add(Qr + k, __dmul_rn(x[u], x[u]), take);
                        if (take) __stcg(Xr + k, 0.0);
                    }
                    k0 += 32 * 8;
                    if (k0 > s_max) break;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        x[u] = k0 + u * 32 + lane <= s_max ? __ldcg(Xr + k0 + u * 32 + lane) : 0.0;
                }
            }
            __syncwarp();
            if (fl) {
                my_steps += ord;
                if (last && first) {
                    if (!whole) {
                        P.tmaxn[own] = 0u;
                        __threadfence();           // (after the barrier above: the emptied row too)
                        *(volatile unsigned int *)(P.outst + own) = kRowFree;
                    }
                    atomicAdd(P.finished, 1ull);
                }
                if (P.alg == PERM_ALG1) {
                    seq_t += 1;
                    if (first) P.seq_M[cur_seq] = (unsigned long long)seq_t;
                }
                own = myrow; did = 0u; donated = false;
                state = kNeed;
                fresh_need = true;
            }
            // the next tours at once where they are known: the sequence's next one, or tickets
            // that the warp holds
            bool next = fl && !xbusy && !exhausted;
            if (P.alg == PERM_ALG2) {
                const unsigned nm = __ballot_sync(kFull, next && first);
                const unsigned long long cnt = (unsigned long long)__popc(nm);
                if (pool_hi - pool_lo >= cnt && (long long)(pool_lo + cnt) <= limit) {
                    if (next) g = pool_lo + (unsigned long long)__popc(nm & lt_mask);
                    pool_lo += cnt;
                } else {
                    next = false;
                }
            } else {
                next = next && seq_t < P.seq_target;
                if (next) g = (unsigned long long)seq_t;
            }
            if (next) start_tour();
        }
        // ---------------- walks with no tour: tickets, shared copies, leaving ----------------
        // (a walk that found nothing to grow looks again every eighth iteration, and at
        // rows and tickets, which are global, every 32nd: the reads and atomics take several
        // round trips to L2, which the warp's other walks wait for)
        if (__any_sync(kFull, state == kNeed)) {
        const bool deep = P.alg == PERM_ALG1 || (iter & 31u) == 0u || __any_sync(kFull, state == kNeed && fresh_need);
        fresh_need = false;
        const bool blocked = state == kNeed && xbusy;
        if (deep && __any_sync(kFull, blocked)) {
            unsigned r0 = 0u, r1 = 0u;
            if (blocked && first) {
                r0 = *(volatile unsigned int *)(P.outst + myrow);
                if (rows_per_walk == 2) r1 = *(volatile unsigned int *)(P.outst + (myrow ^ 1));
            }
            r0 = __shfl_sync(kFull, r0, lead);
            r1 = __shfl_sync(kFull, r1, lead);
            if (blocked) {
                if (r0 == kRowFree) xbusy = false;
                else if (r1 == kRowFree) { myrow ^= 1; xbusy = false; }
            }
        }
        const bool want_t = deep && state == kNeed && !xbusy && !exhausted;
        const unsigned need = __ballot_sync(kFull, want_t && first);
        if (need) {
            if (P.alg == PERM_ALG2) {
                const unsigned cnt = __popc(need);
                const unsigned rank = __popc(need & lt_mask);
                const unsigned long long avail = pool_hi - pool_lo;
                unsigned long long base = 0ull, take = 0ull;
                if (avail < cnt) {
                    // fetch tickets; admission keeps tours in flight at most
                    // c0 + gamma * finished (a partial grant is allowed)
                    const int leader = __ffs(need) - 1;
                    if (lane == leader) {
                        const long long left = limit - (long long)(snapshot ? *(volatile unsigned long long *)&head->Ms
                                                                            : *(volatile unsigned long long *)P.tickets);
                        const unsigned ahead = !(snapshot || own_rows) ? 0u
                                             : P.slots > kFewWalks ? (unsigned)kPoolExtra
                                                                   : tickets_ahead(left, P.tour_slots, kPoolExtraFew);
                        const unsigned long long want = cnt - avail + ahead;
                        // (past the launch's last ticket a walk needs no admission to learn that)
                        const bool over = left <= 0;
                        take = P.ramp_c0 < 0 || over ? want : admitted(P, want, waiting);
                        base = over ? (unsigned long long)limit : (take > 0ull ? atomicAdd(P.tickets, take) : 0ull);
                    }
                    base = __shfl_sync(kFull, base, leader);
                    take = __shfl_sync(kFull, take, leader);
                }
                const bool served = rank < avail + take;
                if (want_t && served) g = (rank < avail) ? pool_lo + rank : base + (rank - avail);
                if (avail >= cnt) {
                    pool_lo += cnt;
                } else if (avail + take > cnt) {
                    pool_lo = base + (cnt - avail);
                    pool_hi = base + take;
                } else {
                    pool_lo = pool_hi = 0ull;      // pool and grant all handed out
                }
                if (want_t && !served) {
                    waiting = true;                // not admitted yet: try again next round
                } else if (want_t) {
                    waiting = false;
                    if ((long long)g >= limit) {
                        if (P.share) exhausted = true;   // idle: may still take shared copies
                        else state = kDone;
                        if (bl != nullptr && first && (atomicOr(bl->closed + P.run_index, 1) & 3) == 0)
                            atomicSub(bl->runs_open, 1);
                    }
                }
            } else {
                // Algorithm 1: a walk owns a sequence until its tours are done
                const bool ask = state == kNeed && (cur_seq < 0 || seq_t >= P.seq_target);
                unsigned long long s = 0ull;
                if (ask && first) s = atomicAdd(P.tickets, 1ull);
                s = __shfl_sync(kFull, s, lead);
                if (ask) {
                    if (s >= (unsigned long long)P.n_seq) {
                        state = kDone;
                    } else {
                        cur_seq = (int)s;
                        seq_t = (long long)P.seq_M[s];
                        Wrow = P.Wn + (size_t)s * L;
                        Srow = P.Sn + (size_t)s * L;
                        if (P.Rn != nullptr) Rrow = P.Rn + (size_t)s * L;
                    }
                }
                if (state == kNeed && cur_seq >= 0 && seq_t < P.seq_target) {
                    g = (unsigned long long)seq_t;
                } else if (state == kNeed) {
                    cur_seq = -1;          // sequence finished: ask again next round
                }
            }
            if (state == kNeed && !waiting && !xbusy && !exhausted && (P.alg == PERM_ALG2 || cur_seq >= 0)) start_tour();
        }
        if (P.share) {
            // ---------------- shared copies: idle walks take queued ones ----------------
            const bool idle = state == kNeed && (waiting || xbusy || exhausted);
            const unsigned hm = __ballot_sync(kFull, idle && first);
            // one lane's read of the queue length decides for the warp (the block
            // below exchanges values across all lanes)
            if (hm && __shfl_sync(kFull, *(volatile int *)&head->queued, 0) > 0) {
                const int leader = __ffs(hm) - 1;
                unsigned long long base = 0ull, take = 0ull;
                if (lane == leader && *(volatile int *)P.queued > 0) {
                    // take from the count of published cells first, what was there; then the
                    // next cells are this warp's (no retries: with a compare-and-swap on the
                    // head, a thousand idle warps took 3.5 copies per microsecond together)
                    const int k = __popc(hm), left = atomicSub(P.queued, k);
                    const int got = left < 0 ? 0 : (left < k ? left : k);
                    if (got < k) atomicAdd(P.queued, k - got);
                    if (got > 0) base = atomicAdd(P.dq_head, (unsigned long long)got);
                    take = (unsigned long long)got;
                }
                base = __shfl_sync(kFull, base, leader);
                take = __shfl_sync(kFull, take, leader);
                const unsigned rk = __popc(hm & lt_mask);
                bool claiming = idle && rk < take;
                const unsigned long long pos = base + rk;
                const uint32_t cell = (uint32_t)pos & dq_mask;
                const uint32_t round = (uint32_t)(pos >> P.dq_log2cap);
                int cdp = -1;
                bool ok = false;
                if (claiming && first) {
                    for (int spin = 0; spin < kCellSpin; ++spin) {
                        if (*(volatile unsigned int *)(P.dq_ready + cell) == round + 1u) { ok = true; break; }
                        __nanosleep(32);
                    }
                    __threadfence();
                }
                __syncwarp();
                ok = __shfl_sync(kFull, (int)ok, lead) != 0;
                if (claiming) {
                    if (!ok || pos + 1ull >= (1ull << 32)) {
                        set_status(P.status, ok ? PERM_EOVERFLOW : PERM_ETIMEOUT);
                        state = kDone;
                        claiming = false;
                    } else {
                        cdp = (int)__ldcg(reinterpret_cast<const unsigned int *>(P.dq_cells + (size_t)cell *
                                                                                (size_t)P.dq_cell_bytes) + 3);
                    }
                }
                // the walk up to the branch point (Sec. 1), each site straight into the
                // slot it had in the donor's hash; the whole warp places one taker's
                // sites at a time (the taker's hash is empty: it had no walk)
                unsigned cm = __ballot_sync(kFull, claiming && first);
                while (cm) {
                    const int src = __ffs(cm) - 1;
                    cm &= cm - 1u;
                    const uint32_t scell = __shfl_sync(kFull, cell, src);
                    const int sdp = __shfl_sync(kFull, cdp, src);
                    const unsigned char *cb = P.dq_cells + (size_t)scell * (size_t)P.dq_cell_bytes;
                    const Key *ck = reinterpret_cast<const Key *>(cb + 32);
                    const uint16_t *cs = reinterpret_cast<const uint16_t *>(cb + 32 + cell_key_bytes);
                    unsigned char *tb = warp_base + wbytes * (size_t)(src / G);
                    place_sites_from_cell<Key>(reinterpret_cast<Key *>(tb), reinterpret_cast<uint16_t *>(tb + hash_b),
                                               sdp, ck, cs, lane);
                }
                if (claiming) {
                    const unsigned char *cb = P.dq_cells + (size_t)cell * (size_t)P.dq_cell_bytes;
                    const uint4 h0 = __ldcg(reinterpret_cast<const uint4 *>(cb));
                    const uint2 h1 = __ldcg(reinterpret_cast<const uint2 *>(cb + 16));
                    const double cw = __longlong_as_double(__ldcg(reinterpret_cast<const long long *>(cb + 24)));
                    const int dp = (int)h0.w;
                    const uint32_t meta = h1.x;
                    own = (int)h0.x; seq = h0.y; tour = h0.z;
                    g = (unsigned long long)tour * (unsigned long long)P.n_seq + seq;
                    did = (uint32_t)(pos + 1ull);
                    ord = 0u; pbase = (uint32_t)-G;
                    donated = false; maxn = 0;
                    top = 0; sbase = 0; bot = 0;
                    acc = first ? Wrow : P.X + (size_t)own * L;
                    const int cnt = (int)((meta >> 16) & 7u);
                    const uint32_t dirs = meta >> 19;
                    pend_dir = (int)(dirs & 7u);
                    pend_w = cw;
                    pend_depth = dp;
                    if (cnt > 1) {
                        if (first) {
                            smeta[0] = (uint32_t)dp | ((uint32_t)(cnt - 1) << 16) | ((dirs >> 3) << 19);
                            sw[0] = cw;
                        }
                        top = 1;
                    }
                    un_lo = dp + 1; un_hi = dp;
                    waiting = false;
                    state = kUnwindState;      // resumes at the branch point below
                }
                // every lane has read the cells: they may be written again
                __threadfence();
                __syncwarp();
                if (claiming && first) {
                    *(volatile unsigned int *)(P.dq_free + cell) = round + 1u;
                    atomicSub(P.dq_used, 1);
                }
            }
            const int hcount = __popc(__ballot_sync(kFull, first && state == kNeed && (waiting || xbusy || exhausted)));
            if (hcount != my_hungry) {
                if (lane == 0) atomicAdd(P.hungry, hcount - my_hungry);
                my_hungry = hcount;
            }
            // walks with no tickets left stop once every tour of the launch has
            // finished (or the run has failed); one lane's reads decide
            const bool over = (long long)*(volatile unsigned long long *)&head->fin >= limit ||
                              *(volatile int *)&head->status != 0;
            const bool leave = *(volatile int *)&head->may_leave != 0;
            const int go = __shfl_sync(kFull, (over ? 1 : 0) | (leave ? 2 : 0), 0);
            if (state == kNeed && exhausted && ((go & 1) || (!xbusy && (go & 2)))) state = kDone;
        }
        }
        if (snapshot ? g + 1ull > tours.M : own_rows && g + 1ull != tours.M) set_tours<!cutoffs>(tours, g + 1ull);
        if (!__any_sync(kFull, state == kNode || state == kUnwindState)) {
            // nothing to grow: the warp backs off, or leaves
            if (!__any_sync(kFull, state != kDone)) break;
            __nanosleep(idle_ns);
            idle_ns = idle_ns < 4000u ? 2u * idle_ns : 4000u;
            fresh_need = true;
            iter |= 7u;                         // (so that the next look is a full one)
            ++my_iters;
            continue;
        }
        idle_ns = 500u;
        }
        ++my_iters;

        // ---------------- one node of every walk that has one ----------------
        // One straight line with few branches, each of them for something rare: on this
        // part a lone warp pays 25 cycles or more for a branch, taken or not, 45 for a vote
        // and a branch on it.
        {
            __syncwarp();                       // the walks' hashes as the last iteration left them
            const bool isn = state == kNode, grows_on = isn && n < P.n_max;
            // the sum of the weights recorded at this length before the node (snapshot form: the
            // refresher may write it meanwhile, so the group takes what its first lane has read,
            // below)
            double Wsum = 0.0;
            longlong2 cut_n = make_longlong2(0, 0);
            if (cutoffs) cut_n = __ldg(cuts.cut + n);
            uint32_t m_low = ms_low;            // low word of the snapshot's M: whether it changed
            if (snapshot) {
                Wsum = *(volatile double *)&Wsnap[n];
                m_low = *(volatile uint32_t *)&head->Ms;
            } else if (own_rows) {
                Wsum = Wrow[n];
            }
            // a_+ (Sec. 1): lane j of the group probes neighbour j
            const bool probes = grows_on && j < 2 * D;
            const Key nkey = cur + dkey;
            uint32_t bucket = hash_home(nkey, log2b);
            bool hit, full;
            int place;
            look_bucket(hash, bucket, nkey, hit, full, place);
            // the node's weight goes into the tables with reductions that return nothing, one
            // lane each.  Fresh form: a row of the walk's own takes a load (of the whole group)
            // and a store (of its first lane) through L1; on a shared one the add returns the
            // sum before it, a round trip to L2
            if (!snapshot && !own_rows) {
                double before = 0.0;
                unsigned long long Mt = 0ull;
                if (isn && first) {
                    before = atomicAdd(&Wrow[n], W);
                    Mt = *(volatile unsigned long long *)P.tickets;
                }
                Wsum = __shfl_sync(kFull, before, lead);
                Mt = __shfl_sync(kFull, Mt, lead);
                if ((long long)Mt > limit) Mt = (unsigned long long)limit;
                Mt = Mt > g + 1ull ? Mt : g + 1ull;
                if (isn && Mt != tours.M) set_tours<!cutoffs>(tours, Mt);
            }
            red_add(acc + n, W, isn && (snapshot ? j < 2 : j == 1));
            double sum = 0.0;
            if (!snapshot) sum = __dadd_rn(Wsum, W);
            if (!snapshot && own_rows && isn && first) Wrow[n] = sum;
            // a full bucket without the key, a used-up block of random words, a new M: one vote
            // for the three
            bool more = probes && full && !hit;
            const bool refill = isn && ord - pbase >= (uint32_t)G;
            if (__any_sync(kFull, more || refill || m_low != ms_low)) {
                if (snapshot) {
                    ms_low = __shfl_sync(kFull, m_low, 0);
                    const unsigned long long Ms = __shfl_sync(kFull, *(volatile unsigned long long *)&head->Ms, 0);
                    const unsigned long long Mn = Ms > g + 1ull ? Ms : g + 1ull;
                    if (Mn != tours.M) set_tours<!cutoffs>(tours, Mn);
                }
                if (__any_sync(kFull, refill)) {
                    pbase = ord;
                    if (isn && ord >= 0xFFFFFFF0u) set_status(P.status, PERM_EOVERFLOW);
                    const Philox4 w = philox4x32_10(ord + (uint32_t)j, did, tour, seq, P.key0, P.key1);
                    pw0 = w.x; pw1 = w.y;
                }
                const uint32_t bmask = (1u << log2b) - 1u;
                for (uint32_t it = 0u; __any_sync(kFull, more); ++it) {
                    if (it >= bmask) { if (more) set_status(P.status, PERM_EOVERFLOW); break; }
                    if (more) {
                        bucket = (bucket + it + 1u) & bmask;
                        look_bucket(hash, bucket, nkey, hit, full, place);
                        more = full && !hit;
                    }
                }
            }
            const bool free_j = probes && !hit && !full;
            const int nslot = (int)(bucket * (uint32_t)Buckets<Key>::kKeys) + place;
            const int fm = (int)((__ballot_sync(kFull, free_j) >> lead) & ((1u << G) - 1u));
            const int a = __popc(fm), a1 = a > 0 ? a : 1;
            const bool decides = grows_on && a > 0;
            // the node's random words, from the lane that holds its block, and what the estimate
            // of r says
            const int wl = lead + (int)((ord - pbase) & (uint32_t)(G - 1));
            const uint32_t w0 = __shfl_sync(kFull, pw0, wl), w1 = __shfl_sync(kFull, pw1, wl);
            // the group's W_n is its first lane's (two lanes with different sums could decide
            // differently and part for good); taken here, where the load is long done: right
            // after the look it cost square n = 512 continued 49.5 -> 51.2 ms, 12 walks to n = 16
            // 22.9 -> 23.9
            if (snapshot && !cutoffs) {
                Wsum = __shfl_sync(kFull, Wsum, lead);
                sum = __dadd_rn(Wsum, W);
            }
            Guess gs;
            if (!cutoffs) gs = guess(W, Wsum, tours.Mf, w0);
            // the first child's step (a draw from the free list), its key and its place in the
            // hash, from the lane that probed it
            const uint32_t list = lists[fm];
            const unsigned long long prod = (unsigned long long)w1 * (uint32_t)a1;
            const int dir0 = (int)((list >> (3 * (int)(prod >> 32))) & 7u);
            const Key ckey = __shfl_sync(kFull, nkey, lead + dir0);
            const int cslot = __shfl_sync(kFull, nslot, lead + dir0);
            Decision o;
            if (cutoffs) o = decide_cutoffs<D>(n, a1, W, cut_n, w0, aoc, cuts);
            else o = decide_node<D>(n, a1, W, sum, gs, tours, !snapshot, snapshot && (uint32_t)tours.M != ms_low, w0, aoc, decides, false);
            const int c = decides ? o.c : 0;
            if (o.exact && decides) my_exact += 1ull;
            const bool extend = c > 0, leaf = isn && c == 0;

            if (extras) {
            if (P.Rn != nullptr) {
                // the observable of Sec. 1, eq. 5: W |omega_n|^2 (exact integer square)
                int cx, cy, cz;
                KeyCodec<D, Key>::decode(cur, cx, cy, cz);
                const long long r2 = (long long)cx * cx + (long long)cy * cy + (long long)cz * cz;
                red_add(Rrow + n, __dmul_rn(W, (double)r2), isn && j == 3);
            }
            const unsigned long long ordinal = ((unsigned long long)did << 32) | ord;
            if (P.trace != nullptr && isn && first && (ordinal % (unsigned long long)P.trace_every) == 0ull &&
                ((unsigned long long)tour % (unsigned long long)P.trace_tour_every) == 0ull) {
                const unsigned long long idx = atomicAdd(P.trace_count, 1ull);
                if (idx < (unsigned long long)P.trace_cap) {
                    perm_trace_record *rec = P.trace + idx;
                    rec->n = n; rec->a_plus = a; rec->free_mask = fm; rec->c = c;
                    rec->outcome = !grows_on ? kLeafNmax : (a == 0 ? kTrapped : (c == 0 ? kPruned : kChildren));
                    rec->exact = decides && o.exact ? 1 : 0;
                    uint32_t dirs = list, xw = w1;
                    for (int i = 0; i < c; ++i) choose_step(i, a, dirs, xw);
                    for (int i = 0; i < 6; ++i)
                        rec->dirs[i] = (i < c) ? (int)((dirs >> (3 * i)) & 7u) : -1;
                    rec->seq = seq; rec->tour = tour;
                    rec->ordinal = ordinal; rec->M = tours.M;
                    rec->W = W; rec->Wsum = Wsum; rec->r = decision_r(o, n, cutoffs); rec->child_w = c > 0 ? o.child_w : 0.0;
                    int32_t *cc = P.trace_coords + (size_t)idx * L * D;
                    for (int k = 0; k <= n; ++k) {
                        int x, y, z;
                        KeyCodec<D, Key>::decode(k < n ? hash[sites[k]] : cur, x, y, z);
                        cc[k * D] = x; cc[k * D + 1] = y;
                        if (D == 3) cc[k * D + 2] = z;
                    }
                }
            }
            }

            if (c > 1) {
                // copies 1..c-1 wait in one record (depth, count, steps, weight): the first
                // draw's exchange, then the others'
                const unsigned gmask = ((1u << G) - 1u) << lead;
                uint32_t dirs = list, xw = w1;
                choose_step(0, a, dirs, xw);
                choose_step(1, a, dirs, xw);
                for (int i = 2; i < c; ++i) choose_step(i, a, dirs, xw);
                my_copies += (unsigned long long)(c - 1);
                if (top - sbase == K || top >= P.n_max) {
                    // ring full: the oldest kChunk records go to global memory (a walk has at
                    // most n_max records: their depths increase)
                    if (top >= P.n_max) {
                        set_status(P.status, PERM_EOVERFLOW);
                        top = P.n_max - 1;
                    }
                    if (top - sbase == K) {
#pragma unroll
                        for (int i = 0; i < kChunk; i += G) {
                            const int idx = sbase + i + j;
                            gmeta[idx] = smeta[idx & (K - 1)];
                            gwt[idx] = sw[idx & (K - 1)];
                        }
                        sbase += kChunk;
                    }
                    __syncwarp(gmask);
                }
                if (first) {
                    const uint32_t rest = (dirs >> 3) & ((1u << (3 * (c - 1))) - 1u);
                    const int ti = top & (K - 1);
                    smeta[ti] = (uint32_t)n | ((uint32_t)(c - 1) << 16) | (rest << 19);
                    sw[ti] = o.child_w;
                }
                ++top;
                my_max_stack = top - bot > my_max_stack ? top - bot : my_max_stack;
            }
            ord += isn ? 1u : 0u;
            cur = extend ? ckey : cur;
            W = extend ? o.child_w : W;
            const int n_leaf = n;
            n += extend ? 1 : 0;
            if (first && extend && n < P.n_max) {
                hash[cslot] = ckey;
                sites[n] = (uint16_t)cslot;
            }

            // ---------------- a leaf, or a backtrack still under way ----------------
            // The most recent waiting copy, or the end of the tour; LIFO deletions, the
            // group's lanes side by side; then the walk resumes.
            if (leaf || state == kUnwindState) {
                const unsigned gmask = ((1u << G) - 1u) << lead;
                if (leaf && top == sbase && sbase > bot) {
                    // ring empty: bring back up to kChunk records, the group's lanes side by side
                    const int lo = sbase - kChunk > bot ? sbase - kChunk : bot;
                    for (int idx = lo + j; idx < sbase; idx += G) {
                        smeta[idx & (K - 1)] = __ldcg(gmeta + idx);
                        sw[idx & (K - 1)] = __ldcg(gwt + idx);
                    }
                    sbase = lo;
                    __syncwarp(gmask);
                }
                // one straight line from here for a group that pops a record, one that ends
                // its tour and one still deleting (selects; a branch costs more)
                const bool pops = leaf && top != bot;
                const int ti = (top - 1) & (K - 1);
                const uint32_t meta = smeta[ti], rest = meta >> 19;
                const double rec_w = sw[ti];
                const int cnt = (int)((meta >> 16) & 7u);
                if (leaf) {
                    maxn = n_leaf > maxn ? n_leaf : maxn;
                    un_hi = n_leaf < P.n_max - 1 ? n_leaf : P.n_max - 1;
                    state = pops ? kUnwindState : kFlush;
                    // one node of each length since the walk started or resumed (Srow:
                    // differences along n)
                    red_count(Srow + (j == 2 ? seg : n_leaf + 1), j == 2 ? 1 : -1,
                              j == 2 || (j == 3 && n_leaf < P.n_max));
                }
                if (pops) {
                    pend_dir = (int)(rest & 7u);
                    pend_w = rec_w;
                    pend_depth = (int)(meta & 0xFFFFu);
                    un_lo = pend_depth + 1;
                    top -= cnt <= 1 ? 1 : 0;
                }
                __syncwarp(gmask);              // every lane has read the record
                if (pops && cnt > 1 && first)
                    smeta[ti] = (meta & 0xFFFFu) | ((uint32_t)(cnt - 1) << 16) | ((rest >> 3) << 19);
                const bool back = state == kUnwindState;
                const Key rkey = hash[sites[back ? pend_depth : 0]] + step_key<D, Key>(pend_dir);
                int sl[kUnwind];
#pragma unroll
                for (int i = 0; i < kUnwind; ++i) {
                    const int k = un_hi - j - i * G;
                    sl[i] = back && k >= un_lo ? (int)sites[k] : -1;
                }
#pragma unroll
                for (int i = 0; i < kUnwind; ++i)
                    if (sl[i] >= 0) hash[sl[i]] = (Key)0;
                un_hi -= back ? kUnwind * G : 0;
                __syncwarp(gmask);
                // the new end-point's place (every lane of the group looks at the same buckets):
                // the first bucket of its sequence that is not full
                const bool resumes = back && un_hi < un_lo;
                const bool places = resumes && pend_depth + 1 < P.n_max;
                uint32_t rb = hash_home(rkey, log2b);
                if (SHARED || places) look_bucket(hash, rb, rkey, hit, full, place);
                if (places && full) {
                    const uint32_t bmask = (1u << log2b) - 1u;
                    for (uint32_t it = 0u; full && it < bmask; ++it) {
                        rb = (rb + it + 1u) & bmask;
                        look_bucket(hash, rb, rkey, hit, full, place);
                    }
                    if (full) set_status(P.status, PERM_EOVERFLOW);
                }
                __syncwarp(gmask);              // every lane has looked
                if (resumes) {
                    n = pend_depth + 1;
                    cur = rkey;
                    W = pend_w;
                    state = places && full ? kDone : kNode;
                    seg = n;
                }
                if (places && first && !full) {
                    const uint32_t rs = rb * (uint32_t)Buckets<Key>::kKeys + (uint32_t)place;
                    hash[rs] = rkey;
                    sites[n] = (uint16_t)rs;
                }
            }
        }
    }
    if (P.share && lane == 0 && my_hungry != 0) atomicAdd(P.hungry, -my_hungry);

    // statistics (a walk cut short by an error counts its part so far), then tell the
    // refresher this warp is done
    if (state == kNode || state == kUnwindState) my_steps += ord;
    red_count(Srow + (j == 2 ? seg : n), j == 2 ? 1 : -1, state == kNode && n > seg && (j == 2 || j == 3));
    unsigned long long tot = first ? my_steps : 0ull, cps = first ? my_copies : 0ull, exn = first ? my_exact : 0ull;
    int ms = my_max_stack;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        tot += __shfl_xor_sync(kFull, tot, off);
        cps += __shfl_xor_sync(kFull, cps, off);
        exn += __shfl_xor_sync(kFull, exn, off);
        const int o = __shfl_xor_sync(kFull, ms, off);
        ms = o > ms ? o : ms;
    }
    if (lane == 0) {
        atomicAdd(P.steps, tot);
        atomicAdd(P.copies, cps);
        if (exn) atomicAdd(P.exact_steps, exn);
        atomicAdd(P.iterations, my_iters);
        atomicMax(P.max_stack, (unsigned long long)ms);
        __threadfence_block();
        atomicAdd(&head->done_warps, 1);
    }
    }   // worker warps
}

// A launch's kernel.  (Walks in the arena: the two forms that are not plain serve them.)
template <int D, typename Key, int MODE, int FORM>
__global__ void __launch_bounds__(32 * (walk_warps_max(sizeof(Key) == 8) + 1), 1) grow_kernel(const __grid_constant__ RunDev P) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (FORM == kPlain || P.arena_mode == kArenaNone)
        grow_run<D, Key, MODE, true, FORM>(P, smem, nullptr, P.worker_warps * P.S);
    else
        grow_run<D, Key, MODE, false, FORM>(P, smem, nullptr, P.worker_warps * P.S);
}

// the largest opt-in shared memory per block, set once per kernel
template <int D, typename Key, int MODE, int FORM>
cudaError_t allow_smem() {
    static int done = 0;
    if (done) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(grow_kernel<D, Key, MODE, FORM>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess) done = 1;
    return e;
}

template <int D, typename Key, int MODE, int FORM>
cudaError_t launch_one(const RunDev &P, int ctas, cudaStream_t stream) {
    const bool snapshot = (MODE == kSnapshot);
    // shared memory holds what the arena does not
    const size_t head = P.arena_mode == kArenaAll ? 0 : head_region_bytes(P.n_max, snapshot);
    const size_t smem = head + (P.arena_mode != kArenaNone ? 0 : walk_region_bytes(P.n_max, P.log2h, P.stack_cache, sizeof(Key)) *
                                                                     (size_t)(P.S * P.worker_warps));
    cudaError_t e = allow_smem<D, Key, MODE, FORM>();
    if (e != cudaSuccess) return e;
    const int threads = 32 * (P.worker_warps + (snapshot ? 1 : 0));
    grow_kernel<D, Key, MODE, FORM><<<ctas, threads, smem, stream>>>(P);
    return cudaGetLastError();
}
template <int D, typename Key, int FORM>
cudaError_t launch_mode(const RunDev &P, int thresh_mode, int ctas, cudaStream_t stream) {
    return thresh_mode == kSnapshot ? launch_one<D, Key, kSnapshot, FORM>(P, ctas, stream)
                                    : launch_one<D, Key, kFresh, FORM>(P, ctas, stream);
}
template <int D, typename Key>
cudaError_t launch_form(const RunDev &P, int thresh_mode, int ctas, cudaStream_t stream) {
    if (P.cut != nullptr) return launch_mode<D, Key, kCutoffs>(P, thresh_mode, ctas, stream);
    if (plain_run(P)) return launch_mode<D, Key, kPlain>(P, thresh_mode, ctas, stream);
    return launch_mode<D, Key, kWatched>(P, thresh_mode, ctas, stream);
}
template <int D, typename Key, int FORM>
cudaError_t allow_form() {
    const cudaError_t e = allow_smem<D, Key, kSnapshot, FORM>();
    return e == cudaSuccess ? allow_smem<D, Key, kFresh, FORM>() : e;
}
template <int D, typename Key>
cudaError_t allow_smem_all() {
    cudaError_t e = allow_form<D, Key, kPlain>();
    if (e == cudaSuccess) e = allow_form<D, Key, kWatched>();
    if (e == cudaSuccess) e = allow_form<D, Key, kCutoffs>();
    return e;
}

}  // namespace
}  // namespace perm
