// perm_device.cuh -- device building blocks of the flatPERM growth step.
//
// Paper: Campbell and Janse van Rensburg, "Parallel PERM".
//   Sec. 1, eqs. (1)-(2): a_+ free neighbours of the end-point; the next step is
//     uniform among them; W = prod a_+.
//   Sec. 2, eq. (6) and the two paragraphs after it: r = W/[W_n]^sample with the
//     own weight included; r >= 1 enriches into c copies (c = floor r with
//     probability ceil r - r, else ceil r) of weight W/c; r < 1 prunes with
//     probability 1 - r, a survivor's weight is multiplied by 1/r.
//
// Layout conventions shared by the kernels:
//   - A group of lanes holds one walk: 4 lanes on the square lattice, 8 on the cubic
//     one.  Every lane of a group carries the walk's state; lane j of the group
//     stands for direction j.
//   - A walk's occupancy hash, its per-site slot list and its stack ring are
//     contiguous.  The hash is made of buckets of 4 keys.
//   - Keys pack the lattice coordinates of a site; 0 is the empty slot.  The key of
//     neighbour j is the site's key plus a constant of the direction.
//   - Directions: j = 0..2d-1 -> axis j/2, sign + for even j (+x,-x,+y,-y,+z,-z).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace perm {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32
// multiplies with round keys bumped by the Weyl constants.
// ---------------------------------------------------------------------------
struct Philox4 { uint32_t x, y, z, w; };

__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2,
                                                 uint32_t c3, uint32_t k0, uint32_t k1) {
    const uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u;
    const uint32_t kW0 = 0x9E3779B9u, kW1 = 0xBB67AE85u;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(kM0, c0), lo0 = kM0 * c0;
        const uint32_t hi1 = __umulhi(kM1, c2), lo1 = kM1 * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += kW0;
        k1 += kW1;
    }
    return {c0, c1, c2, c3};
}

// ---------------------------------------------------------------------------
// Site keys.  Key32<2>: 16-bit fields x+32768 | (y+32768)<<16, |x|,|y| <= 32766.
// Key32<3>: c+512 at bits 0, 11 and 22, for walks with n_max <= 512: every stored
// site has |c| <= 511 (field 1..1023, never 0); a probe at c = -512 gives field 0,
// one at +512 sets the guard bit above the field (for z it leaves field 0), so
// neither matches a stored site, and adding a direction's constant never borrows
// from or carries into another field.  Key64<3>: 21-bit fields.
// ---------------------------------------------------------------------------
template <int D, typename Key> struct KeyCodec;

template <> struct KeyCodec<2, uint32_t> {
    static constexpr int kField = 16;
    __device__ __forceinline__ static uint32_t encode(int x, int y, int) {
        return (uint32_t)(x + 32768) | ((uint32_t)(y + 32768) << 16);
    }
    __device__ __forceinline__ static void decode(uint32_t k, int &x, int &y, int &z) {
        x = (int)(k & 0xFFFFu) - 32768;
        y = (int)(k >> 16) - 32768;
        z = 0;
    }
};

template <> struct KeyCodec<3, uint32_t> {
    static constexpr int kField = 11;
    __device__ __forceinline__ static uint32_t encode(int x, int y, int z) {
        return (uint32_t)(x + 512) + ((uint32_t)(y + 512) << 11) + ((uint32_t)(z + 512) << 22);
    }
    // (the end-point of a walk of 512 steps along z reads z = -512 for +512: the
    // same square)
    __device__ __forceinline__ static void decode(uint32_t k, int &x, int &y, int &z) {
        x = (int)(k & 2047u) - 512;
        y = (int)((k >> 11) & 2047u) - 512;
        z = (int)(k >> 22) - 512;
    }
};

template <> struct KeyCodec<3, unsigned long long> {
    static constexpr int kField = 21;
    __device__ __forceinline__ static unsigned long long encode(int x, int y, int z) {
        return (unsigned long long)(uint32_t)(x + (1 << 20)) |
               ((unsigned long long)(uint32_t)(y + (1 << 20)) << 21) |
               ((unsigned long long)(uint32_t)(z + (1 << 20)) << 42);
    }
    __device__ __forceinline__ static void decode(unsigned long long k, int &x, int &y, int &z) {
        x = (int)(k & 0x1FFFFFull) - (1 << 20);
        y = (int)((k >> 21) & 0x1FFFFFull) - (1 << 20);
        z = (int)((k >> 42) & 0x1FFFFFull) - (1 << 20);
    }
};

// What a step in direction j adds to a site's key.
template <int D, typename Key>
__device__ __forceinline__ Key step_key(int j) {
    const Key one = (Key)1 << (KeyCodec<D, Key>::kField * (j >> 1));
    return (j & 1) ? (Key)0 - one : one;
}

// ---------------------------------------------------------------------------
// The occupancy hash: 2^log2b buckets of 4 keys (16 bytes, or 32 with 64-bit keys),
// probed triangularly from the key's home: the i-th bucket is home + i(i+1)/2 mod
// 2^log2b, which visits every bucket once.  A key sits in the first bucket of its
// sequence with room, in that bucket's first empty place.  Keys are deleted in
// LIFO order only, so a bucket's keys always fill its first places, every bucket
// that a key passed over is full while the key lives, and a probe may stop at the
// first bucket that is not full.  One look at a bucket (a 16-byte load, or two that
// are in flight together) settles a probe unless it is full: at the load of at most
// 1/2 that a walk reaches at n_max, one bucket of four in seven is full, against one
// slot in two with one key per probe.  64-bit keys went in twos before, one load a
// look and more looks: cubic chains (no cut-off active) at n_max 4096, 608 sequences,
// 4 tours 14.8 ms against 15.3, 1000, 1000 sequences, 8 tours 4.8 against 5.05, 10000
// (walks in the arena), 608 sequences, 4 tours 24.5 against 26.3.
// ---------------------------------------------------------------------------
template <typename Key> struct Buckets {
    static constexpr int kKeys = 4, kLog2 = 2;
};

__device__ __forceinline__ uint32_t hash_home(uint32_t k, int log2b) {
    return (k * 0x9E3779B1u) >> (32 - log2b);
}
__device__ __forceinline__ uint32_t hash_home(unsigned long long k, int log2b) {
    const uint32_t f = (uint32_t)k ^ (uint32_t)(k >> 29) ^ (uint32_t)(k >> 53);
    return (f * 0x9E3779B1u) >> (32 - log2b);
}

// One bucket: whether it holds k, whether it is full, its first empty place.
__device__ __forceinline__ void look_bucket(const uint32_t *tab, uint32_t b, uint32_t k, bool &hit, bool &full, int &e) {
    const uint4 v = *reinterpret_cast<const uint4 *>(tab + 4u * b);
    hit = v.x == k || v.y == k || v.z == k || v.w == k;
    full = v.w != 0u;
    e = (v.x != 0u) + (v.y != 0u) + (v.z != 0u);
}
__device__ __forceinline__ void look_bucket(const unsigned long long *tab, uint32_t b, unsigned long long k, bool &hit,
                                            bool &full, int &e) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(tab + 4u * b);
    const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(tab + 4u * b + 2u);
    hit = v.x == k || v.y == k || u.x == k || u.y == k;
    full = u.y != 0ull;
    e = (v.x != 0ull) + (v.y != 0ull) + (u.x != 0ull);
}

// Every lane of the warp probes for its own key in its own walk's table (want:
// the lane takes part).  Returns true if the key is absent; `slot` is then where
// it would be inserted.  `overflow`: the probe ran through the whole table
// (impossible at a load of at most 1/2).
template <typename Key>
__device__ __forceinline__ bool probe(const Key *tab, int log2b, Key k, bool want, int &slot, bool &overflow) {
    const uint32_t mask = (1u << log2b) - 1u;
    uint32_t b = hash_home(k, log2b);
    bool absent = false, pend = want;
    for (uint32_t it = 0;; ++it) {
        bool hit, full;
        int e;
        look_bucket(tab, b, k, hit, full, e);
        if (pend && !hit && !full) { absent = true; slot = (int)(b * (uint32_t)Buckets<Key>::kKeys) + e; }
        pend = pend && !hit && full;
        if (!__any_sync(0xFFFFFFFFu, pend)) break;
        if (it >= mask) { overflow = pend; break; }
        b = (b + it + 1u) & mask;
    }
    return absent;
}

// ---------------------------------------------------------------------------
// The ratio r of Sec. 2 (eq. 6): r = W / [W_n]^sample, [W_n]^sample =
// (Wsum + W) / M with Wsum the sum of the weights recorded at length n before
// the node and M the tours started.
//
// The decision needs r only through comparisons (r >= 1, floor and ceil of r,
// u0 < ceil(r) - r, u0 < r), so each node first takes them on a single-
// precision estimate x of r and falls back to r evaluated exactly as defined,
// in double precision, when x lies too close to a comparison's boundary to
// settle it.  The decision then equals the one taken on the double-precision
// r at every node.
//
// The estimate: x = (M m_w) / (m_w + m_s 2^(e_s - e_w)), with the two doubles
// entering through their mantissas truncated to 24 bits and their exponents.  The
// quotient is a product with the hardware's approximate reciprocal (rcp.approx, at
// most one unit in the last place, i.e. relative error <= 2^-23); the other
// operations are correctly rounded single-precision ones (the scaling by a power
// of two is exact).  Relative errors of x, in 2^-24: the truncated mantissas 2
// each (x depends on W/Wsum with a logarithmic derivative below 1), M 1, M m_w 1,
// the sum 1, the reciprocal 2, the last product 1, with the three roundings of the
// double-precision r (<= 4 2^-53): |x - r| <= 10.02 2^-24 x.  Every margin below
// allows at least 15 2^-24 x.  Doubles with no such bound (W zero, negative,
// subnormal or not finite; Wsum negative, subnormal or not finite; Wsum/W above
// 2^100) set `odd` and take the exact path, and so does M of 2^32 or more (M
// enters through a 32-bit conversion: a 64-bit one costs as much as a
// double-precision operation).  Every operation here is single-precision or integer
// arithmetic: a double-precision one takes 64 cycles or more on this part.  (With
// mantissas rounded to nearest and two reciprocals, M / (1 + Wsum/W), the bound was
// the same and the chain one reciprocal and a dozen integer operations longer.)
// ---------------------------------------------------------------------------
// The top 24 bits of a double's mantissa as a float in [1, 2).
__device__ __forceinline__ float mant24(uint32_t hi, uint32_t lo) {
    return __uint_as_float((__funnelshift_l(lo, hi, 3) & 0x7FFFFFu) | 0x3F800000u);
}

// 1/v to within one unit in the last place (v normal and positive).
__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// M as the estimate takes it (-1: beyond the estimate's range).
__device__ __forceinline__ float tours_float(unsigned long long M) {
    return (M >> 32) != 0ull ? -1.0f : __uint2float_rn((uint32_t)M);
}

__device__ __forceinline__ float ratio_estimate(double W, double Wsum, float Mf, bool &odd) {
    const uint32_t wh = (uint32_t)__double2hiint(W), wl = (uint32_t)__double2loint(W);
    const uint32_t sh = (uint32_t)__double2hiint(Wsum), sl = (uint32_t)__double2loint(Wsum);
    const int ew = (int)(wh >> 20), es = (int)(sh >> 20);      // sign bit and exponent
    const bool s_zero = (sh | sl) == 0u;
    const float mw = mant24(wh, wl);
    // below 2^-100 the ratio only moves the sum by less than 2^-99 of it
    int e = es - ew;
    odd = (uint32_t)(ew - 1) >= 2046u || ((uint32_t)(es - 1) >= 2046u && !s_zero) || (!s_zero && e > 100) || Mf < 0.0f;
    e = e < -100 ? -100 : (e > 100 ? 100 : e);
    float ms = __fmul_rn(mant24(sh, sl), __uint_as_float((uint32_t)(e + 127) << 23));   // exact scaling
    ms = s_zero ? 0.0f : ms;
    return __fmul_rn(__fmul_rn(Mf, mw), rcp_approx(__fadd_rn(mw, ms)));
}

// r exactly as defined, in double precision: three correctly rounded operations
// in the definition's order.
__device__ __forceinline__ double ratio_exact(double W, double Wsum, unsigned long long M) {
    const double avg = __ddiv_rn(__dadd_rn(Wsum, W), __ull2double_rn(M));
    return __ddiv_rn(W, avg);
}

// Stored-weight scale: weight of a length-n walk is kept divided by 2^E(n).
__device__ __forceinline__ int scale_exp(int d, int n) {
    return d == 2 ? (11 * n) >> 3 : (9 * n) >> 2;
}

// Exact float -> double widening by bit manipulation (normal floats and zero).
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f);
    if ((b & 0x7FFFFFFFu) == 0u) return 0.0;
    const unsigned long long e = ((b >> 23) & 0xFFu) + (1023u - 127u);
    const unsigned long long d = ((unsigned long long)(b >> 31) << 63) | (e << 52) |
                                 ((unsigned long long)(b & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)d);
}

// ---------------------------------------------------------------------------
// The decision of Sec. 2 on the estimate x (enrichment: c = floor r iff
// u0 < ceil(r) - r, at most a_+ copies; pruning: survive iff u0 < r, with
// u0 = w0 2^-32).  Both are the floor of one sum: for r >= 1, c = floor(r + u0); for
// r < 1, c = floor(r + 1 - u0) (1: survive).  Sets `amb` when x cannot settle it:
//  - the branch: x >= 1 + 2^-19 gives r > 1, x <= 1 - 2^-19 gives r < 1;
//  - the floor: the sum y for x lies within x 2^-20 + 2^-23 of an integer k <= a_+
//    (past a_+ both neighbours of k give c = a_+).  The sum for r is within
//    10.02 x 2^-24 (the estimate) + 2^-25 (u0 to single precision) + (x + 1) 2^-24
//    (the sum's rounding) of y, which is less.  (r an integer: c = r whatever u0, and
//    so is floor(r + u0).)
// x enters capped at 16, past every a_+ + 1.  Selects, no branches: a warp's walks
// take different sides, and a branch costs a lone warp 25 cycles or more.  (The same
// decision by ceilings and thresholds on w0 took 144 cycles of a lone warp, this
// one 60.)  Everything but the cap a_+ is formed before the probes have settled a_+.
// ---------------------------------------------------------------------------
struct Guess {
    float x;             // the estimate of r
    int c;               // floor of the sum, not yet capped at a_+ (r < 1: 1 survives, 0 is pruned)
    int k;               // the integer next to the sum
    bool up, near_k;     // r >= 1; the sum lies within the margin of k
    bool open;           // no branch of r settled, or no estimate
};
__device__ __forceinline__ Guess guess(double W, double Wsum, float Mf, uint32_t w0) {
    Guess g;
    bool odd = false;
    const float uf = __fmul_rn(__uint2float_rn(w0), 0x1p-32f), vf = __fmul_rn(__uint2float_rn(~w0), 0x1p-32f);
    g.x = ratio_estimate(W, Wsum, Mf, odd);
    const float xc = fminf(g.x, 16.0f);
    g.up = xc >= 1.0f;
    const float y = __fadd_rn(xc, g.up ? uf : vf);
    const float kf = __fsub_rn(__fadd_rn(y, 12582912.0f), 12582912.0f);       // y to the nearest integer
    const float tol = __fmaf_rn(xc, 0x1p-20f, 0x1p-23f);
    g.k = (int)kf;
    g.c = kf > y ? g.k - 1 : g.k;
    g.near_k = fabsf(__fsub_rn(y, kf)) <= tol;
    g.open = odd || fabsf(__fsub_rn(xc, 1.0f)) < 0x1p-19f;
    return g;
}

// The same decision on the double-precision r, with the comparisons taken on
// doubles exactly as defined.
__device__ __forceinline__ int decide_exact(double r, int a, uint32_t w0, bool &surv) {
    const double u0 = __dmul_rn(__uint2double_rn(w0), 0x1p-32);             // exact
    surv = false;
    if (r >= 1.0) {
        const double fl = floor(r), ce = ceil(r);
        const double p = __dsub_rn(ce, r);
        const double craw = (u0 < p) ? fl : ce;
        return (craw >= (double)a) ? a : (int)craw;
    }
    surv = u0 < r;
    return surv ? 1 : 0;
}

// Step i of a partial Fisher-Yates shuffle of the free list (3 bits per entry, a
// entries): entry i changes places with one drawn from i..a-1 by multiply-high on x,
// which keeps the product's low word for the next draw.
__device__ __forceinline__ void choose_step(int i, int a, uint32_t &list, uint32_t &x) {
    const unsigned long long prod = (unsigned long long)x * (uint32_t)(a - i);
    const int si = 3 * i, sj = 3 * (i + (int)(prod >> 32));
    x = (uint32_t)prod;
    const uint32_t t = ((list >> si) ^ (list >> sj)) & 7u;
    list ^= (t << si) ^ (t << sj);                  // the same place: the two cancel
}

}  // namespace perm
