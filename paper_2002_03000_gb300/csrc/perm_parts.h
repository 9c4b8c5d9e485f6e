// perm_parts.h -- how tours are handed out, and how the parts of one tour end (shared
// copies).  Plain C++, so that both can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define PERM_HD __host__ __device__ __forceinline__
#else
#define PERM_HD inline
#endif

namespace perm {

// A part whose sums are in its tour's row reports its depth and leaves.  Returns whether
// it was the tour's last part; `depth` is then the deepest length of all of them.  The
// depth is read after the count of parts has said so: every other part reported its own
// before it left.  (The value that deepen() found is older than the count: a deeper part
// may report between the two and leave first.)
//   Row: deepen(n) depth <- max(depth, n); leave() one part fewer, returns the parts there
//   were; depth(); fence() orders this thread's accesses at the scope of the parts.
template <class Row>
PERM_HD bool end_part(Row &row, unsigned maxn, unsigned &depth) {
    row.deepen(maxn);
    row.fence();
    const unsigned parts = row.leave();
    row.fence();
    if (parts != 1u) return false;
    depth = row.depth();
    return true;
}

// Tour tickets that a warp fetches beyond those its walks need now, at most `most`: a warp
// keeps what it has fetched, so no more than half of a walk's even share of the tours
// that the launch has left to start.
PERM_HD unsigned tickets_ahead(long long left, long long walks, unsigned most) {
    if (left >= 2 * walks * (long long)(most + 1u)) return most;
    const long long half = left / (2 * walks);
    return half > 1 ? (unsigned)(half - 1) : 0u;
}

}  // namespace perm
