// Every order in which the parts of one tour can end, on end_part of perm_parts.h.
//
// A part runs until its next access to the row: what it has done before is replayed from
// its record, then one access is made and the part is left (an exception).  So the accesses
// of all parts can be put in any order.  Prints "ok <orders>" or the first order after
// which the last part's depth is not the deepest one.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "perm_parts.h"

struct Shared { unsigned tmaxn, outst; };
struct Yield {};

struct Part {
    unsigned maxn;
    std::vector<unsigned> done;      // what its accesses returned
    bool ended = false, last = false;
    unsigned depth = 0u;
};

struct Row {
    Shared &s;
    Part &p;
    size_t at = 0;
    template <class F> unsigned access(F f) {
        if (at < p.done.size()) return p.done[at++];
        p.done.push_back(f());
        throw Yield();
    }
    void deepen(unsigned n) { access([&] { const unsigned o = s.tmaxn; s.tmaxn = std::max(o, n); return o; }); }
    unsigned leave() { return access([&] { return s.outst--; }); }
    unsigned depth() { return access([&] { return s.tmaxn; }); }
    void fence() {}
};

static long orders = 0;

static void explore(const Shared &s, const std::vector<Part> &parts, unsigned deepest, const std::string &order) {
    bool any = false;
    for (size_t i = 0; i < parts.size(); ++i) {
        if (parts[i].ended) continue;
        any = true;
        Shared t = s;
        std::vector<Part> q = parts;
        Row row{t, q[i]};
        try {
            q[i].last = perm::end_part(row, q[i].maxn, q[i].depth);
            q[i].ended = true;
        } catch (const Yield &) {
        }
        explore(t, q, deepest, order + (char)('A' + i));
    }
    if (any) return;
    ++orders;
    int last = 0;
    bool good = true;
    for (const Part &p : parts)
        if (p.last) { ++last; good = good && p.depth == deepest; }
    if (last != 1 || !good) {
        std::printf("order %s: %d last parts, depth %s\n", order.c_str(), last, good ? "right" : "too small");
        std::exit(1);
    }
}

int main() {
    for (unsigned n = 1; n <= 3; ++n) {
        std::vector<unsigned> depths;
        for (unsigned i = 0; i < n; ++i) depths.push_back(3u + i);
        do {
            std::vector<Part> parts(n);
            for (unsigned i = 0; i < n; ++i) parts[i].maxn = depths[i];
            explore(Shared{0u, n}, parts, 2u + n, "");
        } while (std::next_permutation(depths.begin(), depths.end()));
    }
    std::printf("ok %ld\n", orders);
    return 0;
}
