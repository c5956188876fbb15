// Host arrays of the graph's set-up: uninitialised vectors, and records dealt out by
// ranges of keys so that each range can be ordered in cache, in parallel.
#pragma once

#include <algorithm>
#include <cstdint>
#include <memory>
#include <new>
#include <utility>
#include <vector>

// A vector's allocator that leaves new plain elements as they are: large arrays are
// then first touched by the threads that fill them, not zeroed by one.
template <class T>
struct NoInit : std::allocator<T> {
    template <class U> struct rebind { using other = NoInit<U>; };
    template <class U> void construct(U* p) { ::new ((void*)p) U; }
    template <class U, class... A> void construct(U* p, A&&... a) { ::new ((void*)p) U(std::forward<A>(a)...); }
};
template <class T> using Raw = std::vector<T, NoInit<T>>;

constexpr int kParts = 64;  // parts that a pass over a graph's arcs is cut into

// Vertices [cut[q], cut[q + 1]) have about a 64th of the arcs of the offsets off[0 .. n].
template <class Off>
std::vector<int> equal_parts(int n, const Off* off) {
    std::vector<int> cut(kParts + 1, n);
    cut[0] = 0;
    for (int q = 1; q < kParts; ++q) cut[q] = (int)(std::lower_bound(off, off + n, (Off)((uint64_t)off[n] * q / kParts)) - off);
    return cut;
}

// Records of keys [r << shift, (r + 1) << shift) lie at rec[at[r] .. at[r + 1]), those of
// one part in the order in which it gave them, parts in their order.
template <class Rec>
struct Dealt {
    int shift = 0, ranges = 0;
    std::vector<uint32_t> at;
    Raw<Rec> rec;
};

// visit(q, give) calls give(key, record) for each record of part q, keys in [0, n); it is
// called twice for every part, in parallel.  Fewer than 2^32 records.
template <class Rec, class Visit>
void deal(int n, Visit visit, Dealt<Rec>* out) {
    out->shift = 0;
    while (n >> out->shift >= 1024) ++out->shift;
    const int shift = out->shift, ranges = out->ranges = ((n - 1) >> shift) + 1;
    std::vector<uint32_t> to((size_t)kParts * ranges, 0);
#pragma omp parallel for schedule(dynamic, 1)
    for (int q = 0; q < kParts; ++q) {
        uint32_t* const count = to.data() + (size_t)q * ranges;
        visit(q, [&](int32_t key, const Rec&) { ++count[key >> shift]; });
    }
    out->at.assign(ranges + 1, 0);
    uint32_t total = 0;
    for (int r = 0; r < ranges; ++r) {
        out->at[r] = total;
        for (int q = 0; q < kParts; ++q) total += std::exchange(to[(size_t)q * ranges + r], total);
    }
    out->at[ranges] = total;
    out->rec.resize(total);
#pragma omp parallel for schedule(dynamic, 1)
    for (int q = 0; q < kParts; ++q) {
        uint32_t* const place = to.data() + (size_t)q * ranges;
        visit(q, [&](int32_t key, const Rec& r) { out->rec[place[key >> shift]++] = r; });
    }
}
