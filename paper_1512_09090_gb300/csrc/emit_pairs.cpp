// Input arcs as vertex pairs for emission (host side).
//
// An arc is an isochrone edge for a query iff exactly one endpoint is in range
// (Section 3), whichever way it points: both arcs of a two-way road cross
// together.  Emission therefore looks at each pair of vertices once and reports
// up to two arc ids for it (more arcs between two vertices make more pairs).
// Pairs are listed at the endpoint of lower BFS rank, which keeps the masks that
// neighbouring pairs read close together.
#include "emit_pairs.h"

#include <algorithm>
#include <utility>

void iso_make_emit_pairs(int n, const int64_t* orig_off, const int32_t* orig_head, const int32_t* orig_id,
                         const int32_t* bfs, EmitPairs* out) {
    // arcs by owner's rank (parts of the vertices deal them out by ranges of ranks, each
    // range is then put in order by itself)
    struct Arc { int32_t owner, other, id; };
    Dealt<Arc> by;
    {
        const std::vector<int> cut = equal_parts(n, orig_off);
        deal<Arc>(n, [&](int q, auto give) {
            for (int v = cut[q]; v < cut[q + 1]; ++v)
                for (int64_t a = orig_off[v]; a < orig_off[v + 1]; ++a) {
                    const int32_t r = bfs[v], h = bfs[orig_head[a]];
                    if (h != r) give(std::min(r, h), Arc{std::min(r, h), std::max(r, h), orig_id[a]});
                }
        }, &by);
    }
    Raw<int32_t> at(n);  // sweep position of each rank
    Raw<uint32_t> start((size_t)n + 1);
    Raw<std::pair<int32_t, int32_t>> arc(by.rec.size());  // {other endpoint's rank, id}
    out->off.assign((size_t)n + 1, 0);
#pragma omp parallel for schedule(static)
    for (int v = 0; v < n; ++v) at[bfs[v]] = v;
#pragma omp parallel for schedule(dynamic, 1)
    for (int q = 0; q < by.ranges; ++q) {
        const int lo = q << by.shift, hi = (int)std::min<int64_t>(n, (int64_t)(q + 1) << by.shift);
        for (int r = lo; r < hi; ++r) start[r] = 0;
        for (uint32_t i = by.at[q]; i < by.at[q + 1]; ++i) ++start[by.rec[i].owner];
        uint32_t end = by.at[q];
        for (int r = lo; r < hi; ++r) start[r] = end += start[r];
        for (uint32_t i = by.at[q]; i < by.at[q + 1]; ++i)
            arc[--start[by.rec[i].owner]] = {by.rec[i].other, by.rec[i].id};
        for (int r = lo; r < hi; ++r) {
            const uint32_t e = r + 1 < hi ? start[r + 1] : by.at[q + 1];
            std::sort(arc.begin() + start[r], arc.begin() + e);
            uint32_t pairs = 0;
            for (uint32_t a = start[r]; a < e; ++pairs) a += a + 1 < e && arc[a].first == arc[a + 1].first ? 2 : 1;
            out->off[r + 1] = pairs;
        }
    }
    start[n] = by.at[by.ranges];
    for (int r = 0; r < n; ++r) out->off[r + 1] += out->off[r];
    const size_t pairs = out->off[n];
    out->head.resize(std::max<size_t>(pairs, 1));
    out->ids.resize(2 * std::max<size_t>(pairs, 1));
    if (pairs == 0) { out->head[0] = 0; out->ids[0] = out->ids[1] = -1; }
#pragma omp parallel for schedule(dynamic, 4096)
    for (int r = 0; r < n; ++r) {
        uint32_t o = out->off[r];
        for (uint32_t a = start[r]; a < start[r + 1]; ++o) {
            const bool two = a + 1 < start[r + 1] && arc[a].first == arc[a + 1].first;
            out->head[o] = at[arc[a].first];
            out->ids[2 * (size_t)o] = arc[a].second;
            out->ids[2 * (size_t)o + 1] = two ? arc[a + 1].second : -1;
            a += two ? 2 : 1;
        }
    }
}
