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
    // arcs by owner's rank: {other endpoint's rank, id}
    std::vector<uint32_t> start((size_t)n + 1, 0);
    std::vector<int32_t> at(n);  // sweep position of each rank
    for (int v = 0; v < n; ++v) at[bfs[v]] = v;
    for (int v = 0; v < n; ++v)
        for (int64_t a = orig_off[v]; a < orig_off[v + 1]; ++a)
            if (orig_head[a] != v) start[std::min(bfs[v], bfs[orig_head[a]]) + 1]++;
    for (int r = 0; r < n; ++r) start[r + 1] += start[r];
    std::vector<std::pair<int32_t, int32_t>> arc(start[n]);
    {
        std::vector<uint32_t> fill(start.begin(), start.end() - 1);
        for (int r = 0; r < n; ++r) {  // by rank, so that the writes stay close together
            const int v = at[r];
            for (int64_t a = orig_off[v]; a < orig_off[v + 1]; ++a) {
                const int h = bfs[orig_head[a]];
                if (h != r) arc[fill[std::min(r, h)]++] = {std::max(r, h), orig_id[a]};
            }
        }
    }
    out->off.assign((size_t)n + 1, 0);
#pragma omp parallel for schedule(static)
    for (int r = 0; r < n; ++r) {
        std::sort(arc.begin() + start[r], arc.begin() + start[r + 1]);
        uint32_t pairs = 0;
        for (uint32_t a = start[r]; a < start[r + 1]; ++pairs)
            a += a + 1 < start[r + 1] && arc[a].first == arc[a + 1].first ? 2 : 1;
        out->off[r + 1] = pairs;
    }
    for (int r = 0; r < n; ++r) out->off[r + 1] += out->off[r];
    const size_t pairs = std::max<size_t>(out->off[n], 1);
    out->head.assign(pairs, 0);
    out->ids.assign(2 * pairs, -1);
#pragma omp parallel for schedule(static)
    for (int r = 0; r < n; ++r) {
        uint32_t o = out->off[r];
        for (uint32_t a = start[r]; a < start[r + 1]; ++o) {
            const bool two = a + 1 < start[r + 1] && arc[a].first == arc[a + 1].first;
            out->head[o] = at[arc[a].first];
            out->ids[2 * (size_t)o] = arc[a].second;
            if (two) out->ids[2 * (size_t)o + 1] = arc[a + 1].second;
            a += two ? 2 : 1;
        }
    }
}
