// Input arcs as vertex pairs for emission, built on the host (emit_pairs.cpp).
#pragma once

#include <cstdint>
#include <vector>

#include "host_arrays.h"

// Pairs of vertices joined by input arcs, listed at the endpoint of lower BFS
// rank (the owner), in the order of the owners' ranks.
struct EmitPairs {
    std::vector<uint32_t> off;       // [n + 1] first pair of each owner, by BFS rank
    Raw<int32_t> head;               // the other endpoint's sweep position
    Raw<int32_t> ids;                // per pair {arc id, second arc id or -1}
};

// orig_off/head/id: input arcs grouped by tail, by sweep position; bfs: BFS rank of
// each position (a permutation).  Self-loops are left out: they never cross.
void iso_make_emit_pairs(int n, const int64_t* orig_off, const int32_t* orig_head, const int32_t* orig_id,
                         const int32_t* bfs, EmitPairs* out);
