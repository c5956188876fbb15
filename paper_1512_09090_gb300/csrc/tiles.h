// Tile plan of the sweep, built on the host (tiles.cpp): the vertices below the
// per-lane core cut into tiles that a CTA sweeps out of its shared memory.
#pragma once

#include <cstdint>
#include <vector>

#include "host_arrays.h"

// What one tile may hold (the kernel's shared-memory layout, per lane class).
struct TileLimits {
    int rows;        // label rows in shared memory: sources from outside + own vertices read inside
    int blob_bytes;  // the tile's record (a multiple of 16)
    int comp;        // vertices of a component
    int width;       // vertices of a phase: what the CTA sweeps at once
    int arcs;        // a vertex's arcs are padded to a multiple of this (2 or 4)
};

// A tile's record, in 32-bit words (16-byte aligned and padded, one bulk copy):
//   [0] sources from outside (n_ext)   [1] own vertices (n_own)   [2] phases
//   [3] word of the first vertex record   [4] word of the first arc   [5..7] 0
//   phase ends: index one past each phase's last own vertex
//   n_ext sweep positions; source i is row i
//   n_own + 1 vertex records of two words (8-byte aligned), by phase:
//     {sweep position | kTileStore if another tile reads its row,
//      first arc | row << 16 (kTileNoRow: no own vertex of the tile reads it)}
//   arcs of two words: {source row, length}, grouped by own vertex, a multiple of
//   lim.arcs for each: a spare one has length 0x7FFFFFFF, which never lowers a
//   label, and the row of the arc before it
constexpr int kTileHeader = 8;
constexpr uint32_t kTileStore = 0x80000000u;
constexpr uint32_t kTileNoRow = 0xFFFFu;

constexpr int kTileMaxTiers = 511;  // a plan with more is not made (a barrier each)

struct TilePlan {
    int tiers = 0;
    std::vector<int32_t> tier_off;   // [tiers + 1] first tile of each tier, in sweep order
    std::vector<uint32_t> dir;       // per tile {record start / 16 bytes, record bytes}
    Raw<uint32_t> blob;              // the records
    std::vector<int32_t> level_tier; // [L] last tier with vertices of each level block (-1: core)
    int max_arcs = 0, max_ext = 0;   // extremes over the tiles
};

// Builds the plan for sweep positions [core_n, n).  down_off/src/len: incoming
// downward arcs by sweep position (arcs of length 0x7FFFFFFF never lower a
// label and are left out); bfs: spatial key of each position.  Returns 0;
// -1 if some vertex cannot be placed within the limits, whenever it is tried, or -2
// if memory ran out (the caller then uses the chunk schedule).
int iso_make_tiles(int n, int L, const int32_t* level_off, const uint32_t* down_off, const int32_t* down_src,
                   const int32_t* down_len, const int32_t* bfs, int core_n, const TileLimits& lim, TilePlan* out);
