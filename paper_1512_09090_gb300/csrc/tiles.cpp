// Tile plan of the sweep (host side).
//
// PHAST's scanning phase (Section 2) may sweep vertices in any order in which
// every vertex follows the sources of its downward arcs.  Swept level by level,
// every arc fetches its source's label row from L2 or HBM: 4.9 rows per vertex.
// Here the vertices below the per-lane core are cut into tiles that need few
// rows from outside: a tile's vertices are swept by one CTA out of shared
// memory, rows read by several of its arcs are fetched once, and rows read only
// inside it are never written out.  On the 18M-vertex grid, 64 lanes, a
// tile holds 50 vertices; all tiles together fetch 1.2 rows per vertex and store
// 0.35.
//
// Tiers.  Going up from the lowest level, a vertex joins the tier of its
// successors (the heads of its outgoing downward arcs; the largest tier among
// them) and there merges the components that they belong to, as long as the
// merged component stays within lim.comp vertices; otherwise it starts the next
// tier.  So all successors of a vertex are in its own tier or a later-swept one,
// all arcs within a tier join vertices of one component, and components of one
// tier are independent: the sweep needs a barrier per tier (27 on the 18M grid
// at 64 lanes, 17 at one) instead of one per level or flags between chunks.
//
// Tiles.  Within a tier, a tile grows over components that share sources
// (starting from the first component left in BFS order), so that neighbouring
// components, which read the same rows, end up in one tile.  Own vertices of a
// tile are list-scheduled into phases (one CTA barrier each) of at most
// lim.width vertices, those with the longest chain of readers below them first,
// so that the CTA is full in most phases; within a phase they go by falling arc
// count, so that neighbouring threads do equal work.
//
// Tiers are split into jobs of consecutive components in BFS order that grow
// tiles independently (in parallel; the split does not depend on the number of
// threads, so the plan is the same on every machine).
//
// Time to build, 18M vertices on 8 cores: about 8 s at 64 lanes, 7 at one (a chunk
// schedule takes 2.6 and 1.3); 16 and 14 with the lists of successors, the components and
// their order made by one core.  Everything but the tiers' loop is spread over the
// cores; that loop takes one vertex after another and is bound by cache misses, so
// what it reads of a vertex lies in one record that is fetched ahead.
#include "tiles.h"

#include <algorithm>
#include <atomic>
#include <new>
#include <utility>

namespace {

constexpr int kJobVertices = 250000;  // vertices per job: bands of the map far wider than a tile
constexpr int kMaxMisses = 8;         // components that did not fit before a tile is closed
constexpr uint32_t kNever = 0x7FFFFFFFu;

// Small set of positions with the order of insertion (the rows from outside).
struct RowSet {
    std::vector<int32_t> key, val, list;
    std::vector<uint32_t> at;  // slots of the list's keys
    uint32_t mask;
    explicit RowSet(int cap) {
        uint32_t s = 64;
        while (s < 4u * (uint32_t)cap) s <<= 1;
        key.assign(s, -1);
        val.assign(s, 0);
        mask = s - 1;
    }
    uint32_t slot(int32_t k) const {
        uint32_t s = ((uint32_t)k * 0x9E3779B1u) & mask;
        while (key[s] != -1 && key[s] != k) s = (s + 1) & mask;
        return s;
    }
    void add(int32_t k) {
        const uint32_t s = slot(k);
        if (key[s] == k) return;
        key[s] = k;
        list.push_back(k);
        at.push_back(s);
    }
    // Takes out all but the first `size` keys; the last ones in go first, so that no
    // probe sequence of a key that stays is cut.
    void shrink(size_t size) {
        while (list.size() > size) {
            key[at.back()] = -1;
            at.pop_back();
            list.pop_back();
        }
    }
};

// A vertex while tiers are formed: its parent in its component's tree and its tier; of
// a component's root also the component's vertices and arcs.
struct alignas(16) Node {
    int32_t parent, size, arcs, tier;
};

struct Job {
    int tier;
    int32_t lo, hi;  // components by_order[lo .. hi)
    std::vector<uint32_t> dir;
    Raw<uint32_t> blob;
    int max_arcs = 0, max_ext = 0;
    bool ok = true, no_memory = false;
};

// Small lists whose entries were put in any order, sorted (in parallel).
void sort_lists(const std::vector<int32_t>& off, Raw<int32_t>& list) {
#pragma omp parallel for schedule(dynamic, 4096)
    for (int64_t i = 0; i < (int64_t)off.size() - 1; ++i) std::sort(list.begin() + off[i], list.begin() + off[i + 1]);
}

// Heads of the arcs by source, ascending for each: so[n + 1], succ; and node[v] of a
// vertex alone.
void by_source(int n, const uint32_t* down_off, const int32_t* down_src, const int32_t* down_len, Raw<uint32_t>& so,
               Raw<int32_t>& succ, Raw<Node>& node) {
    struct Arc { int32_t src, head; };
    const std::vector<int> cut = equal_parts(n, down_off);
    Dealt<Arc> by;
    deal<Arc>(n, [&](int q, auto give) {
        for (int v = cut[q]; v < cut[q + 1]; ++v) {
            int32_t arcs = 0;
            for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a)
                if ((uint32_t)down_len[a] < kNever) { give(down_src[a], Arc{down_src[a], v}); ++arcs; }
            node[v] = {v, 1, arcs, 0};
        }
    }, &by);
    succ.resize(std::max<size_t>(by.rec.size(), 1));
#pragma omp parallel for schedule(dynamic, 1)
    for (int r = 0; r < by.ranges; ++r) {
        const int lo = r << by.shift, hi = (int)std::min<int64_t>(n, (int64_t)(r + 1) << by.shift);
        for (int u = lo; u < hi; ++u) so[u] = 0;
        for (uint32_t i = by.at[r]; i < by.at[r + 1]; ++i) ++so[by.rec[i].src];
        uint32_t end = by.at[r];
        for (int u = lo; u < hi; ++u) so[u] = end += so[u];
        for (uint32_t i = by.at[r + 1]; i-- > by.at[r];) succ[--so[by.rec[i].src]] = by.rec[i].head;
    }
    so[n] = by.at[by.ranges];
}

}  // namespace

int iso_make_tiles(int n, int L, const int32_t* level_off, const uint32_t* down_off, const int32_t* down_src,
                   const int32_t* down_len, const int32_t* bfs, int core_n, const TileLimits& lim, TilePlan* out) {
    if (n <= 0 || L <= 0 || core_n < 0 || core_n > n || lim.rows < 2 || lim.rows >= (int)kTileNoRow || lim.comp < 1 ||
        lim.width < 1 || (lim.arcs != 2 && lim.arcs != 4) ||
        lim.blob_bytes < 64)
        return -1;
    const uint32_t m = down_off[n];
    *out = TilePlan();
    // successors (heads by source, ascending); arcs that can never lower a label are no dependencies
    Raw<uint32_t> so((size_t)n + 1);
    Raw<int32_t> succ;
    Raw<Node> node(n);
    by_source(n, down_off, down_src, down_len, so, succ, node);
    // tiers (0 = swept last) and components, from the lowest level up
    auto find = [&](int32_t x) {
        while (node[x].parent != x) { node[x].parent = node[node[x].parent].parent; x = node[x].parent; }
        return x;
    };
    int tiers = core_n < n ? 1 : 0;
    {
        constexpr int kAhead = 24;  // vertices whose successors' records are on their way (their parents': half that)
        std::vector<int32_t> roots;
        for (int u = n - 1; u >= core_n; --u) {
            if (u - kAhead >= core_n)
                for (uint32_t i = so[u - kAhead]; i < so[u - kAhead + 1]; ++i) __builtin_prefetch(&node[succ[i]], 1);
            if (u - kAhead / 2 >= core_n)
                for (uint32_t i = so[u - kAhead / 2]; i < so[u - kAhead / 2 + 1]; ++i)
                    __builtin_prefetch(&node[node[succ[i]].parent], 1);
            int t = 0;
            for (uint32_t i = so[u]; i < so[u + 1]; ++i) t = std::max(t, node[succ[i]].tier);
            roots.clear();
            int64_t sum = 1, arcs = node[u].arcs;
            for (uint32_t i = so[u]; i < so[u + 1] && sum <= lim.comp && arcs <= lim.rows; ++i) {
                if (node[succ[i]].tier != t) continue;
                const int32_t r = find(succ[i]);
                if (std::find(roots.begin(), roots.end(), r) != roots.end()) continue;
                roots.push_back(r);
                sum += node[r].size;
                arcs += node[r].arcs;
            }
            // (a vertex alone is placed in any case; the tile builder rejects it if it is too large)
            if (roots.empty() || (sum <= lim.comp && arcs <= lim.rows)) {
                int32_t top = u;
                for (int32_t r : roots)
                    if (node[r].size > node[top].size) top = r;
                for (int32_t r : roots) node[r].parent = top;
                node[u].parent = top;
                node[top].size = (int32_t)sum;
                node[top].arcs = (int32_t)std::min<int64_t>(arcs, INT32_MAX);
                node[u].tier = t;
            } else {
                node[u].tier = t + 1;
            }
            tiers = std::max(tiers, node[u].tier + 1);
        }
    }
    if (tiers > kTileMaxTiers) return -1;
    out->tiers = tiers;
    out->level_tier.assign(L, -1);
#pragma omp parallel for schedule(dynamic, 1)
    for (int j = 0; j < L; ++j)
        for (int v = std::max(level_off[j], core_n); v < level_off[j + 1]; ++v)
            out->level_tier[j] = std::max(out->level_tier[j], tiers - 1 - node[v].tier);
    // components, numbered by their first vertex, and their vertices in sweep order
    std::vector<int32_t> comp(n, -1), coff(1, 0), ctier;
    Raw<int32_t> cver((size_t)(n - core_n));
    int32_t nc = 0;
    {
        std::vector<int32_t> first(n, INT32_MAX);  // of each root
#pragma omp parallel for schedule(dynamic, 4096)
        for (int v = core_n; v < n; ++v) {
            int32_t r = v;
            while (node[r].parent != r) r = node[r].parent;
            comp[v] = r;
            int32_t seen = __atomic_load_n(&first[r], __ATOMIC_RELAXED);
            while (v < seen && !__atomic_compare_exchange_n(&first[r], &seen, v, true, __ATOMIC_RELAXED, __ATOMIC_RELAXED)) {}
        }
        Raw<int32_t> id(n);  // of each root
        for (int v = core_n; v < n; ++v)
            if (first[comp[v]] == v) {
                id[comp[v]] = nc++;
                coff.push_back(coff.back() + node[comp[v]].size);
                ctier.push_back(node[v].tier);
            }
        std::vector<int32_t> fill(coff.begin(), coff.end() - 1);
#pragma omp parallel for schedule(dynamic, 4096)
        for (int v = core_n; v < n; ++v) {
            comp[v] = id[comp[v]];
            cver[__atomic_fetch_add(&fill[comp[v]], 1, __ATOMIC_RELAXED)] = v;
        }
        sort_lists(coff, cver);
    }
    Raw<Node>().swap(node);
    // where each arc leads: to a vertex of its own component (kIn), to another (kOut), nowhere
    enum : uint8_t { kNone, kOut, kIn };
    Raw<uint8_t> kind(m);
    Raw<int32_t> scomp(succ.size());  // the successors' components (-1: core)
#pragma omp parallel for schedule(dynamic, 4096)
    for (int v = 0; v < n; ++v) {
        for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a)
            kind[a] = (uint32_t)down_len[a] >= kNever ? kNone : comp[v] >= 0 && comp[down_src[a]] == comp[v] ? kIn : kOut;
        for (uint32_t i = so[v]; i < so[v + 1]; ++i) scomp[i] = comp[succ[i]];
    }
    // jobs: runs of components of one tier in BFS order
    std::vector<int32_t> order(nc), job_of(nc);
    {
        std::vector<int32_t> at(tiers + 1, 0);
        for (int32_t c = 0; c < nc; ++c) at[tiers - ctier[c]]++;
        for (int t = 0; t < tiers; ++t) at[t + 1] += at[t];
        Raw<uint64_t> key(nc);  // rank of the first vertex, component
        {
            std::vector<int32_t> fill(at);
            for (int32_t c = 0; c < nc; ++c)
                key[fill[tiers - 1 - ctier[c]]++] = (uint64_t)(uint32_t)bfs[cver[coff[c]]] << 32 | (uint32_t)c;
        }
#pragma omp parallel for schedule(dynamic, 1)
        for (int t = 0; t < tiers; ++t) {
            std::sort(key.begin() + at[t], key.begin() + at[t + 1]);
            for (int32_t i = at[t]; i < at[t + 1]; ++i) order[i] = (int32_t)(uint32_t)key[i];
        }
    }
    std::vector<Job> jobs;
    for (int32_t i = 0; i < nc;) {
        const int t = ctier[order[i]];
        int32_t e = i;
        int64_t nv = 0;
        while (e < nc && ctier[order[e]] == t) { nv += coff[order[e] + 1] - coff[order[e]]; ++e; }
        const int64_t parts = std::max<int64_t>(1, nv / kJobVertices);
        int64_t seen = 0, part = 0;
        int32_t lo = i;
        for (int32_t c = i; c < e; ++c) {
            seen += coff[order[c] + 1] - coff[order[c]];
            job_of[order[c]] = (int32_t)jobs.size();
            if (c + 1 == e || seen * parts >= nv * (part + 1)) {
                Job j;
                j.tier = t;
                j.lo = lo;
                j.hi = c + 1;
                jobs.push_back(std::move(j));
                lo = c + 1;
                ++part;
            }
        }
        i = e;
    }
    // job of each component that is in no tile and no tile's queue, else -1 (a job changes
    // those of its own components; others may look at them meanwhile)
    std::vector<int32_t> free_in(job_of);
    std::vector<uint8_t> done(nc, 0);
    auto is_free = [&](int32_t c, int32_t ji) { return __atomic_load_n(&free_in[c], __ATOMIC_RELAXED) == ji; };
    auto set_free = [&](int32_t c, int32_t ji) { __atomic_store_n(&free_in[c], ji, __ATOMIC_RELAXED); };
    Raw<int32_t> row(n), height(n), open(n);
    std::atomic<bool> failed{false};
#pragma omp parallel for schedule(dynamic, 1)
    for (int32_t ji = 0; ji < (int32_t)jobs.size(); ++ji) {
        if (failed.load()) continue;
        Job& job = jobs[ji];
        try {
            RowSet ext(lim.rows);
            std::vector<int32_t> queue, own, heap, placed, rows;
            std::vector<uint32_t> ends, w;
            int32_t seed = job.lo;
            while (true) {
                while (seed < job.hi && done[order[seed]]) ++seed;
                if (seed == job.hi) break;
                ext.shrink(0);
                queue.clear();
                own.clear();
                int inner = 0, misses = 0;
                int64_t arcs = 0;
                size_t qh = 0;
                int32_t next_seed = seed;
                while (misses < kMaxMisses) {
                    int32_t c;
                    if (qh < queue.size()) {
                        c = queue[qh++];
                    } else {  // nothing next to the tile is left: go on with the next component in BFS order
                        while (next_seed < job.hi && !is_free(order[next_seed], ji)) ++next_seed;
                        if (next_seed == job.hi) break;
                        c = order[next_seed];
                        set_free(c, -1);
                        queue.push_back(c);
                        qh = queue.size();
                    }
                    // what the next components and this one's arcs take comes while others are looked at
                    if (qh + 1 < queue.size()) __builtin_prefetch(cver.data() + coff[queue[qh + 1]]);
                    if (qh < queue.size())
                        for (int32_t i = coff[queue[qh]]; i < coff[queue[qh] + 1]; ++i) {
                            __builtin_prefetch(down_off + cver[i]);
                            __builtin_prefetch(so.data() + cver[i]);
                        }
                    for (int32_t i = coff[c]; i < coff[c + 1]; ++i) {
                        __builtin_prefetch(down_src + down_off[cver[i]]);
                        __builtin_prefetch(kind.data() + down_off[cver[i]]);
                        __builtin_prefetch(scomp.data() + so[cver[i]]);
                    }
                    const size_t had = ext.list.size();
                    int in = 0;
                    int64_t ca = 0;  // (a multiple of lim.arcs for each vertex)
                    for (int32_t i = coff[c]; i < coff[c + 1]; ++i) {
                        const int32_t v = cver[i];
                        for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                            if (scomp[s] == c) { ++in; break; }
                        // (far too many rows: given up at once, which keeps the set's table sparse)
                        for (uint32_t a = down_off[v]; a < down_off[v + 1] && (int)ext.list.size() <= 2 * lim.rows; ++a) {
                            if (kind[a] == kNone) continue;
                            ++ca;
                            if (kind[a] == kOut) ext.add(down_src[a]);
                        }
                        ca = (ca + lim.arcs - 1) / lim.arcs * lim.arcs;
                    }
                    const int64_t n_own = (int64_t)own.size() + coff[c + 1] - coff[c];
                    // (phases: full ones, and others that each shorten the longest path; three gaps)
                    const int64_t words = kTileHeader + std::min<int64_t>(n_own, lim.comp + n_own / lim.width + 1) +
                                          (int64_t)ext.list.size() + 2 * (n_own + 1) + 2 * (arcs + ca) + 7;
                    if ((int64_t)ext.list.size() + inner + in > lim.rows || words * 4 > lim.blob_bytes) {
                        if (own.empty()) { job.ok = false; break; }
                        ext.shrink(had);
                        ++misses;
                        continue;
                    }
                    done[c] = 1;
                    inner += in;
                    arcs += ca;
                    for (int32_t i = coff[c]; i < coff[c + 1]; ++i) own.push_back(cver[i]);
                    for (size_t k = had; k < ext.list.size(); ++k) __builtin_prefetch(so.data() + ext.list[k]);
                    for (size_t k = had; k < ext.list.size(); ++k) __builtin_prefetch(scomp.data() + so[ext.list[k]]);
                    for (size_t k = had; k < ext.list.size(); ++k)  // components that read its new rows too
                        for (uint32_t s = so[ext.list[k]]; s < so[ext.list[k] + 1]; ++s)
                            if (scomp[s] >= 0 && is_free(scomp[s], ji)) {
                                set_free(scomp[s], -1);
                                queue.push_back(scomp[s]);
                            }
                }
                for (int32_t c : queue)
                    if (!done[c]) set_free(c, ji);
                if (!job.ok) break;
                // the record: rows from outside by position, own vertices by phase
                rows = ext.list;
                std::sort(rows.begin(), rows.end());
                for (size_t i = 0; i < rows.size(); ++i) ext.val[ext.slot(rows[i])] = (int32_t)i;
                // phases by list scheduling: height[v] = arcs of the longest path
                // from v inside the tile, open[v] = sources not scheduled yet
                std::sort(own.begin(), own.end());
                for (size_t i = own.size(); i-- > 0;) {
                    const int32_t v = own[i];
                    int h = 0;
                    for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                        if (scomp[s] == comp[v]) h = std::max(h, height[succ[s]] + 1);
                    height[v] = h;
                    open[v] = 0;
                    for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a)
                        open[v] += kind[a] == kIn;
                }
                auto degree = [&](int32_t v) { return (int)(down_off[v + 1] - down_off[v]); };
                auto later = [&](int32_t a, int32_t b) {  // heap order: the first to schedule on top
                    if (height[a] != height[b]) return height[a] < height[b];
                    return degree(a) != degree(b) ? degree(a) < degree(b) : a > b;
                };
                heap.clear();
                for (int32_t v : own)
                    if (open[v] == 0) heap.push_back(v);
                std::make_heap(heap.begin(), heap.end(), later);
                placed.clear();
                ends.clear();
                while (!heap.empty()) {
                    const size_t p0 = placed.size();
                    while (!heap.empty() && (int)(placed.size() - p0) < lim.width) {
                        std::pop_heap(heap.begin(), heap.end(), later);
                        placed.push_back(heap.back());
                        heap.pop_back();
                    }
                    std::sort(placed.begin() + p0, placed.end(), [&](int32_t a, int32_t b) {
                        return degree(a) != degree(b) ? degree(a) > degree(b) : a < b;
                    });
                    for (size_t i = p0; i < placed.size(); ++i) {
                        const int32_t v = placed[i];
                        for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                            if (scomp[s] == comp[v] && --open[succ[s]] == 0) {
                                heap.push_back(succ[s]);
                                std::push_heap(heap.begin(), heap.end(), later);
                            }
                    }
                    ends.push_back((uint32_t)placed.size());
                }
                uint32_t next_row = (uint32_t)rows.size();
                const int n_own = (int)placed.size();
                w.assign(kTileHeader, 0u);
                w.insert(w.end(), ends.begin(), ends.end());
                for (int32_t u : rows) w.push_back((uint32_t)u);
                if (w.size() & 1) w.push_back(0u);
                const size_t vert = w.size();
                w.resize((vert + 2 * ((size_t)n_own + 1) + 3) & ~(size_t)3);
                const size_t arc = w.size();
                uint32_t at = 0;
                for (int i = 0; i < n_own; ++i) {
                    const int32_t v = placed[i];
                    bool inside = false, outside = false;
                    for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                        (scomp[s] == comp[v] ? inside : outside) = true;
                    row[v] = inside ? (int32_t)next_row++ : (int32_t)kTileNoRow;
                    w[vert + 2 * i] = (uint32_t)v | (outside ? kTileStore : 0u);
                    w[vert + 2 * i + 1] = at | ((uint32_t)row[v] << 16);
                    for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a) {
                        if (kind[a] == kNone) continue;
                        const int32_t u = down_src[a];
                        w.push_back(kind[a] == kIn ? (uint32_t)row[u] : (uint32_t)ext.val[ext.slot(u)]);
                        w.push_back((uint32_t)down_len[a]);
                        ++at;
                    }
                    for (; at % (uint32_t)lim.arcs; ++at) {  // the last arc's row again
                        w.push_back(w[w.size() - 2]);
                        w.push_back(kNever);
                    }
                }
                w[vert + 2 * n_own] = 0;
                w[vert + 2 * n_own + 1] = at;
                while (w.size() & 3) w.push_back(0u);
                w[0] = (uint32_t)rows.size();
                w[1] = (uint32_t)n_own;
                w[2] = (uint32_t)ends.size();
                w[3] = (uint32_t)vert;
                w[4] = (uint32_t)arc;
                job.dir.push_back((uint32_t)(job.blob.size() / 4));
                job.dir.push_back((uint32_t)(w.size() * 4));
                job.blob.insert(job.blob.end(), w.begin(), w.end());
                job.max_arcs = std::max(job.max_arcs, (int)at);
                job.max_ext = std::max(job.max_ext, (int)rows.size());
            }
        } catch (const std::bad_alloc&) {
            job.ok = false;
            job.no_memory = true;
        }
        if (!job.ok) failed.store(true);
    }
    if (failed.load()) {
        // (a job that found a vertex too large says so whatever became of the others)
        for (const Job& j : jobs)
            if (!j.ok && !j.no_memory) return -1;
        return -2;
    }
    // jobs are in sweep order (highest tier first): join their records
    out->tier_off.assign((size_t)tiers + 1, 0);
    size_t words = 0, tiles = 0;
    for (const Job& j : jobs) {
        words += j.blob.size();
        tiles += j.dir.size() / 2;
        out->tier_off[tiers - j.tier] += (int32_t)(j.dir.size() / 2);
    }
    for (int t = 0; t < tiers; ++t) out->tier_off[t + 1] += out->tier_off[t];
    out->dir.resize(2 * tiles);
    out->blob.resize(words);
    std::vector<size_t> first_word(1, 0), first_tile(1, 0);  // of each job
    for (const Job& j : jobs) {
        first_word.push_back(first_word.back() + j.blob.size());
        first_tile.push_back(first_tile.back() + j.dir.size() / 2);
        out->max_arcs = std::max(out->max_arcs, j.max_arcs);
        out->max_ext = std::max(out->max_ext, j.max_ext);
    }
#pragma omp parallel for schedule(dynamic, 1)
    for (int32_t ji = 0; ji < (int32_t)jobs.size(); ++ji) {
        Job& j = jobs[ji];
        for (size_t i = 0; i < j.dir.size(); i += 2) {
            out->dir[2 * first_tile[ji] + i] = j.dir[i] + (uint32_t)(first_word[ji] / 4);
            out->dir[2 * first_tile[ji] + i + 1] = j.dir[i + 1];
        }
        std::copy(j.blob.begin(), j.blob.end(), out->blob.begin() + first_word[ji]);
        Raw<uint32_t>().swap(j.blob);
    }
    return 0;
}
