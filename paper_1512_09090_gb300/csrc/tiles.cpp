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
// tier are independent: the sweep needs a barrier per tier (20 on the
// 18M grid) instead of one per level or flags between chunks.
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
    bool has(int32_t k) const { return key[slot(k)] == k; }
    void add(int32_t k) { key[slot(k)] = k; list.push_back(k); }
    void clear() {
        // every probe sequence of the set's keys ends in the set, so clearing
        // the whole table is only needed where it is dense
        if (list.size() * 8 > key.size()) std::fill(key.begin(), key.end(), -1);
        else {
            std::vector<uint32_t> at;
            for (int32_t k : list) at.push_back(slot(k));
            for (uint32_t s : at) key[s] = -1;
        }
        list.clear();
    }
};

struct Job {
    int tier;
    int32_t lo, hi;  // components by_order[lo .. hi)
    std::vector<uint32_t> dir, blob;
    int max_arcs = 0, max_ext = 0;
    bool ok = true, no_memory = false;
};

}  // namespace

int iso_make_tiles(int n, int L, const int32_t* level_off, const uint32_t* down_off, const int32_t* down_src,
                   const int32_t* down_len, const int32_t* bfs, int core_n, const TileLimits& lim, TilePlan* out) {
    if (n <= 0 || L <= 0 || core_n < 0 || core_n > n || lim.rows < 2 || lim.rows >= (int)kTileNoRow || lim.comp < 1 ||
        lim.width < 1 || (lim.arcs != 2 && lim.arcs != 4) ||
        lim.blob_bytes < 64)
        return -1;
    const uint32_t m = down_off[n];
    *out = TilePlan();
    // successors (heads by source); arcs that can never lower a label are no dependencies
    std::vector<uint32_t> so((size_t)n + 1, 0);
    for (uint32_t a = 0; a < m; ++a)
        if ((uint32_t)down_len[a] < kNever) so[down_src[a] + 1]++;
    for (int v = 0; v < n; ++v) so[v + 1] += so[v];
    std::vector<int32_t> succ(std::max<uint32_t>(so[n], 1));
    {
        std::vector<uint32_t> fill(so.begin(), so.end() - 1);
        for (int v = 0; v < n; ++v)
            for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a)
                if ((uint32_t)down_len[a] < kNever) succ[fill[down_src[a]]++] = v;
    }
    // tiers (0 = swept last) and components, from the lowest level up
    std::vector<int32_t> parent(n), size(n, 1), arcs_of(n, 0), tier(n, 0);
    auto find = [&](int32_t x) {
        while (parent[x] != x) { parent[x] = parent[parent[x]]; x = parent[x]; }
        return x;
    };
    int tiers = core_n < n ? 1 : 0;
    {
        std::vector<int32_t> roots;
        for (int u = n - 1; u >= core_n; --u) {
            parent[u] = u;
            for (uint32_t a = down_off[u]; a < down_off[u + 1]; ++a) arcs_of[u] += (uint32_t)down_len[a] < kNever;
            int t = 0;
            for (uint32_t i = so[u]; i < so[u + 1]; ++i) t = std::max(t, tier[succ[i]]);
            roots.clear();
            int64_t sum = 1, arcs = arcs_of[u];
            for (uint32_t i = so[u]; i < so[u + 1] && sum <= lim.comp && arcs <= lim.rows; ++i) {
                if (tier[succ[i]] != t) continue;
                const int32_t r = find(succ[i]);
                if (std::find(roots.begin(), roots.end(), r) != roots.end()) continue;
                roots.push_back(r);
                sum += size[r];
                arcs += arcs_of[r];
            }
            // (a vertex alone is placed in any case; the tile builder rejects it if it is too large)
            if (roots.empty() || (sum <= lim.comp && arcs <= lim.rows)) {
                int32_t top = u;
                for (int32_t r : roots)
                    if (size[r] > size[top]) top = r;
                for (int32_t r : roots) parent[r] = top;
                parent[u] = top;
                size[top] = (int32_t)sum;
                arcs_of[top] = (int32_t)std::min<int64_t>(arcs, INT32_MAX);
                tier[u] = t;
            } else {
                tier[u] = t + 1;
            }
            tiers = std::max(tiers, tier[u] + 1);
        }
    }
    if (tiers > kTileMaxTiers) return -1;
    out->tiers = tiers;
    out->level_tier.assign(L, -1);
    for (int j = 0; j < L; ++j)
        for (int v = std::max(level_off[j], core_n); v < level_off[j + 1]; ++v)
            out->level_tier[j] = std::max(out->level_tier[j], tiers - 1 - tier[v]);
    // components, their vertices in sweep order
    std::vector<int32_t> comp(n, -1), coff(1, 0), cver((size_t)(n - core_n));
    int32_t nc = 0;
    {
        std::vector<int32_t>& id = size;  // reuse: component number of each root
        std::fill(id.begin(), id.end(), -1);
        for (int v = core_n; v < n; ++v) {
            const int32_t r = find(v);
            if (id[r] < 0) { id[r] = nc++; coff.push_back(0); }
            comp[v] = id[r];
            coff[comp[v] + 1]++;
        }
        for (int32_t c = 0; c < nc; ++c) coff[c + 1] += coff[c];
        std::vector<int32_t> fill(coff.begin(), coff.end() - 1);
        for (int v = core_n; v < n; ++v) cver[fill[comp[v]]++] = v;
    }
    // jobs: runs of components of one tier in BFS order
    std::vector<int32_t> order(nc), job_of(nc);
    for (int32_t c = 0; c < nc; ++c) order[c] = c;
    auto first = [&](int32_t c) { return cver[coff[c]]; };
    std::sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
        const int32_t va = first(a), vb = first(b);
        return tier[va] != tier[vb] ? tier[va] > tier[vb] : bfs[va] < bfs[vb];
    });
    std::vector<Job> jobs;
    for (int32_t i = 0; i < nc;) {
        const int t = tier[first(order[i])];
        int32_t e = i;
        int64_t nv = 0;
        while (e < nc && tier[first(order[e])] == t) { nv += coff[order[e] + 1] - coff[order[e]]; ++e; }
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
    std::vector<uint8_t> done(nc, 0), queued(nc, 0);
    std::vector<int32_t> row(n, 0), height(n, 0), open(n, 0);
    std::atomic<bool> failed{false};
#pragma omp parallel for schedule(dynamic, 1)
    for (int64_t ji = 0; ji < (int64_t)jobs.size(); ++ji) {
        if (failed.load()) continue;
        Job& job = jobs[ji];
        try {
            RowSet ext(lim.rows);
            std::vector<int32_t> queue, fresh, own, members;
            std::vector<int32_t> heap, placed;
            std::vector<uint32_t> ends;
            int32_t seed = job.lo;
            while (true) {
                while (seed < job.hi && done[order[seed]]) ++seed;
                if (seed == job.hi) break;
                ext.clear();
                queue.clear();
                own.clear();
                members.clear();
                int inner = 0, misses = 0;
                int64_t arcs = 0;
                size_t qh = 0;
                int32_t next_seed = seed;
                while (misses < kMaxMisses) {
                    int32_t c;
                    if (qh < queue.size()) {
                        c = queue[qh++];
                    } else {  // nothing next to the tile is left: go on with the next component in BFS order
                        while (next_seed < job.hi && (done[order[next_seed]] || queued[order[next_seed]])) ++next_seed;
                        if (next_seed == job.hi) break;
                        c = order[next_seed];
                        queued[c] = 1;
                        queue.push_back(c);
                        qh = queue.size();
                    }
                    if (done[c]) continue;
                    fresh.clear();
                    int in = 0;
                    int64_t ca = 0;  // (a multiple of lim.arcs for each vertex)
                    for (int32_t i = coff[c]; i < coff[c + 1]; ++i) {
                        const int32_t v = cver[i];
                        for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                            if (comp[succ[s]] == c) { ++in; break; }
                        // (far too many rows: given up at once, which keeps the set's table sparse)
                        for (uint32_t a = down_off[v]; a < down_off[v + 1] && (int)ext.list.size() <= 2 * lim.rows; ++a) {
                            if ((uint32_t)down_len[a] >= kNever) continue;
                            ++ca;
                            const int32_t u = down_src[a];
                            if (comp[u] != c && !ext.has(u)) { ext.add(u); fresh.push_back(u); }
                        }
                        ca = (ca + lim.arcs - 1) / lim.arcs * lim.arcs;
                    }
                    const int64_t n_own = (int64_t)own.size() + coff[c + 1] - coff[c];
                    // (phases: full ones, and others that each shorten the longest path; three gaps)
                    const int64_t words = kTileHeader + std::min<int64_t>(n_own, lim.comp + n_own / lim.width + 1) +
                                          (int64_t)ext.list.size() + 2 * (n_own + 1) + 2 * (arcs + ca) + 7;
                    if ((int64_t)ext.list.size() + inner + in > lim.rows || words * 4 > lim.blob_bytes) {
                        if (members.empty()) { job.ok = false; break; }
                        // take the fresh rows out again (they are the last ones added)
                        std::vector<int32_t> keep(ext.list.begin(), ext.list.end() - fresh.size());
                        ext.clear();
                        for (int32_t u : keep) ext.add(u);
                        ++misses;
                        continue;
                    }
                    done[c] = 1;
                    members.push_back(c);
                    inner += in;
                    arcs += ca;
                    for (int32_t i = coff[c]; i < coff[c + 1]; ++i) own.push_back(cver[i]);
                    for (int32_t u : fresh)
                        for (uint32_t s = so[u]; s < so[u + 1]; ++s) {
                            const int32_t d = comp[succ[s]];
                            if (d >= 0 && job_of[d] == (int32_t)ji && !done[d] && !queued[d]) {
                                queued[d] = 1;
                                queue.push_back(d);
                            }
                        }
                }
                for (int32_t c : queue) queued[c] = 0;
                if (!job.ok) break;
                // the record: rows from outside by position, own vertices by phase
                std::vector<int32_t> rows = ext.list;
                std::sort(rows.begin(), rows.end());
                for (size_t i = 0; i < rows.size(); ++i) ext.val[ext.slot(rows[i])] = (int32_t)i;
                // phases by list scheduling: height[v] = arcs of the longest path
                // from v inside the tile, open[v] = sources not scheduled yet
                std::sort(own.begin(), own.end());
                for (size_t i = own.size(); i-- > 0;) {
                    const int32_t v = own[i];
                    int h = 0;
                    for (uint32_t s = so[v]; s < so[v + 1]; ++s)
                        if (comp[succ[s]] == comp[v]) h = std::max(h, height[succ[s]] + 1);
                    height[v] = h;
                    open[v] = 0;
                    for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a)
                        open[v] += (uint32_t)down_len[a] < kNever && comp[down_src[a]] == comp[v];
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
                            if (comp[succ[s]] == comp[v] && --open[succ[s]] == 0) {
                                heap.push_back(succ[s]);
                                std::push_heap(heap.begin(), heap.end(), later);
                            }
                    }
                    ends.push_back((uint32_t)placed.size());
                }
                uint32_t next_row = (uint32_t)rows.size();
                const int n_own = (int)placed.size();
                std::vector<uint32_t> w(kTileHeader, 0u);
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
                        (comp[succ[s]] == comp[v] ? inside : outside) = true;
                    row[v] = inside ? (int32_t)next_row++ : (int32_t)kTileNoRow;
                    w[vert + 2 * i] = (uint32_t)v | (outside ? kTileStore : 0u);
                    w[vert + 2 * i + 1] = at | ((uint32_t)row[v] << 16);
                    for (uint32_t a = down_off[v]; a < down_off[v + 1]; ++a) {
                        if ((uint32_t)down_len[a] >= kNever) continue;
                        const int32_t u = down_src[a];
                        w.push_back(comp[u] == comp[v] ? (uint32_t)row[u] : (uint32_t)ext.val[ext.slot(u)]);
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
    out->dir.reserve(2 * tiles);
    out->blob.reserve(words);
    for (Job& j : jobs) {
        const uint32_t base = (uint32_t)(out->blob.size() / 4);
        for (size_t i = 0; i < j.dir.size(); i += 2) {
            out->dir.push_back(j.dir[i] + base);
            out->dir.push_back(j.dir[i + 1]);
        }
        out->blob.insert(out->blob.end(), j.blob.begin(), j.blob.end());
        out->max_arcs = std::max(out->max_arcs, j.max_arcs);
        out->max_ext = std::max(out->max_ext, j.max_ext);
        std::vector<uint32_t>().swap(j.blob);
    }
    return 0;
}
