"""Host test of the tile plan of the sweep (csrc/tiles.cpp).

A small C++ driver links tiles.cpp, builds plans for random hierarchies (any
arcs from higher to lower levels, parallel and never-lowering ones among them)
and checks the records against what the kernel relies on: every vertex below
the core in exactly one tile, rows from outside final before the tile's tier,
rows and record sizes within the limits, arcs of a phase only from outside or
from earlier phases, rows stored exactly where another tile reads them.  It
then sweeps the records the way the kernel does, from poisoned shared memory,
and compares every label with a plain scan in sweep order (integers: equal)."""

import os
import shutil
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1512_09090_gb300", "csrc")

DRIVER = textwrap.dedent(r"""
    #include <algorithm>
    #include <cstdio>
    #include <cstdlib>
    #include <random>
    #include <vector>
    #include "tiles.h"

    static int fail(const char* what, long a, long b) {
        std::printf("FAIL %s %ld %ld\n", what, a, b);
        return 1;
    }

    static int check(unsigned seed, int local, int core_levels, TileLimits lim, bool must_fail) {
        std::mt19937 rng(seed);
        const int L = 2 + (int)(rng() % 14);
        std::vector<int32_t> lo(L + 1, 0);
        for (int j = 0; j < L; ++j) lo[j + 1] = lo[j] + 1 + (int)(rng() % (j < 3 ? 4 : 400));
        const int n = lo[L];
        const int core_n = lo[std::min(core_levels, L)];
        std::vector<uint32_t> off(n + 5, 0);
        std::vector<int32_t> src, len;
        for (int j = 0; j < L; ++j)
            for (int v = lo[j]; v < lo[j + 1]; ++v) {
                off[v] = (uint32_t)src.size();
                for (int d = j ? (int)(rng() % 6) : 0; d > 0; --d) {
                    // near the vertex's own place in a random higher level, or anywhere above
                    const int k = (int)(rng() % (uint32_t)j);
                    const int w = lo[k + 1] - lo[k];
                    const long at = (long)(v - lo[j]) * w / (lo[j + 1] - lo[j]) + (long)(rng() % 5) - 2;
                    src.push_back(local ? lo[k] + (int)std::min<long>(std::max<long>(at, 0), w - 1)
                                        : (int32_t)(rng() % (uint32_t)lo[j]));
                    len.push_back(rng() % 9 == 0 ? 0x7FFFFFFF : (int32_t)(rng() % 100));
                }
            }
        for (int i = n; i < n + 5; ++i) off[i] = (uint32_t)src.size();
        std::vector<int32_t> bfs(n);
        for (int j = 0; j < L; ++j)
            for (int v = lo[j]; v < lo[j + 1]; ++v) bfs[v] = (int32_t)((long)(v - lo[j]) * n / (lo[j + 1] - lo[j]));
        TilePlan P;
        const int rc = iso_make_tiles(n, L, lo.data(), off.data(), src.data(), len.data(), bfs.data(), core_n, lim, &P);
        if (rc != 0) return must_fail ? 0 : fail("build", seed, rc);
        if (must_fail) return fail("built within limits that hold no vertex", seed, 0);

        // labels by the plain scan; start labels play the upward search's part
        const uint32_t inf = 0x7FFFFFFFu, poison = 0xDEADBEEFu;
        std::vector<uint32_t> start(n), want(n);
        for (int v = 0; v < n; ++v) start[v] = rng() % 7 == 0 ? rng() % 1000 : inf;
        for (int v = 0; v < n; ++v) {
            want[v] = start[v];
            for (uint32_t a = off[v]; a < off[v + 1]; ++a) want[v] = std::min(want[v], want[src[a]] + (uint32_t)len[a]);
        }
        std::vector<int> tier_of(n, -1), tile_of(n, -1), stored(n, 0), read_outside(n, 0);
        std::vector<uint32_t> rows(n, poison), got(n, poison);
        for (int v = 0; v < core_n; ++v) rows[v] = got[v] = want[v];
        if ((int)P.tier_off.size() != P.tiers + 1 || P.tier_off[0] != 0) return fail("tier offsets", seed, 0);
        for (int t = 0; t < P.tiers; ++t)
            for (int q = P.tier_off[t]; q < P.tier_off[t + 1]; ++q) {
                const uint32_t* r = P.blob.data() + (size_t)P.dir[2 * q] * 4;
                const uint32_t bytes = P.dir[2 * q + 1];
                if (bytes % 16 || (int)bytes > lim.blob_bytes) return fail("record bytes", q, bytes);
                const int n_ext = (int)r[0], n_own = (int)r[1], phases = (int)r[2];
                const uint32_t *ph = r + kTileHeader, *ext = ph + phases, *vert = r + r[3], *arc = r + r[4];
                if (r[3] % 2 || r[4] % 4 || n_own < 1) return fail("record layout", q, 0);
                std::vector<uint32_t> row(lim.rows, poison);
                std::vector<int> row_phase(lim.rows, 1 << 30);
                if (n_ext > lim.rows) return fail("rows from outside", q, n_ext);
                for (int i = 0; i < n_ext; ++i) {
                    const int u = (int)ext[i];
                    if (u >= core_n && (tier_of[u] < 0 || tier_of[u] >= t)) return fail("source not final", q, u);
                    if (u >= core_n) read_outside[u] = 1;
                    row[i] = rows[u];
                    row_phase[i] = -1;
                }
                int phase = 0;
                for (int j = 0; j < n_own; ++j) {
                    while (j >= (int)ph[phase]) ++phase;
                    const int v = (int)(vert[2 * j] & ~kTileStore);
                    if (v < core_n || tier_of[v] >= 0) return fail("vertex twice or in the core", q, v);
                    tier_of[v] = t;
                    tile_of[v] = q;
                    uint32_t x = start[v];
                    const uint32_t a0 = vert[2 * j + 1] & 0xFFFFu, a1 = vert[2 * j + 3] & 0xFFFFu;
                    for (uint32_t a = a0; a < a1; ++a) {
                        const uint32_t s = arc[2 * a];
                        if (a0 % lim.arcs || a1 % lim.arcs) return fail("padded arcs", q, a);
                        if ((int)s >= lim.rows || row_phase[s] >= phase) return fail("row of a later phase", q, s);
                        x = std::min(x, row[s] + arc[2 * a + 1]);
                    }
                    got[v] = x;
                    const uint32_t slot = vert[2 * j + 1] >> 16;
                    if (slot != kTileNoRow) {
                        if ((int)slot >= lim.rows || row_phase[slot] != (1 << 30)) return fail("row taken", q, slot);
                        row[slot] = x;
                        row_phase[slot] = phase;
                    }
                    if (vert[2 * j] & kTileStore) { rows[v] = x; stored[v] = 1; }
                }
                if ((int)ph[phases - 1] != n_own) return fail("phases", q, phases);
                for (int i = 0; i < phases; ++i)
                    if ((int)ph[i] - (i ? (int)ph[i - 1] : 0) > lim.width) return fail("phase width", q, i);
            }
        for (int v = core_n; v < n; ++v) {
            if (tier_of[v] < 0) return fail("vertex in no tile", v, 0);
            if (got[v] != want[v]) return fail("label", v, (long)got[v]);
            if (stored[v] != read_outside[v]) return fail("stored iff read elsewhere", v, stored[v]);
        }
        for (int j = 0; j < L; ++j) {
            int last = -1;
            for (int v = lo[j]; v < lo[j + 1]; ++v) last = std::max(last, tier_of[v]);
            if (P.level_tier[j] != last) return fail("level's last tier", j, P.level_tier[j]);
        }
        return 0;
    }

    int main() {
        const TileLimits sizes[] = {{200, 8192, 32, 16, 2}, {24, 768, 4, 3, 4}, {12, 640, 1, 1, 4}, {3000, 32768, 64, 128, 4}};
        for (unsigned seed = 1; seed <= 60; ++seed)
            for (const TileLimits& lim : sizes)
                for (int local = 0; local < 2; ++local)
                    if (check(seed, local, (int)(seed % 4), lim, false)) return 1;
        // a vertex with more sources than a tile has rows: no plan
        int none = 0;
        for (unsigned seed = 1; seed <= 20; ++seed) none += check(seed, 0, 0, TileLimits{2, 64, 1, 8, 2}, true);
        if (none) return 1;
        std::printf("OK\n");
        return 0;
    }
""")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_tile_plans(tmp_path):
    src = tmp_path / "driver.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.run(["g++", "-O1", "-g", "-std=c++17", "-fopenmp", "-fsanitize=address,undefined", "-I", CSRC, str(src),
                    os.path.join(CSRC, "tiles.cpp"), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300,
                       env={**os.environ, "ASAN_OPTIONS": "detect_leaks=0"})
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-500:] + r.stderr[-2000:]
