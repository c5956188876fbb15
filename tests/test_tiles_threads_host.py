"""The tile plan does not depend on how many threads build it (csrc/tiles.cpp): plans of
a hierarchy of 700,000 vertices, several jobs to a tier, are compared byte for byte
between one, three and eight threads, in two lane classes' limits."""

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
    #include <random>
    #include <vector>
    #include "tiles.h"

    int main() {
        std::mt19937 rng(7);
        std::vector<int32_t> lo(1, 0);
        for (int w : {3, 40, 900, 9000, 30000, 120000, 240000, 300054}) lo.push_back(lo.back() + w);
        const int L = (int)lo.size() - 1, n = lo[L];
        std::vector<uint32_t> off(n + 1, 0);
        std::vector<int32_t> src, len, bfs(n);
        for (int j = 0; j < L; ++j)
            for (int v = lo[j]; v < lo[j + 1]; ++v) {
                off[v] = (uint32_t)src.size();
                for (int d = j ? (int)(rng() % 6) : 0; d > 0; --d) {
                    const int k = std::max(0, j - 1 - (int)(rng() % 3)), w = lo[k + 1] - lo[k];
                    const long at = (long)(v - lo[j]) * w / (lo[j + 1] - lo[j]) + (long)(rng() % 5) - 2;
                    src.push_back(lo[k] + (int)std::min<long>(std::max<long>(at, 0), w - 1));
                    len.push_back(rng() % 9 == 0 ? 0x7FFFFFFF : (int32_t)(rng() % 100));
                }
            }
        off[n] = (uint32_t)src.size();
        // ranks by place on the map, a permutation
        std::vector<std::pair<long, int32_t>> place;
        for (int j = 0; j < L; ++j)
            for (int v = lo[j]; v < lo[j + 1]; ++v) place.push_back({(long)(v - lo[j]) * n / (lo[j + 1] - lo[j]), v});
        std::sort(place.begin(), place.end());
        for (int r = 0; r < n; ++r) bfs[place[r].second] = r;
        for (const TileLimits& lim : {TileLimits{100, 6144, 16, 16, 2}, TileLimits{2500, 24576, 64, 128, 4}}) {
            TilePlan P;
            if (iso_make_tiles(n, L, lo.data(), off.data(), src.data(), len.data(), bfs.data(), lo[2], lim, &P)) return 1;
            unsigned long long h = 1469598103934665603ull;
            auto add = [&](const auto& v) { for (auto x : v) h = (h ^ (uint32_t)x) * 1099511628211ull; };
            add(P.tier_off); add(P.dir); add(P.blob); add(P.level_tier);
            std::printf("%d %d %d %d %llx\n", P.tiers, P.tier_off.back(), P.max_arcs, P.max_ext, h);
        }
        return 0;
    }
""")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_same_plan_on_any_number_of_threads(tmp_path):
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fopenmp", "-I", CSRC, str(src), os.path.join(CSRC, "tiles.cpp"),
                    "-o", str(exe)], check=True, capture_output=True, text=True)
    out = [subprocess.run([str(exe)], capture_output=True, text=True, timeout=300,
                          env={**os.environ, "OMP_NUM_THREADS": str(t)}) for t in (1, 3, 8)]
    assert all(r.returncode == 0 for r in out), out
    assert len(out[0].stdout.split()) == 10 and len({r.stdout for r in out}) == 1, [r.stdout for r in out]
