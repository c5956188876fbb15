"""Host test of the vertex pairs that emission walks (csrc/emit_pairs.cpp): on
random multigraphs every input arc but the self-loops appears in exactly one
pair, at its endpoint of lower BFS rank, next to the other endpoint's sweep
position, and both arcs of a two-way road share a pair."""

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
    #include <map>
    #include <random>
    #include <utility>
    #include <vector>
    #include "emit_pairs.h"

    int main() {
        for (unsigned seed = 1; seed <= 200; ++seed) {
            std::mt19937 rng(seed);
            const int n = 1 + (int)(rng() % 40);
            std::vector<int32_t> bfs(n);
            for (int v = 0; v < n; ++v) bfs[v] = v;
            std::shuffle(bfs.begin(), bfs.end(), rng);
            std::vector<int64_t> off(n + 1, 0);
            std::vector<int32_t> head, id, tail;
            for (int v = 0; v < n; ++v) {
                off[v] = (int64_t)head.size();
                for (int d = (int)(rng() % 7); d > 0; --d) {
                    tail.push_back(v);
                    head.push_back((int32_t)(rng() % (unsigned)n));
                    id.push_back((int32_t)id.size());
                }
            }
            off[n] = (int64_t)head.size();
            EmitPairs P;
            iso_make_emit_pairs(n, off.data(), head.data(), id.data(), bfs.data(), &P);
            std::vector<int> seen(id.size(), 0);
            std::map<std::pair<int, int>, std::pair<int, int>> count;  // arcs and pairs per couple of vertices
            for (int r = 0; r < n; ++r)
                for (uint32_t i = P.off[r]; i < P.off[r + 1]; ++i) {
                    const int h = bfs[P.head[i]];
                    if (h <= r || P.ids[2 * i] < 0) { std::printf("FAIL head\n"); return 1; }
                    count[{r, h}].second++;
                    for (int k = 0; k < 2; ++k) {
                        const int e = P.ids[2 * i + k];
                        if (e < 0) continue;
                        const int a = bfs[tail[e]], b = bfs[head[e]];
                        if (seen[e]++ || std::min(a, b) != r || std::max(a, b) != h) { std::printf("FAIL id\n"); return 1; }
                        count[{r, h}].first++;
                    }
                }
            for (size_t e = 0; e < id.size(); ++e)
                if (seen[e] != (tail[e] != head[e])) { std::printf("FAIL arc\n"); return 1; }
            for (auto& c : count)
                if (c.second.second != (c.second.first + 1) / 2) { std::printf("FAIL pairs\n"); return 1; }
        }
        std::printf("OK\n");
        return 0;
    }
""")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_emit_pairs(tmp_path):
    src = tmp_path / "driver.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.run(["g++", "-O1", "-g", "-std=c++17", "-fopenmp", "-fsanitize=address,undefined", "-I", CSRC, str(src),
                    os.path.join(CSRC, "emit_pairs.cpp"), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120,
                       env={**os.environ, "ASAN_OPTIONS": "detect_leaks=0"})
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-500:] + r.stderr[-2000:]
