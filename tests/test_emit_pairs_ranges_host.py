"""The vertex pairs of emission where the owners are ordered in ranges of several
(csrc/emit_pairs.cpp deals arcs out by ranges of ranks from 1,024 vertices on): the
driver of the small random multigraphs on sizes about that line and above it."""

import os
import shutil
import subprocess

import pytest

from test_emit_pairs_host import CSRC, DRIVER

SIZES = (1023, 1024, 1025, 2047, 2048, 5000, 70001)


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_ranges_of_owners(tmp_path):
    big = DRIVER.replace("seed <= 200", f"seed <= {len(SIZES)}")
    big = big.replace("const int n = 1 + (int)(rng() % 40);",
                      "const int n = (const int[]){" + ", ".join(map(str, SIZES)) + "}[seed - 1];")
    assert "seed <= 200" not in big and "% 40" not in big
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(big)
    subprocess.run(["g++", "-O1", "-g", "-std=c++17", "-fopenmp", "-fsanitize=address,undefined", "-I", CSRC, str(src),
                    os.path.join(CSRC, "emit_pairs.cpp"), "-o", str(exe)], check=True, capture_output=True, text=True)
    for threads in ("1", "8"):
        r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300,
                           env={**os.environ, "ASAN_OPTIONS": "detect_leaks=0", "OMP_NUM_THREADS": threads})
        assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-500:] + r.stderr[-2000:]
