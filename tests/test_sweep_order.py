"""The rule on the order of FP32 sums (csrc/vegas_order.h) on the host: which sweeps the tiled one may
stand for."""

import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1803_07030_gb300", "csrc")

# columns, widest class, sites, replicas, run of the tile; sweep, sites of a class it takes at once -> stands for it
CASES = [
    ((1, 847, 1694, 1, 2), 1, 512, 0),        # a resident block adds two sites of the class per thread
    ((1, 300, 600, 1, 2), 1, 256, 0),         # so does one of 256 threads with a class of 300
    ((1, 256, 512, 1, 2), 1, 256, 1),
    ((1, 300, 600, 1, 2), 1, 512, 1),
    ((1, 2746, 5491, 1, 2), 3, 2048, 0),      # a cluster of four blocks of 512
    ((1, 2048, 4096, 8, 2), 3, 2048, 1),
    ((1, 3300, 13000, 8, 4), 2, 4864, 1),     # the cooperative grid, a thread per site
    ((1, 3300, 13000, 8, 4), 2, 2432, 0),
    ((0, 5324, 10648, 16, 4), 2, 9728, 0),    # parts of several rounds, several replicas
    ((0, 131072, 262144, 1, 4), 2, 77824, 1),  # one replica, a large sample
    ((0, 131072, 262144, 1, 4), 1, 512, 0),
    ((0, 13500, 27000, 1, 28), 2, 512, 0),    # few blocks: long runs on a small sample
    ((1, 256, 512, 1, 2), 0, 512, 0),         # the per-class sweep adds class by class
    ((1, 256, 512, 32, 2), 4, 512, 0),
]


@pytest.mark.skipif(shutil.which("g++") is None, reason="no C++ compiler")
def test_tile_stands_for_sweeps_of_its_order(tmp_path):
    rows = ",\n".join("{{%s, %d, %d, %d, %d}, %d, %d, %d}" % (("true" if t[0] else "false",) + t[1:] + (v, once, want))
                      for t, v, once, want in CASES)
    src = tmp_path / "order.cpp"
    src.write_text('#include "vegas_order.h"\n#include <cstdio>\nstruct Case { vegas::TileOrder t; int v; long long once; int want; };\n'
                   "int main() {\n    const Case cases[] = {\n" + rows + "};\n"
                   "    for (const Case &c : cases) std::printf(\"%d\\n\", (int)vegas::tile_in_order(c.t, c.v, c.once));\n"
                   "    std::printf(\"%.3f %.3f\\n\", vegas::per_class_us(20.0, false), vegas::per_class_us(50.0, true));\n}\n")
    exe = tmp_path / "order"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    assert [int(x) for x in out[:len(CASES)]] == [c[3] for c in CASES]
    assert out[len(CASES)].split() == ["24.000", "62.000"]
