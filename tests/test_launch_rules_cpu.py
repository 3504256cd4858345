"""Which periodic passes start as dependents of the kernel ahead of them (periodic_early in
csrc/wlbm_internal.hpp, compiled by the host's C++ compiler): in a replayed graph a pass straight
behind a step of many tiles, or one that is mostly columns, does not, whatever the grid's size."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1911_00180_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "wlbm_internal.hpp"
int main() {
  long long cells;
  int graph, after_pass, tiles, ny;
  while (std::scanf("%lld %d %d %d %d", &cells, &graph, &after_pass, &tiles, &ny) == 5)
    std::printf("%d\n", wlbm::periodic_early(cells, graph, after_pass, wlbm::few_tiles(tiles, ny)));
}
"""
CASES = [  # cells, in a graph, behind another boundary pass, tiles of the step, ny: early
    (64 * 64, 0, 0, 5, 64, 1), (256 * 3000, 0, 0, 430, 3000, 1), (1 << 21, 0, 1, 1184, 1024, 1),
    (2048 * 2048, 0, 0, 2352, 2048, 0), (3000 * 100, 1, 0, 192, 100, 1), (64 * 64, 1, 0, 5, 64, 1),
    (129 * 1800, 1, 0, 129, 1800, 0), (256 * 3000, 1, 0, 430, 3000, 0), (1 << 20, 1, 0, 592, 1024, 0),
    (256 * 3000, 1, 1, 430, 3000, 1), (2048 * 2048, 1, 1, 2352, 2048, 0)]


def test_periodic_pass_in_graphs(tmp_path):
    from paper_1911_00180_gb300 import build
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    try:
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    except RuntimeError:
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    text = "".join("%d %d %d %d %d\n" % c[:5] for c in CASES)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
    assert [int(v) for v in out.split()] == [c[5] for c in CASES]
