"""Which bands k_step_cluster's blocks take (csrc/cluster_layout.hpp, compiled by the host's
C++ compiler): the bytes of a block against the same sums in Python's integers, which do not wrap,
over the bands of every cluster size and both splits.  No grid whose values alone exceed a
block's shared memory may fit, however large it is."""
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1911_00180_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "cluster_layout.hpp"
int main() {
  int q, per, minor, es;
  while (std::scanf("%d %d %d %d", &q, &per, &minor, &es) == 4)
    std::printf("%llu %d\n", (unsigned long long)wlbm::cl_bytes(q, per, minor, es),
                wlbm::cl_fits(q, per, minor, es) ? 1 : 0);
}
"""
SMEM = 227 * 1024
# blocks whose sums in 32 bits come out below SMEM, and the largest frame a grid may have
WRAP = [(448, 4416, 532, 2), (128, 3072, 2684, 4), (96, 11008, 7936, 4), (512, 46338, 46338, 4)]


def _bytes(q, per, minor, es):
    up = lambda n: (n + 15) // 16 * 16  # noqa: E731
    lines, line = per + 2, (minor + 2) | 1
    cells = lines * line
    n = 2 * q * up(cells * es) + up(8 * cells) + 2 * up(4 * cells)
    if es == 2:
        n += up(8 * cells) + up(4 * cells)
    return n + up(32 * q) + up(12 * q) + up(4 * q) + up(64 * max(lines, line))


@pytest.fixture(scope="module")
def fits(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fit")
    src, exe = d / "fit.cpp", d / "fit"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def ask(bands):
        text = "".join("%d %d %d %d\n" % b for b in bands)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return ask


def _bands(nx, ny, q, es):
    for nc in (16, 8, 4, 2, 1):
        for major, minor in ((ny, nx), (nx, ny)):
            yield q, -(-major // nc), minor, es


@pytest.mark.parametrize("kind", ["named", "small", "large"])
def test_fit_is_exact(fits, kind):
    rng = random.Random(5)
    if kind == "named":
        bands = [b for q, nx, ny, es in WRAP for b in _bands(nx, ny, q, es)]
    else:
        top = {"small": 2.8, "large": 4.6}[kind]
        bands = [b for _ in range(4000)
                 for b in _bands(int(10 ** rng.uniform(0, top)), int(10 ** rng.uniform(0, top)),
                                 8 * rng.randint(1, 64), rng.choice((2, 4)))]
    for band, (got, fit) in zip(bands, fits(bands), strict=True):
        assert got == _bytes(*band), band
        assert fit == (got <= SMEM), band
        q, per, minor, es = band
        assert not (fit and 2 * q * (per + 2) * (minor + 2) * es > SMEM), band
    assert kind != "small" or sum(f for _, f in fits(bands)) > 1000   # both answers occur
