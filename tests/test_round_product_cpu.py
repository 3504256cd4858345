"""The start field's product (csrc/round_product.cuh, compiled by the host's C++ compiler with the
device's rounded operations in their place) against float32(float64(w) * dE), bit for bit: the
lattices' weights, deviations over the whole range of float64, products on and beside the ties
between two float32 values, where the split has to leave the decision to float64, and deviations
too small or too large to split.  That fallback must occur, and be rare for ordinary values."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import lattice as L

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1911_00180_gb300", "csrc")
MAIN = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
#define __noinline__
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
#include "round_product.cuh"
int main(int, char** v) {
  std::FILE* f = std::fopen(v[1], "rb");
  float w;
  double d;
  std::vector<float> out;
  long fallback = 0;
  while (std::fread(&w, 4, 1, f) == 1 && std::fread(&d, 8, 1, f) == 1) {
    const wlbm::SplitDouble x = wlbm::split_double(d);
    out.push_back(wlbm::round_product(w, x));   // and whether it left the product to float64:
    const float ph = w * x.hi, s = std::fmaf(w, x.lo, std::fmaf(w, x.hi, -ph));
    const float tol = std::fabs(ph) * 0x1p-44f;
    fallback += x.small || ph + (s - tol) != ph + (s + tol);
  }
  std::fwrite(out.data(), 4, out.size(), stdout);
  std::fprintf(stderr, "%ld\n", fallback);
}
"""


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("product")
    src, exe = d / "product.cpp", d / "product"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)

    def run(w, de):
        rec = np.zeros(len(w), np.dtype([("w", "<f4"), ("d", "<f8")]))
        rec["w"], rec["d"] = w, de
        (d / "in").write_bytes(rec.tobytes())
        p = subprocess.run([str(exe), str(d / "in")], capture_output=True, check=True)
        return np.frombuffer(p.stdout, np.float32), int(p.stderr)
    return run


def _weights(rng, n):
    w = np.concatenate([L.angular_weights(L.ring_directions(q)) for q in (8, 16, 40, 128, 1024)])
    return rng.choice(w.astype(np.float32), n)


def _inputs(kind, rng, n):
    w = _weights(rng, n)
    if kind == "ordinary":      # dE of start fields: 1e-13 to 1e3
        de = 10.0 ** rng.uniform(-13, 3, n)
    elif kind == "extreme":     # any exponent, subnormals, zero, infinities, NaN
        de = rng.integers(0, 1 << 63, n).view(np.float64)
        de[:6] = (0.0, 5e-324, np.inf, np.nan, 1e-18, 1e30)
    else:                       # w dE within a few units of float64 of a tie of float32
        m = rng.integers(1 << 23, 1 << 24, n).astype(np.float64) + 0.5
        de = m * 2.0 ** rng.integers(-45, -18, n) / w.astype(np.float64)
        de = (de.view(np.int64) + rng.integers(-4, 5, n)).view(np.float64)
    return w, np.copysign(de, rng.choice([-1.0, 1.0], n))


@pytest.mark.parametrize("kind", ["ordinary", "extreme", "ties"])
def test_product_has_the_bits_of_float64(product, kind):
    rng = np.random.default_rng(7)
    w, de = _inputs(kind, rng, 1 << 20)
    got, fallback = product(w, de)
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        want = (w.astype(np.float64) * de).astype(np.float32)
    same = (got.view(np.uint32) == want.view(np.uint32)) | (np.isnan(got) & np.isnan(want))
    assert np.all(same), (w[~same][:3], de[~same][:3], got[~same][:3], want[~same][:3])
    if kind == "ordinary":
        assert fallback < 40        # expected 2 in 2^20
    else:
        assert fallback > len(w) // 4
