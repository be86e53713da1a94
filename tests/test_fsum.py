"""The three-part FP32 sums of the correction's threshold against exact sums (CPU).

The header is host code as well as device code, so it is compiled here as it
is.  Bar: a sum of k values in any order in FP64 is off by at most
(k - 1) 2^-53 of the sum of absolute values; the three-part form must not be
further off, neither value by value nor joined from lanes.
"""
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <vector>
#include "fsum.hpp"
// stdin: k lanes; per row k * lanes floats; one line per row: the rows' sums, lanes joined as a warp joins them
int main() {
  int k, lanes, rows;
  if (std::fread(&k, 4, 1, stdin) != 1 || std::fread(&lanes, 4, 1, stdin) != 1 || std::fread(&rows, 4, 1, stdin) != 1) return 1;
  std::vector<float> v((size_t)k * lanes);
  for (int r = 0; r < rows; ++r) {
    if (std::fread(v.data(), 4, v.size(), stdin) != v.size()) return 1;
    std::vector<ccs::Sum3> s(lanes);
    for (int l = 0; l < lanes; ++l)
      for (int i = 0; i < k; ++i) s[l].add(v[(size_t)l * k + i]);
    for (int o = lanes / 2; o; o /= 2)
      for (int l = 0; l < o; ++l) s[l].add(s[l + o]);
    std::printf("%.17g\n", s[0].value());
  }
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    d = tmp_path_factory.mktemp("fsum")
    (d / "t.cpp").write_text(SRC)
    exe = str(d / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2303_10788_gb300", "csrc"),
                    str(d / "t.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("k,lanes", [(1, 1), (2, 1), (16, 1), (16, 32), (1000, 32)])
@pytest.mark.parametrize("kind", ["eigenvalues", "spread", "cancelling"])
def test_no_further_off_than_fp64(prog, k, lanes, kind):
    rng = np.random.default_rng(k + lanes)
    n, rows = k * lanes, 300
    x = rng.normal(size=(rows, n))
    if kind == "eigenvalues":
        x = 0.02 + 0.01 * x
    elif kind == "spread":
        x = x * 10.0 ** rng.uniform(-9, 2, size=(rows, n))
    else:
        x[:, n // 2:2 * (n // 2)] = -x[:, :n // 2] * (1 + 1e-6)
        x = rng.permuted(x, axis=1)
    x = x.astype(np.float32)
    out = subprocess.run([prog], input=np.array([k, lanes, rows], np.int32).tobytes() + x.tobytes(),
                         capture_output=True, check=True).stdout.split()
    got = [float(t) for t in out]
    for row, g in zip(x.tolist(), got):
        exact = math.fsum(row)
        # (fsum and the program's own conversion each round the result once)
        assert abs(g - exact) <= (n - 1) * 2.0 ** -53 * sum(map(abs, row)) + 2.0 ** -52 * abs(exact)
