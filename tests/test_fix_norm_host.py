"""The point of the largest norm of a vector of two fixed-point components, as the OE
statistics find it (``fx_norm_shift`` and ``fx_square`` of ``csrc/dg_fix.cuh``, built as plain C++
on the CPU), against exact integers: nearly equal norms, values of any magnitude in their
blocks, blocks of different exponents.

Bound: scaled to 62 bits (a value to 1 unit where it is shifted down), the squares of the largest
norm are at least 2^122 and their top parts at least 2^58; each is truncated by one unit and by
2^-60 of a value's square: the norm squared of the point found is within 2^-55 of the largest."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_09620_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "dg_fix.cuh"
using namespace dg;
int main() {
  int n, down[2];
  while (std::scanf("%d %d %d", &n, &down[0], &down[1]) == 3) {
    long long r[2][16];
    uint64_t top[2] = {0, 0};
    for (int i = 0; i < 2 * n; ++i) {
      if (std::scanf("%lld", &r[i & 1][i >> 1]) != 1) return 1;
      const uint64_t a = fx_mag(r[i & 1][i >> 1]);
      if (a > top[i & 1]) top[i & 1] = a;
    }
    const uint64_t a = top[0] >> down[0], b = top[1] >> down[1];
    const int sh = fx_norm_shift(a > b ? a : b);
    int best = 0;
    uint64_t bs = 0;
    for (int i = 0; i < n; ++i) {
      const uint64_t s = fx_square(fx_mag(r[0][i]), sh - down[0]) + fx_square(fx_mag(r[1][i]), sh - down[1]);
      if (i == 0 || s > bs) { bs = s; best = i; }
    }
    std::printf("%d\n", best);
  }
  return 0;
}
"""


def test_largest_norm(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", CSRC,
                    str(tmp_path / "driver.cpp"), "-o", str(exe)], check=True)
    rng = np.random.default_rng(8)
    cases = []
    for _ in range(3000):
        n = int(rng.integers(1, 13))
        bits = int(rng.integers(1, 62))
        down = [0, int(rng.integers(0, 64))] if rng.integers(2) else [int(rng.integers(0, 20)), 0]
        ang = rng.uniform(0, 6.3, n)
        size = 2.0 ** bits * (1 - 2.0 ** -50 * rng.integers(0, 4, n))   # nearly equal norms
        v = [[int(size[i] * np.cos(ang[i])), int(size[i] * np.sin(ang[i])) << min(max(down[1] - down[0], 0), 61 - bits)]
             for i in range(n)]
        cases.append((n, down, v))
    cases += [(3, [0, 0], [[0, 0]] * 3), (1, [0, 0], [[-(2 ** 61), 2 ** 61]]), (2, [63, 0], [[2 ** 60, 0], [0, 1]])]
    text = "\n".join(f"{n} {d[0]} {d[1]} " + " ".join(f"{a} {b}" for a, b in v) for n, d, v in cases)
    out = subprocess.run([str(exe)], input=text + "\n", capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    out = out.stdout.split()
    assert len(out) == len(cases)
    for (n, d, v), best in zip(cases, out):
        # exact squares in the common scale (times 2^(2 (d0 + d1)))
        sq = [(a << d[1]) ** 2 + (b << d[0]) ** 2 for a, b in v]
        top = max(max(abs(a) >> d[0] for a, _ in v), max(abs(b) >> d[1] for _, b in v))
        if top == 0:
            continue   # below a unit of the common block
        assert (max(sq) - sq[int(best)]) << 55 <= max(sq), (n, d, v, best)
