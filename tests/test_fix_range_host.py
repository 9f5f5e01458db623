"""``fx_to`` of ``csrc/dg_fix.cuh`` (plain C++ on the CPU) up to the end of FP64's range: integers
of any length and sign at exponents from the smallest that a block's sum has to beyond the
largest.  The result is the nearest number, infinite from 2^1024 - 2^970 up, with the sign."""
import math
import os
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_09620_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "dg_fix.cuh"
int main() {
  long long r;
  int E;
  while (std::scanf("%lld %d", &r, &E) == 2) std::printf("%a\n", dg::fx_to(r, E));
  return 0;
}
"""


def test_ends_of_the_range(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-fno-sanitize=shift", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o", str(exe)], check=True)
    rng = np.random.default_rng(6)
    pairs = []
    for _ in range(6000):
        bits = int(rng.integers(1, 64))
        r = int(rng.integers(1 << (bits - 1), (1 << bits) - 1, endpoint=True, dtype=np.uint64 if bits > 62 else np.int64))
        top = 2104 - bits   # the exponent at which r reaches 2^1024
        E = int(rng.choice([top, top - 1, top + 1, top + 500, 58, 59, 64, 1080]))
        pairs.append((r if rng.integers(2) else -r, E))
    pairs += [((1 << 62) + d, E) for d in (-1, 0, 1) for E in (2040, 2041, 2042, 58)] + [(0, 58), (0, 3000)]
    out = subprocess.run([str(exe)], input="\n".join(f"{r} {E}" for r, E in pairs) + "\n", capture_output=True,
                         text=True, check=True).stdout.split()
    assert len(out) == len(pairs)
    seen = set()
    for (r, E), w in zip(pairs, out):
        got, a = float.fromhex(w), abs(r)
        v = F(a) * F(2) ** (E - 1080)
        if v >= F(2) ** 1024 - F(2) ** 970:
            want = math.inf
        else:   # halves round up
            ulp = F(math.ulp(float(v))) if float(v) <= v else F(math.ulp(math.nextafter(float(v), 0.0)))
            want = float((v / ulp + F(1, 2)).__floor__() * ulp)
        seen.add("inf" if math.isinf(want) else "normal")
        assert abs(got) == want and (r >= 0 or math.copysign(1.0, got) < 0.0), (r, E, got, want)
    assert seen == {"inf", "normal"}
