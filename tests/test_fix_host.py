"""The block fixed-point sums of the FP64 kernels (``csrc/dg_fix.cuh``), built
as plain C++ on the CPU, against exact rational arithmetic.

Bound per sum of n terms c_j x_j, from the format: with B = 2^(E - 1022) the
power of two above the block's largest magnitude, each x_j is truncated by
less than 2^-58 B (times |c_j| <= 4), the dropped product of the low limbs is
at most 2^-57 B, rounding c_j to 2^-57 costs at most 2^-57 B, the sum's shift
2^-58 B, and the result rounds once to FP64 (a negative one after dropping
one unit of 2^-58 B)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_09620_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "dg_fix.cuh"
using namespace dg;
int main() {
  int n;
  while (std::scanf("%d", &n) == 1) {
    double c[32], x[32];
    int mx = 0;
    for (int i = 0; i < n; ++i) {
      if (std::scanf("%la %la", &c[i], &x[i]) != 2) return 1;
      const int a = fx_abs_hi(x[i]);
      mx = a > mx ? a : mx;
    }
    const int E = fx_exp(mx);
    FxAcc s{0, 0}, s1{0, 0};
    for (int i = 0; i < n; ++i) fx_mac(s, fxc(c[i]), fx_from(x[i], E));
    for (int i = n - 1; i >= 0; --i) fx_mac(s1, fxc(c[i]), fx_from(x[i], E));
    int E2;
    const int64_t r2 = fx_add(fx_sum(s), E, fx_sum(s), E - 40, E2);
    FxAcc s3{0, 0};   // the halved constants as run-time coefficients
    for (int i = 0; i < n; ++i) fx_mac(s3, fx_coef(c[i], -1), fx_from(x[i], E));
    const Fx w = fx_value(fx_sum(s3), 6);
    std::printf("%d %a %d %a %a %d\n", E, fx_to(fx_sum(s), E), (int)(fx_sum(s) == fx_sum(s1)), fx_to(r2, E2),
                fx_to(fx_sum(s3), E + 1), (int)((((int64_t)w.h << FX_LIMB) + w.l) == fx_sum(s3) >> 6 && w.l >= 0));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fix")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-fno-sanitize=shift", "-I", CSRC, str(d / "driver.cpp"), "-o", str(exe)], check=True)
    return exe


def _run(exe, sums):
    text = "\n".join(" ".join([str(len(s))] + [f"{float(c).hex()} {float(x).hex()}" for c, x in s]) for s in sums)
    out = subprocess.run([str(exe)], input=text + "\n", capture_output=True, text=True, check=True).stdout.split("\n")
    return [(int(a), float.fromhex(b), int(o), float.fromhex(d), float.fromhex(e), int(v))
            for a, b, o, d, e, v in (line.split() for line in out if line)]


def _sums(kind, rng, count=300):
    out = []
    for _ in range(count):
        n = int(rng.integers(1, 13))
        c = rng.uniform(-4, 4, n)
        x = rng.uniform(-1, 1, n)
        if kind == "spread":        # magnitudes over 80 binary orders
            x = x * np.exp2(rng.integers(-80, 1, n).astype(float))
        elif kind == "cancel":      # terms that cancel to round-off
            c[:], x = 1.0, np.concatenate([x, -x])[:n] * (1 + 1e-15 * rng.uniform(-1, 1, n))
        elif kind == "whole":       # exact in the format: small integers
            c, x = rng.integers(-4, 5, n).astype(float), rng.integers(-1000, 1001, n).astype(float)
        elif kind == "scale":       # the whole block far from 1
            x = x * 2.0 ** float(rng.integers(-900, 990))
        elif kind == "edge":        # powers of two, the largest constants, a zero
            c, x = rng.choice([-4.0, 4.0, 1.0, 0.0], n), rng.choice([0.0, 1.0, -1.0, 2.0, -2.0, 0.5], n)
        out.append(list(zip(c.tolist(), x.tolist())))
    return out


@pytest.mark.parametrize("kind", ["plain", "spread", "cancel", "whole", "scale", "edge"])
def test_sum_within_the_format_bound(driver, kind):
    sums = _sums(kind, np.random.default_rng([3, len(kind)]))
    for s, (E, r, same, r2, r3, split) in zip(sums, _run(driver, sums)):
        exact = sum((Fraction(c) * Fraction(x) for c, x in s), Fraction(0))
        B = Fraction(2) ** (E - 1022)
        tol = B * Fraction(8 * len(s) + 2, 2 ** 58) + abs(exact) / 2 ** 53
        assert same == 1                       # the order of the terms does not matter
        assert abs(Fraction(r) - exact) <= tol, (kind, s, r)
        if kind == "whole":
            assert Fraction(r) == exact
        # the sum of two blocks 40 exponents apart: one more unit each, of the larger block's
        assert abs(Fraction(r2) - exact * (1 + Fraction(1, 2 ** 40))) <= 2 * tol + B / 2 ** 56
        # run-time coefficients c / 2 are truncated at 2^-56, their low limbs reach 2^29, and the
        # sum is doubled: the terms of the bound above are 4, 2 * 4 and 2 * 4 units
        assert abs(Fraction(r3) - exact) <= B * Fraction(20 * len(s) + 4, 2 ** 58) + abs(exact) / 2 ** 53
        assert split == 1


def test_zeros_and_subnormals(driver):
    res = _run(driver, [[(1.0, 0.0)], [(1.0, -0.0), (-3.5, 0.0)], [(1.0, 5e-324)], [(1.0, 1.5), (4.0, 0.0)],
                        [(1.0, 3.0), (-1.0, 3.0)]])
    assert [r[1] for r in res] == [0.0, 0.0, 0.0, 1.5, 0.0]


def test_tiny_block_keeps_its_absolute_bound(driver):
    # the block exponent stops at 64: one unit is 2^-1016
    (E, r, *_), = _run(driver, [[(2.0, 1e-300), (1.0, 0.0)]])
    assert E == 64 and abs(Fraction(r) - 2 * Fraction(1e-300)) <= Fraction(18, 2 ** 1016)


def test_non_finite_block_is_marked(driver):
    res = _run(driver, [[(1.0, float("inf"))], [(1.0, float("nan")), (1.0, 1.0)], [(1.0, 1e308)]])
    assert [r[0] >= 0x7ff for r in res] == [True, True, False]
