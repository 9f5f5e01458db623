"""Reference derivatives of the scalar solver's P2 and P3 polynomials at the vertices in block
fixed point (``csrc/dg_fix_scalar.cuh``), built as plain C++ on the CPU, against exact rational
arithmetic and the FP64 FMA chain over the modes, from modes of the average's size to smooth
ones that fall with the degree.

Bound in units of 2^(E + S - 1080): a truncated mode costs its coefficient, at most 12 in sum,
and the sum rounds by half a unit; the coefficients are exact."""
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
#include "dg_fix_scalar.cuh"
using namespace dg;
using namespace dg::sc;
template <int K, int J> static void order(const double *c) {
  Fx f[SC_NB<K>];
  const int E = sfx_deriv_block<K, J>(c, f);
  for (int v = 0; v < 3; ++v) {
    double t[J + 1];
    sfx_derivs<K, J>(f, E, v, t);
    for (int r = 0; r <= J; ++r) {
      std::printf(" %d %a", E + sc_scale<K, J>(), t[r]);
      for (int l = 1; l < SC_NB<K>; ++l) std::printf(" %a", psi_rs(l, r, J - r, vert_xi(v), vert_eta(v)));
    }
  }
}
int main() {
  int k;
  while (std::scanf("%d", &k) == 1) {
    double c[10];
    for (int l = 0; l < (k + 1) * (k + 2) / 2; ++l) if (std::scanf("%la", &c[l]) != 1) return 1;
    if (k == 2) { order<2, 1>(c); order<2, 2>(c); }
    if (k == 3) { order<3, 1>(c); order<3, 2>(c); order<3, 3>(c); }
    std::printf("\n");
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("scalar")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-fno-sanitize=shift", "-I", CSRC, str(d / "driver.cpp"), "-o", str(exe)], check=True)
    return exe


def _run(driver, k, cells):
    text = "\n".join(" ".join([str(k)] + [q.hex() for q in c]) for c in cells)
    out = subprocess.run([str(driver)], input=text + "\n", capture_output=True, text=True, check=True).stdout
    nb = (k + 1) * (k + 2) // 2
    for c, line in zip(cells, out.split("\n")):
        w = line.split()
        rows = [w[i:i + nb + 1] for i in range(0, len(w), nb + 1)]
        i = 0
        for j in range(1, k + 1):
            for _ in range(3 * (j + 1)):
                yield c, j, int(rows[i][0]), float.fromhex(rows[i][1]), [0.0] + [float.fromhex(q) for q in rows[i][2:]]
                i += 1


@pytest.mark.parametrize("fall", [1.0, 2.0 ** -10, 1e-5, 8.0])
@pytest.mark.parametrize("k", [2, 3])
def test_no_further_off_than_the_fma_chain(driver, k, fall):
    rng = np.random.default_rng([k, 3])
    deg = [0, 1, 1, 2, 2, 2, 3, 3, 3, 3]
    cells = [[1.0 + 0.1 * rng.uniform(-1, 1)] + [float(rng.uniform(-1, 1) * fall ** deg[l])
                                                 for l in range(1, (k + 1) * (k + 2) // 2)] for _ in range(300)]
    err = np.zeros((4, 2))
    for c, j, E, got, coef in _run(driver, k, cells):
        exact = sum(F(a) * F(x) for a, x in zip(coef, c))
        chain = 0.0
        for a, x in zip(coef, c):
            chain = float(F(a) * F(x) + F(chain)) if a else chain
        e = abs(F(got) - exact)
        assert e <= F(13) * F(2) ** (E - 1080) + abs(exact) / 2 ** 53, (c, j, got)
        size = float(sum(abs(F(a) * F(x)) for a, x in zip(coef, c)))
        if size > 0.0:
            err[j] += float(e) / size, float(abs(F(chain) - exact)) / size
    assert (err[1:, 0] <= err[1:, 1]).all(), err


@pytest.mark.parametrize("k", [2, 3])
def test_extremes(driver, k):
    """Equal magnitudes with every sign, zeros, and modes that are not finite."""
    nb = (k + 1) * (k + 2) // 2
    one = float(1 - 2.0 ** -53)
    cells = [[1.0] + [one * (1 if s >> l & 1 else -1) for l in range(nb - 1)] for s in range(1 << (nb - 1))]
    cells.append([3.0] + [0.0] * (nb - 1))
    for c, j, E, got, coef in _run(driver, k, cells):
        exact = float(sum(F(a) * F(x) for a, x in zip(coef, c)))
        assert abs(got - exact) <= 4e-16 * sum(abs(a * x) for a, x in zip(coef, c))
    for bad in (float("nan"), float("inf")):
        for c, j, E, got, coef in _run(driver, k, [[1.0] * (nb - 1) + [bad]]):
            assert np.isnan(got)
