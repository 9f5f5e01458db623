"""Vertex gradients and Hessians in block fixed point (``csrc/dg_fix_vertex.cuh``), built as
plain C++ on the CPU, against exact rational arithmetic and against the FP64 FMA chain
(sums over the modes at the vertices, then J^-T) on the same data, for modes of the average's
size down to 10^-15 of it.

Bound of a gradient in units of 2^-58 of the modes' block B = 2^(E - 1022), times the scale of
the coefficients (8 in P1, 16 in P2) and 2^E[d]: a reference derivative misses at most 0.6 by
truncated modes and 0.5 by rounding; J^-1 is truncated at 2^-56, 4 units of a derivative below
0.63 * 2^58; two such terms and the rounding of the sum, a unit for the dropped bits of the low
products: 2 (1.1 + 2.6) + 2 < 10.  Hessian: rounding and truncation 1.3 (twice), and per turn 2 (4 *
0.75) + 1, the first turn's doubled by the second: below 2 * 2 * 1.3 + 3 * 7 < 28 units of 64 2^-58 B."""
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
#include "dg_fix_vertex.cuh"
using namespace dg;
template <int NB> static void run(const double *h, const FxRows &J) {
  Fx g[3][2];
  FxDerivs<NB> d(h, J, [&](int v, Fx gx, Fx gy) { g[v][0] = gx; g[v][1] = gy; });
  std::printf("%d %d", d.EG[0], d.EG[1]);
  for (int v = 0; v < 3; ++v)
    for (int i = 0; i < 2; ++i) std::printf(" %a", fx_to(fx_join(g[v][i]), d.EG[i]));
  if (NB == 6) {
    std::printf(" %d", d.EH);
    for (int r = 0; r < 3; ++r) std::printf(" %a", fx_to(fx_join(d.hess[r]), d.EH + r * (d.EG[1] - d.EG[0])));
  }
  std::printf("\n");
}
int main() {
  int nb;
  while (std::scanf("%d", &nb) == 1) {
    double h[6] = {0}, xi[2], eta[2];
    for (int l = 0; l < nb; ++l) if (std::scanf("%la", &h[l]) != 1) return 1;
    if (std::scanf("%la %la %la %la", &xi[0], &xi[1], &eta[0], &eta[1]) != 4) return 1;
    const FxRows J = fx_rows(xi, eta);
    if (nb == 3) run<3>(h, J); else run<6>(h, J);
  }
  return 0;
}
"""

VERT = ((0, 0), (1, 0), (0, 1))


def _dpsi(l, v):
    x, y = VERT[v]
    return ((0, 0), (4, 2), (0, 3), (48 * x + 24 * y - 24, 24 * x + 8 * y - 8), (20 * y - 4, 20 * x + 20 * y - 12),
            (0, 20 * y - 8))[l]


D2 = {3: (48, 24, 8), 4: (0, 20, 20), 5: (0, 0, 20)}


def _exact(h, xi, eta):
    h, xi, eta = [F(q) for q in h], [F(q) for q in xi], [F(q) for q in eta]
    g = []
    for v in range(3):
        p, q = (sum(_dpsi(l, v)[r] * h[l] for l in range(1, len(h))) for r in (0, 1))
        g.append([p * xi[d] + q * eta[d] for d in (0, 1)])
    xx, xe, ee = (sum(D2[l][r] * h[l] for l in range(3, len(h))) for r in range(3))
    return g, [xx * xi[a] * xi[b] + xe * (xi[a] * eta[b] + xi[b] * eta[a]) + ee * eta[a] * eta[b]
               for a, b in ((0, 0), (0, 1), (1, 1))]


def _fma(a, b, c):
    return float(F(a) * F(b) + F(c))


def _chain(h, xi, eta):
    """The same in FP64: values at vertex 0 and the constant second derivatives by FMA chains."""
    p0 = q0 = 0.0
    for l in range(1, len(h)):
        p0, q0 = (_fma(_dpsi(l, 0)[r], h[l], s) for r, s in ((0, p0), (1, q0)))
    d2 = []
    for r in range(3):
        s = 0.0
        for l in range(3, len(h)):
            s = _fma(D2[l][r], h[l], s)
        d2.append(s)
    g = []
    for v in range(3):
        p, q = p0 + (0.0, d2[0], d2[1])[v], q0 + (0.0, d2[1], d2[2])[v]
        g.append([_fma(p, xi[d], q * eta[d]) for d in (0, 1)])
    hs = [_fma(d2[0], xi[a] * xi[b], _fma(d2[1], _fma(xi[a], eta[b], xi[b] * eta[a]) if a != b else 2 * xi[a] * eta[a],
                                          d2[2] * (eta[a] * eta[b]))) for a, b in ((0, 0), (0, 1), (1, 1))]
    return g, hs


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("vertex")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-fno-sanitize=shift", "-I", CSRC, str(d / "driver.cpp"), "-o", str(exe)], check=True)
    return exe


def _cells(nb, s1, s2, aspect, count, seed):
    rng = np.random.default_rng([seed, nb])
    out = []
    while len(out) < count:
        h = [1.0 + 0.1 * rng.uniform(-1, 1)] + [float(rng.uniform(-1, 1) * (s1 if l < 3 else s2)) for l in range(1, nb)]
        a, b = rng.uniform(-3, 3), rng.uniform(0.7, 1.4)
        x1, y1 = 0.01 / aspect * np.cos(a), 0.01 * np.sin(a)
        x2, y2 = 0.01 / aspect * np.cos(a + b), 0.01 * np.sin(a + b)
        det = x1 * y2 - x2 * y1
        out.append((h, [float(y2 / det), float(-x2 / det)], [float(-y1 / det), float(x1 / det)]))
    return out


@pytest.mark.parametrize("aspect", [1.0, 8.0])
@pytest.mark.parametrize("nb,s1,s2", [(3, 1.0, 0.0), (3, 2.0 ** -10, 0.0), (3, 1e-15, 0.0), (6, 1.0, 1.0),
                                      (6, 2.0 ** -10, 2.0 ** -20), (6, 1e-8, 1e-15), (6, 1e-6, 1e-3)])
def test_no_further_off_than_the_fma_chain(driver, nb, s1, s2, aspect):
    cells = _cells(nb, s1, s2, aspect, 400, 5)
    text = "\n".join(" ".join([str(nb)] + [q.hex() for q in h + xi + eta]) for h, xi, eta in cells)
    lines = subprocess.run([str(driver)], input=text + "\n", capture_output=True, text=True, check=True).stdout.split("\n")
    err = np.zeros((2, 2))   # (fixed point, chain) x (gradient, Hessian): summed errors relative to the vector's norm
    for (h, xi, eta), line in zip(cells, lines):
        w = line.split()
        E = int(w[0]), int(w[1])
        got = [[float.fromhex(w[2 + 2 * v + d]) for d in (0, 1)] for v in range(3)]
        g, hs = _exact(h, xi, eta)
        cg, ch = _chain(h, xi, eta)
        for v in range(3):
            norm = float(sum(abs(q) for q in g[v]))
            for d in (0, 1):
                e = abs(F(got[v][d]) - g[v][d])
                # the scale of the coefficients and J's are in E
                assert e <= F(10) * F(2) ** (E[d] - 1080) + abs(g[v][d]) / 2 ** 53, (h, v, d)
                err[0, 0] += float(e) / norm
                err[1, 0] += float(abs(F(cg[v][d]) - g[v][d])) / norm
        if nb == 6:
            H, got = int(w[8]), [float.fromhex(q) for q in w[9:12]]
            norm = float(sum(abs(q) for q in hs))
            for r in range(3):
                e = abs(F(got[r]) - hs[r])
                assert e <= F(28) * F(2) ** (H + r * (E[1] - E[0]) - 1080) + abs(hs[r]) / 2 ** 53
                err[0, 1] += float(e) / norm
                err[1, 1] += float(abs(F(ch[r]) - hs[r])) / norm
    assert err[0, 0] <= err[1, 0] and err[0, 1] <= err[1, 1], err


JUMPS = r"""
#include <cstdio>
#include "dg_fix_vertex.cuh"
using namespace dg;
// jumps between two cells' values at a vertex (index v of one, w of the other) of two components,
// and their rotation by (nx, ny), as the edge records take them
int main() {
  double h[2][2][6], n[2];
  int v[2];
  while (std::scanf("%d %d %la %la", &v[0], &v[1], &n[0], &n[1]) == 4) {
    Fx val[2][2];
    int E[2][2], z[2];
    int64_t d[2];
    for (int s = 0; s < 2; ++s)
      for (int c = 0; c < 2; ++c) {
        for (int l = 0; l < 6; ++l) if (std::scanf("%la", &h[s][c][l]) != 1) return 1;
        Fx f[6];
        E[s][c] = fx_block<6>(h[s][c], f) + 2;
        FxAcc a{0, 0};
        for (int l = 0; l < 6; ++l) fx_mac(a, fxc(psi(l, vert_xi(v[s]), vert_eta(v[s]))), f[l]);
        val[s][c] = fx_value(fx_sum(a), 2);
      }
    int Es = E[0][0];
    for (int q = 1; q < 4; ++q) Es = E[q >> 1][q & 1] > Es ? E[q >> 1][q & 1] : Es;
    for (int c = 0; c < 2; ++c) {
      d[c] = fx_diff(val[0][c], E[0][c], val[1][c], E[1][c], Es);
      z[c] = fx_room(d[c]);
    }
    const int zz = z[0] < z[1] ? z[0] : z[1];
    const Fx a = fx_value_up(d[0], zz), b = fx_value_up(d[1], zz), cx = fx_coef(n[0], 0), cy = fx_coef(n[1], 0);
    FxAcc t{0, 0};
    fx_mac(t, cx, a);
    fx_mac(t, cy, b);
    std::printf("%a\n", fx_to(fx_sum(t), Es - zz));
  }
  return 0;
}
"""


@pytest.mark.parametrize("small,whole", [(1.0, False), (2.0 ** -12, False), (2.0 ** -40, True)])
def test_rotated_jumps_of_values(tmp_path, small, whole):
    """Normal jump of a vector between two cells.  In general no further off in the mean than
    FP64 values, their differences and a rotation; where the values are exact, to a few 2^-53 of the jump."""
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "driver.cpp").write_text(JUMPS)
    exe = tmp_path / "driver"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-fno-sanitize=shift", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o", str(exe)], check=True)
    rng = np.random.default_rng(9)
    psi = lambda l, x, y: (1, 4 * x + 2 * y - 2, 3 * y - 1, 24 * x * x + 24 * x * y + 4 * y * y - 24 * x - 8 * y + 4,
                           20 * x * y + 10 * y * y - 4 * x - 12 * y + 2, 10 * y * y - 8 * y + 1)[l]
    cases, lines = [], []
    for _ in range(1500):
        v = [int(q) for q in rng.integers(0, 3, 2)]
        t = rng.uniform(0, 6.3)
        n = [float(np.cos(t)), float(np.sin(t))]
        avg = [1.0, -0.5] if whole else [float(q) for q in rng.uniform(-1, 1, 2)]
        h = [[[avg[c]] + [float(rng.integers(-8, 9) * small if whole else rng.uniform(-1, 1) * small) for _ in range(5)]
              for c in range(2)] for _ in range(2)]
        cases.append((v, n, h))
        lines.append(" ".join([str(v[0]), str(v[1]), n[0].hex(), n[1].hex()] + [q.hex() for s in h for c in s for q in c]))
    out = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(cases)
    err = np.zeros(2)
    for (v, n, h), w in zip(cases, out):
        ex = [sum(psi(l, *VERT[v[0]]) * F(h[0][c][l]) - psi(l, *VERT[v[1]]) * F(h[1][c][l]) for l in range(6)) for c in (0, 1)]
        exact = ex[0] * F(n[0]) + ex[1] * F(n[1])
        val = [[0.0, 0.0], [0.0, 0.0]]
        for s in (0, 1):
            for c in (0, 1):
                a = h[s][c][0]
                for l in range(1, 6):
                    a = _fma(psi(l, *VERT[v[s]]), h[s][c][l], a)
                val[s][c] = a
        d = [val[0][c] - val[1][c] for c in (0, 1)]
        chain = _fma(d[0], n[0], d[1] * n[1])
        e = abs(F(float.fromhex(w)) - exact)
        if whole:   # coefficients truncated at 2^-56, two products, two roundings
            assert e <= F(5, 2 ** 54) * (abs(ex[0]) + abs(ex[1])), (v, n, h)
        err += float(e), float(abs(F(chain) - exact))
    assert whole or err[0] <= err[1], err


def test_largest_coefficients_stay_in_the_limbs(driver):
    """Modes of one size and the signs that add up, and J^-1 of equal entries just below a power of two."""
    one = float(1 - 2.0 ** -53)
    cells = []
    for nb in (3, 6):
        for signs in range(1 << (nb - 1)):
            h = [0.0] + [one * (1 if signs >> l & 1 else -1) * (0.125 if l >= 2 else 1.0) for l in range(nb - 1)]
            cells.append((h, [one, one], [one, one]))
            if nb == 6:
                cells.append(([0.0, 0.0, 0.0] + [8 * q for q in h[3:]], [one, one], [one, one]))
    text = "\n".join(" ".join([str(len(h))] + [q.hex() for q in h + xi + eta]) for h, xi, eta in cells)
    lines = subprocess.run([str(driver)], input=text + "\n", capture_output=True, text=True, check=True).stdout.split("\n")
    for (h, xi, eta), line in zip(cells, lines):
        w = line.split()
        g, hs = _exact(h, xi, eta)
        top = float(max(abs(q) for v in g for q in v))
        for v in range(3):
            for d in (0, 1):
                assert abs(float.fromhex(w[2 + 2 * v + d]) - float(g[v][d])) <= 1e-14 * top
        if len(h) == 6:
            top = float(max(abs(q) for q in hs))
            assert all(abs(float.fromhex(q) - float(x)) <= 1e-14 * max(top, 1e-300) for q, x in zip(w[9:12], hs))
