"""OE damping of modes far below the cell averages.  The averages, the modes (small integers
times 2^-40), and so the vertex values and the reference derivatives are exact in FP64, and
the normalisers are given, so that the damping exponents of the GPU and of the plain numpy form
below differ by the rounding of J^-1, the wave speeds and the sums alone, a few 2^-53 of
exponents of order one; allowed: 1e-12.  (The CPU oracle evaluates the polynomials at mapped points, which rounds
the values at 2^-53 of the average, far above these jumps.)"""
import math

import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu

VERT = ((0.0, 0.0), (1.0, 0.0), (0.0, 1.0))
PSI = [lambda x, y: 1.0, lambda x, y: 4 * x + 2 * y - 2, lambda x, y: 3 * y - 1,
       lambda x, y: 24 * x * x + 24 * x * y + 4 * y * y - 24 * x - 8 * y + 4,
       lambda x, y: 20 * x * y + 10 * y * y - 4 * x - 12 * y + 2, lambda x, y: 10 * y * y - 8 * y + 1]
DX = [lambda x, y: 0.0, lambda x, y: 4.0, lambda x, y: 0.0, lambda x, y: 48 * x + 24 * y - 24, lambda x, y: 20 * y - 4,
      lambda x, y: 0.0]
DY = [lambda x, y: 0.0, lambda x, y: 2.0, lambda x, y: 3.0, lambda x, y: 24 * x + 8 * y - 8,
      lambda x, y: 20 * x + 20 * y - 12, lambda x, y: 20 * y - 8]
D2 = [(0, 0, 0), (0, 0, 0), (0, 0, 0), (48, 24, 8), (0, 20, 20), (0, 0, 20)]


def damped(mesh, nbr, nbr_edge, k, u, dt, stats, component_wise, gamma=1.4):
    """The OE procedure of a periodic mesh (eqs. oe:sys, OEScalar:Coef1, RIOESys:Coef1) in numpy."""
    nb, nt = u.shape[1], u.shape[2]
    x = mesh.xy[mesh.tri]
    d1, d2 = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0]
    det = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0]
    xi, eta = np.array([d2[:, 1], -d2[:, 0]]) / det, np.array([-d1[:, 1], d1[:, 0]]) / det
    val = np.array([sum(PSI[l](*v) * u[:, l] for l in range(nb)) for v in VERT])        # [vertex][c][nt]
    p = np.array([sum(DX[l](*v) * u[:, l] for l in range(1, nb)) for v in VERT])
    q = np.array([sum(DY[l](*v) * u[:, l] for l in range(1, nb)) for v in VERT])
    grad = np.array([p * xi[d] + q * eta[d] for d in (0, 1)])                           # [d][vertex][c][nt]
    xx, xe, ee = (sum(D2[l][r] * u[:, l] for l in range(1, nb)) + 0.0 * u[:, 0] for r in range(3))
    hess = np.array([xx * xi[a] * xi[b] + xe * (xi[a] * eta[b] + xi[b] * eta[a]) + ee * eta[a] * eta[b]
                     for a, b in ((0, 0), (0, 1), (1, 1))])                             # [3][c][nt]
    D = stats[[4, 8, 9, 6]] if component_wise else stats[[4, 5, 5, 6]]
    cells, sigma = np.arange(nt), np.zeros((k + 1, 4, nt))
    for i in range(3):
        a, b = x[:, (i + 1) % 3], x[:, (i + 2) % 3]
        ln = np.hypot(*(b - a).T)
        nx, ny = (b - a)[:, 1] / ln, -(b - a)[:, 0] / ln
        h, K, j = det / ln, nbr[:, i], nbr_edge[:, i]

        def rotated(d):   # jumps of (rho, m_n, m_t, E), or of the components
            return d if component_wise else np.array([d[0], d[1] * nx + d[2] * ny, d[2] * nx - d[1] * ny, d[3]])
        J, beta = np.zeros((k + 1, 4, nt)), np.zeros(nt)
        for ev in (0, 1):
            v, w = (i + 1 + ev) % 3, (j + 2 - ev) % 3
            own, oth = val[v], val[w, :, K].T
            for s in (own, oth):
                pr = (gamma - 1) * (s[3] - 0.5 * (s[1] ** 2 + s[2] ** 2) / s[0])
                beta = np.maximum(beta, np.abs(s[1] * nx + s[2] * ny) / s[0] + np.sqrt(gamma * pr / s[0]))
            J[0] += 0.5 * rotated(own - oth) ** 2
            for d in (0, 1):
                J[1] += 0.5 * rotated(grad[d, v] - grad[d, w, :, K].T) ** 2
            if k == 2:
                for r, binom in enumerate((1, 2, 1)):
                    J[2] += 0.5 * binom * rotated(hess[r] - hess[r][:, K]) ** 2
        if not component_wise:
            J[:, 1] = J[:, 2] = np.maximum(J[:, 1], J[:, 2])
        for o in range(k + 1):
            A = (2 * o + 1) / ((2 * k - 1) * math.factorial(o))
            sigma[o] += beta / h * A * h ** o * np.sqrt(J[o]) / D[:, None]
    out = u.copy()
    for l in range(1, nb):
        out[:, l] *= np.exp(-dt * sigma[:(1 if l < 3 else 2) + 1].sum(axis=0))
    return out


@pytest.mark.parametrize("oe", [N.OE_RI, N.OE_CW])
@pytest.mark.parametrize("k", [1, 2])
def test_damping_of_modes_far_below_the_average(k, oe):
    mesh = W.jittered_grid(9, 7, seed=4, periodic=True)
    nb = 3 if k == 1 else 6
    rng = np.random.default_rng(k)
    u = np.empty((4, nb, mesh.nt))
    u[:, 0] = np.array([1.0, 0.25, -0.5, 2.5])[:, None]
    u[:, 1:] = rng.integers(-8, 9, (4, nb - 1, mesh.nt)) * 2.0 ** -40
    stats = np.concatenate([u[:, 0, 0], np.full(3, 2.0 ** -36), [1.0], np.full(2, 2.0 ** -36)])
    dt = 2.0 ** -9
    m = N.Mesh.from_mesh(mesh)
    got = N.Solver(m, N.make_config(k, oe=oe), u).op_oe(u, dt, stats)
    exp = damped(mesh, *m.neighbors(), k, u, dt, stats, oe == N.OE_CW)
    assert np.array_equal(got[:, 0], u[:, 0])
    live = u[:, 1:] != 0.0
    ratio = exp[:, 1:][live] / u[:, 1:][live]
    assert ratio.min() > 1e-3 and np.median(ratio) < 0.9   # exponents of order one
    np.testing.assert_allclose(got[:, 1:], exp[:, 1:], rtol=1e-12)
