"""OE statistics of a state whose second momentum component varies far less than the
first: each component's deviation is accurate relative to itself.  Deviations of 2^-30 and
less of the other component's, made of exact sums (small integers times a power of two, one
cell's modes); allowed: 1e-13, for oracle and GPU round the basis values at the points (a few
2^-53 of their terms, with cancellation) and sum in other orders."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [1, 2])
@pytest.mark.parametrize("k", [1, 2])
def test_component_far_smaller_than_the_other(oracle_mod, k, small):
    O = oracle_mod
    mesh = W.jittered_grid(6, 5, seed=2, periodic=True)
    om = O.OracleMesh.from_mesh(mesh)
    nb = 3 if k == 1 else 6
    rng = np.random.default_rng(k)
    u = np.zeros((4, nb, mesh.nt))
    u[0, 0], u[3, 0] = 1.0, 2.5
    for c in (1, 2):   # the averages are zero: so is the mean
        u[c, 1:] = rng.integers(-99, 100, (nb - 1, mesh.nt)) * (2.0 ** -50 if c == small else 2.0 ** -7)
    m = N.Mesh.from_mesh(mesh)
    got = N.Solver(m, N.make_config(k, oe=N.OE_CW), u).op_stats(u)
    exp = om.stats(O.make_config(k, oe=2), u)
    assert got[1] == 0.0 and got[2] == 0.0
    np.testing.assert_allclose(got[[5, 8, 9]], exp[[5, 8, 9]], rtol=1e-13)
