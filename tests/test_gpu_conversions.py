"""FP64 to FP32 and back on the integer units (``f32_of`` and ``f64_of`` of
``csrc/dg_common.cuh``, the mixed form's flux pass) against exact conversions: every exponent
that FP32 has and those beyond its ends, ties, signs, zeros, infinities and NaN.  And what
hangs on it: a state with a NaN average gives no finite or infinite neighbour."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _values():
    rng = np.random.default_rng(3)
    n = 1 << 17
    x = ((rng.integers(1023 - 160, 1023 + 140, n) << 52) | rng.integers(0, 1 << 52, n)).view(np.float64)
    with np.errstate(over="ignore"):
        x[:n // 4] = x[:n // 4].astype(np.float32)                                   # exact in FP32 (or 0, inf)
    ties = (rng.integers(1 << 23, 1 << 24, 4096) * 2 + 1) * 2.0 ** rng.integers(-140, 90, 4096)
    tiny = 2.0 ** -126 * np.array([1.0, 1 - 2.0 ** -24, 1 - 2.0 ** -25, 1 - 2.0 ** -26, 0.5, 0.75, 0.625, 0.25])
    top = float(np.finfo(np.float32).max) * np.array([1.0, 1 + 2.0 ** -26, 1 + 2.0 ** -25, 1 + 2.0 ** -24, 2.0])
    x = np.concatenate([x, ties, tiny, top, [0.0, 5e-324, 1e300, 1.7e308]])
    return np.concatenate([x, -x])


def test_to_fp32_and_back():
    x = _values()
    with np.errstate(over="ignore"):
        near = x.astype(np.float32).astype(np.float64)   # to nearest, ties to even
    m, e = np.frexp(np.abs(x))
    up = np.ldexp(np.floor(np.ldexp(m, 24) + 0.5), e - 24)            # to nearest, ties away from zero
    want = np.where(up < 2.0 ** -126, 0.0, np.where(np.isinf(near), np.inf, up))
    want = np.copysign(want, x)
    got = N.probe_math(N.MATH_F32, x)
    assert np.array_equal(got, want) and np.array_equal(np.signbit(got), np.signbit(x))
    back = N.probe_math(N.MATH_F64, x)
    want = np.where(np.abs(near) < 2.0 ** -126, 0.0, near)
    assert np.array_equal(back, want)


def test_infinities_and_nan():
    x = np.array([np.inf, -np.inf, np.nan, -np.nan])
    x = np.concatenate([x, np.array([0x7ff0000000000001, 0x7ff8000000000000, 0x7fffffffffffffff,
                                     0x7ff0000020000000], np.uint64).view(np.float64)])
    for kind in (N.MATH_F32, N.MATH_F64):
        got = N.probe_math(kind, x)
        assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2:]).all(), (kind, got)


@pytest.mark.parametrize("prec", [N.PREC_FP64, N.PREC_MIXED])
@pytest.mark.parametrize("k", [1, 2])
def test_a_nan_average_reaches_its_neighbours_as_nan(k, prec):
    """The flux pass with a NaN in one cell's averages: the cell and its three neighbours are NaN in
    every average, all other cells are what they are without it."""
    wl = W.riemann4_workload(n=8, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    u = N.initial_state(mesh, wl)
    s = N.Solver(mesh, N.config_for(wl, precision=prec), u)
    nbr = mesh.neighbors()[0]
    cell = int(np.flatnonzero((nbr >= 0).all(axis=1))[5])
    clean = s.op_rk_stage(u, u, 0.0, 1.0, 1e-3, 3.0)
    for c in range(4):
        v = u.copy()
        v[c, 0, cell] = np.nan
        got = s.op_rk_stage(v, v, 0.0, 1.0, 1e-3, 3.0)
        hit = np.zeros(mesh.nt, bool)
        hit[[cell, *nbr[cell]]] = True
        assert np.isnan(got[c][0][hit]).all()
        assert not np.isinf(got).any()
        assert np.array_equal(got[:, :, ~hit], clean[:, :, ~hit])


def test_first_stage_is_taken_for_what_it_is():
    """a = 0, b = 1 leaves u_n out; the smallest a, or b next to 1, does not."""
    wl = W.riemann4_workload(n=6, k=2)
    mesh = N.Mesh.from_mesh(wl.mesh)
    u = N.initial_state(mesh, wl)
    for prec in (N.PREC_FP64, N.PREC_MIXED):
        s = N.Solver(mesh, N.config_for(wl, precision=prec), u)
        first = s.op_rk_stage(u, u, 0.0, 1.0, 1e-3, 3.0)
        nan = np.full_like(u, np.nan)
        for a in (0.0, -0.0):
            assert np.array_equal(s.op_rk_stage(nan, u, a, 1.0, 1e-3, 3.0), first)
        for a, b in ((5e-324, 1.0), (0.0, np.nextafter(1.0, 2.0)), (0.0, np.nextafter(1.0, 0.0)), (0.0, -1.0)):
            assert np.isnan(s.op_rk_stage(nan, u, a, b, 1e-3, 3.0)).all(), (a, b)
