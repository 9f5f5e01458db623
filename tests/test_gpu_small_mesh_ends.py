"""The rest of a small mesh's fused steps against steps with a finalize launch after every
kernel, bit for bit: OE or the limiter off, a moving shock at the boundary, and runs to an end
time -- the clamped last step, the idle steps after it in the same chunk, and going on from
there -- against the batch's work-list form, which never fuses."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _numbers(st):
    return {q: st[q] for q in st if isinstance(st[q], (int, float))}


@pytest.mark.parametrize("oe,bp", [(N.OE_OFF, N.BP_ON), (N.OE_RI, N.BP_OFF), (N.OE_OFF, N.BP_OFF)])
@pytest.mark.parametrize("prec,n", [(N.PREC_FP64, 5), (N.PREC_FP64, 60), (N.PREC_MIXED, 23), (N.PREC_MIXED, 100)])
@pytest.mark.parametrize("k", [1, 2])
def test_options_off(k, prec, n, oe, bp):
    wl = W.riemann4_workload(n=n, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    # mild data, which needs neither
    u0 = mesh.project(k, fn=lambda x, y: np.stack([1 + 0.1 * np.sin(6 * x), 0.1 * np.cos(5 * y), 0 * x, 2.5 + 0 * x], -1))
    got = []
    for fused in (True, False):
        s = N.Solver(mesh, N.config_for(wl, precision=prec, oe=oe, bp=bp), u0)
        s.advance_async(1)
        if fused:
            s.advance_async(4)
        else:
            launches = sum(q[1] for q in s.profile_steps(4).values())
            assert launches == 4 * (13 if oe == N.OE_OFF else 19)
        st = s.sync()
        got.append((s.get_state(), _numbers(st)))
    (a, ta), sa = got[0]
    (b, tb), sb = got[1]
    assert np.isfinite(a).all() and ta == tb and np.array_equal(a, b) and sa == sb


@pytest.mark.parametrize("oe", [N.OE_RI, N.OE_OFF])
@pytest.mark.parametrize("prec", [N.PREC_FP64, N.PREC_MIXED])
@pytest.mark.parametrize("k", [1, 2])
def test_moving_shock_to_an_end_time(k, prec, oe):
    wl = W.dmr_workload(nx=32, ny=8, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    u0 = N.initial_state(mesh, wl)
    cfg = N.config_for(wl, precision=prec, oe=oe)
    s = N.Solver(mesh, cfg, u0)
    b = N.Batch([mesh], [cfg], [u0])
    assert b.shape()["launches_per_stage"] == 3
    dt = s.advance(1.0, max_steps=1)[0]["dt_last"]
    b.advance(max_steps=1)
    for t_end in (3.3 * dt, 3.3 * dt, 5.0 * dt, 5.0 * dt + 1e-3 * dt):   # clamped, idle, on, a sliver
        st = s.advance(t_end)[0]
        sb = b.advance(t_end)[0]
        (ua, ta), (ub, tb) = s.get_state(), b.solver(0).get_state()
        assert ta == tb == t_end and np.array_equal(ua, ub)
        assert _numbers(st) == _numbers(sb)
