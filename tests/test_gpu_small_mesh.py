"""Steps of a small mesh, whose kernels finish each other's reductions, against
the same steps with a finalize launch after every kernel (dg_profile_steps):
the arithmetic and its order are the same, so states, times and counters must
be equal bit for bit.  Sizes around one and two groups of 128 tiles (32 cells a
tile in FP64, 128 mixed) and one beyond, where both take finalize launches."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("oe", [N.OE_RI, N.OE_CW])
@pytest.mark.parametrize("prec,n", [(N.PREC_FP64, 4), (N.PREC_FP64, 45), (N.PREC_FP64, 46), (N.PREC_FP64, 64),
                                    (N.PREC_FP64, 65), (N.PREC_MIXED, 23), (N.PREC_MIXED, 91), (N.PREC_MIXED, 128),
                                    (N.PREC_MIXED, 129)])
@pytest.mark.parametrize("k", [1, 2])
def test_fused_steps_equal_separate_ones(k, prec, n, oe):
    wl = W.riemann4_workload(n=n, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    u0 = N.initial_state(mesh, wl)
    got = []
    for fused in (True, False):
        s = N.Solver(mesh, N.config_for(wl, precision=prec, oe=oe), u0)
        s.advance_async(1)
        if fused:
            s.advance_async(4)
        else:
            s.profile_steps(4)
        st = s.sync()
        got.append((s.get_state(), {q: st[q] for q in st if isinstance(st[q], (int, float))}))
    (a, ta), sa = got[0]
    (b, tb), sb = got[1]
    assert ta == tb and np.array_equal(a, b) and sa == sb
