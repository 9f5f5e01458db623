"""A cell average that is not a number is not in G: dg_init refuses it and the limiter
counts it, in every component and both precisions, whatever the sign of the NaN; a
density or energy of -inf likewise."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [N.PREC_FP64, N.PREC_MIXED])
@pytest.mark.parametrize("k", [1, 2])
def test_nan_averages_are_refused_and_counted(k, prec):
    wl = W.riemann4_workload(n=6, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    u0 = N.initial_state(mesh, wl)
    cfg = N.config_for(wl, precision=prec)
    s = N.Solver(mesh, cfg, u0)
    bad = [(c, v) for c in range(4) for v in (np.nan, -np.nan)] + [(0, -np.inf), (3, -np.inf)]
    for c, v in bad:
        u = u0.copy()
        u[c, 0, 7] = v
        _, counters = s.op_limit(u)
        assert counters[1] == 1, (c, v, counters)
        with pytest.raises(N.DGError) as e:
            N.Solver(mesh, cfg, u)
        assert e.value.code == N.DG_ENONPHYS, (c, v)
    assert s.op_limit(u0)[1][1] == 0
