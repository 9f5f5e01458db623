"""Transfers of a mixed-form state: the averages cross unchanged, the modes are
rounded to FP32 once (to nearest even), whatever the cell count and degree;
two threads may read one solver."""
import threading

import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _solver(nx, ny, k, seed=5):
    mesh = W.jittered_grid(nx, ny, seed=seed, periodic=True)
    m = N.Mesh.from_mesh(mesh)
    u = W.random_modal_state(mesh.nt, k, seed)
    u[:, 1:] *= np.random.default_rng(seed).choice([1.0, 1e-5, 1e-30, 1e-42], (4, u.shape[1] - 1, mesh.nt))
    return m, N.Solver(m, N.make_config(k, precision=N.PREC_MIXED), W.random_modal_state(mesh.nt, k, seed + 1)), u


@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("nx,ny", [(3, 3), (7, 9), (8, 8), (65, 31)])
def test_roundtrip_rounds_the_modes_once(nx, ny, k):
    _, s, u = _solver(nx, ny, k)
    s.set_state(u, 0.25)
    got, t = s.get_state()
    want = u.copy()
    want[:, 1:] = u[:, 1:].astype(np.float32)
    assert t == 0.25 and np.array_equal(got, want)


def test_two_threads_read_one_solver():
    _, s, u = _solver(65, 31, 2)
    s.set_state(u)
    want, _ = s.get_state()
    bad = []

    def read():
        for _ in range(20):
            if not np.array_equal(s.get_state()[0], want):
                bad.append(1)
    th = [threading.Thread(target=read) for _ in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad
