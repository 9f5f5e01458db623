"""Threads that read a solver's state (dg_get_state) beside the thread that writes it:
every copy is one of the states at a step boundary, bit for bit, and the writer's
results are those of a run without readers.  1,058 and 180,000 P2 cells and 700,000 P1 cells: a
reader of the mixed form converts two components' modes at a time, one's, or one mode."""
import math
import threading

import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(N.PREC_MIXED, 23, 2), (N.PREC_MIXED, 300, 2), (N.PREC_MIXED, 592, 1), (N.PREC_FP64, 23, 2)]


def _setup(prec, n, k):
    wl = W.riemann4_workload(n=n, k=k)
    mesh = N.Mesh.from_mesh(wl.mesh)
    return mesh, N.config_for(wl, precision=prec), N.initial_state(mesh, wl)


def _beside(solver, allowed, write, rounds):
    """write() `rounds` times while two threads read; every state read is in `allowed` (bytes)."""
    stop, bad, seen = threading.Event(), [], []

    def read():
        out = np.empty((4, solver.nb, solver.mesh.nt))
        while not stop.is_set():
            seen.append(1)
            if solver.get_state(out=out)[0].tobytes() not in allowed:
                bad.append(1)
    th = [threading.Thread(target=read) for _ in range(2)]
    for t in th:
        t.start()
    try:
        for _ in range(rounds):
            write()
    finally:
        stop.set()
        for t in th:
            t.join()
    assert seen and not bad, (len(bad), len(seen))


@pytest.mark.parametrize("prec,n,k", SIZES)
def test_readers_beside_set_state(prec, n, k):
    mesh, cfg, u0 = _setup(prec, n, k)
    s = N.Solver(mesh, cfg, u0)
    rng = np.random.default_rng(n)
    states, want = [], []
    for _ in range(2):
        u = u0 * rng.uniform(1.0, 1.1, u0.shape)
        s.set_state(u)
        states.append(u)
        want.append(s.get_state()[0].tobytes())
    out = np.empty_like(u0)

    def write():
        for u, w in zip(states, want):
            s.set_state(u)
            assert s.get_state(out=out)[0].tobytes() == w
    _beside(s, set(want), write, 10)


@pytest.mark.parametrize("prec,n,k", SIZES)
def test_readers_beside_advance(prec, n, k):
    mesh, cfg, u0 = _setup(prec, n, k)
    s = N.Solver(mesh, cfg, u0)
    steps = [s.get_state()[0].copy()]
    for _ in range(36):
        s.advance(math.inf, max_steps=1)
        steps.append(s.get_state()[0].copy())
    allowed = {u.tobytes() for u in steps}
    last = steps[-1].tobytes()
    s = N.Solver(mesh, cfg, u0)

    def write():
        s.set_state(steps[0])
        s.advance(math.inf, max_steps=36)
        assert s.get_state()[0].tobytes() == last
    _beside(s, allowed, write, 6)


@pytest.mark.parametrize("form", [3, 0])
@pytest.mark.parametrize("prec,n,k", SIZES)
def test_readers_beside_a_batch(prec, n, k, form):
    mesh, cfg, u0 = _setup(prec, n, k)
    s = N.Solver(mesh, cfg, u0)
    steps = [s.get_state()[0].copy()]
    for _ in range(10):
        s.advance(math.inf, max_steps=1)
        steps.append(s.get_state()[0].copy())
    b = N.Batch([mesh, mesh], [cfg, cfg], [u0, u0])
    b.set_shape(256, 2, form)

    def write():
        for i in range(2):
            b.solver(i).set_state(steps[0])
        b.advance(max_steps=10)
        for i in range(2):
            assert np.array_equal(b.solver(i).get_state()[0], steps[-1])
    _beside(b.solver(1), {u.tobytes() for u in steps}, write, 6)


@pytest.mark.parametrize("prec", [N.PREC_MIXED, N.PREC_FP64])
def test_readers_beside_set_shape(prec):
    """The step graphs are captured while the readers' copies go on."""
    mesh, cfg, u0 = _setup(prec, 23, 2)
    b = N.Batch([mesh, mesh], [cfg, cfg], [u0, u0])
    start = b.solver(1).get_state()[0].tobytes()
    s = N.Solver(mesh, cfg, u0)
    s.advance(math.inf, max_steps=3)

    def write():
        for form in (0, 3, 1):
            b.set_shape(128, 2, form)
    _beside(b.solver(1), {start}, write, 30)
    for form in (0, 3, 1):
        b.set_shape(128, 2, form)
        b.advance(max_steps=1)
    assert np.array_equal(b.solver(1).get_state()[0], s.get_state()[0])


@pytest.mark.parametrize("prec", [N.PREC_MIXED, N.PREC_FP64])
def test_readers_beside_autotune(prec):
    """The tuning steps (at most 400 states) and the restored start."""
    mesh, cfg, u0 = _setup(prec, 12, 1)
    s = N.Solver(mesh, cfg, u0)
    allowed = {s.get_state()[0].tobytes()}
    for _ in range(400):
        s.advance(math.inf, max_steps=1)
        allowed.add(s.get_state()[0].tobytes())
    b = N.Batch([mesh, mesh], [cfg, cfg], [u0, u0])
    start = b.solver(1).get_state()[0].tobytes()

    def write():
        b.autotune(steps=1)
        assert b.solver(1).get_state()[0].tobytes() == start
    _beside(b.solver(1), allowed, write, 3)
