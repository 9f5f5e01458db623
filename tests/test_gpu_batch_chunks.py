"""Work chunks of the batch's work-list forms: a block takes the tickets of its whole chunk, also
where the chunk lies across two reduction groups (128 tiles) or beyond the last tile, and the
results are bitwise those of the solves alone; an FP64 chunk, four lanes per cell, is
dealt to four blocks."""
import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [3, 1])
@pytest.mark.parametrize("cells_per_block", [128, 384, 640, 1024])
@pytest.mark.parametrize("prec,sizes", [(N.PREC_FP64, (3, 65, 92)), (N.PREC_MIXED, (5, 129, 183))])
def test_chunks_across_groups(prec, sizes, cells_per_block, form):
    solves = [(n, 1 + i % 2) for i, n in enumerate(sizes)]
    wls = [W.riemann4_workload(n=n, k=k) for n, k in solves]
    meshes = [N.Mesh.from_mesh(w.mesh) for w in wls]
    cfgs = [N.config_for(w, precision=prec) for w in wls]
    u0 = [N.initial_state(m, w) for m, w in zip(meshes, wls)]
    b = N.Batch(meshes, cfgs, u0)
    b.set_shape(cells_per_block, 2, form)
    stats = b.advance(max_steps=3)
    for i in range(3):
        s = N.Solver(meshes[i], cfgs[i], u0[i])
        alone = s.advance(np.inf, max_steps=3)[0]
        assert np.array_equal(b.solver(i).get_state()[0], s.get_state()[0])
        assert alone == stats[i]


@pytest.mark.parametrize("prec,blocks_per_chunk", [(N.PREC_FP64, 4), (N.PREC_MIXED, 1)])
def test_blocks_of_a_chunk(prec, blocks_per_chunk):
    wl = W.riemann4_workload(n=32, k=1)            # 2,048 cells
    mesh = N.Mesh.from_mesh(wl.mesh)
    b = N.Batch([mesh], [N.config_for(wl, precision=prec)], [N.initial_state(mesh, wl)])
    b.set_shape(512, 4, 3)
    assert b.shape()["grid"] == 4 * blocks_per_chunk
