"""The device bytes a server charges for a solve (``solve_bytes`` of ``csrc/dg_serve_sched.cpp``,
on the CPU) against a count of the arrays that dg_mesh_create and dg_init allocate: never less,
and no more than the fixed 4 KB above it, for closed meshes (1.5 edges per cell), strips one cell
wide (2) and small meshes of separate triangles (3); tags on interior edges, which the mesh
ignores, cost no more than a strip."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2409_09620_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "dg_serve_sched.h"
int main() {
  long long nt, tagged;
  int k, p;
  while (std::scanf("%lld %lld %d %d", &nt, &tagged, &k, &p) == 4)
    std::printf("%zu\n", dg::solve_bytes(nt, tagged, k, p));
  return 0;
}
"""


def _count(nt, boundary, k, precision):
    """Bytes of the arrays, one by one (precision 0 FP64, 1 mixed)."""
    ne = (3 * nt + boundary) // 2
    tiles = -(-nt // 32)
    real, modes = (8, 4) if precision else (8, 8)
    nm = 2 if k == 1 else 5
    mesh = (8 * nt * (1 + 4 + 6 + 3 + 6 + 6 + 4 + 4 + 1 + 10)      # area jinv nrm len hgeo vxy node c_area iarea psi_node
            + 4 * nt * (4 + 6 + 3 + 6 + 4)                         # jinv_f nrm_f len_f hgeo_f node_f
            + 2 * nt + 4 * 3 * nt + 4 * 3 * nt                     # limv conn cedge
            + 4 * ne + ne + 4 * (tiles + 1))                       # e_cell e_loc etile
    state = 3 * nt * (4 * real + 4 * nm * modes)
    exchange = 0 if precision else 8 * (nt * 3 * (k + 1) * 8 + nt * 52 + nt * 12 + ne * 16)   # tr vd hs ej
    parts = -(-nt // (128 if precision else 32))
    groups = -(-parts // 128)
    sums = (parts + groups) * (4 * 8 + 5 * 8 + 8 + 2 * 8) + 4 * 3 * (groups + 1)
    return mesh + state + exchange + sums


def test_charge_covers_the_arrays(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "driver.cpp"),
                    os.path.join(CSRC, "dg_serve_sched.cpp"), "-o", str(exe)], check=True)
    cases = []
    for nt in (1, 2, 30, 31, 33, 128, 1000, 50000, 1036800):
        for boundary in (nt % 2, nt, 3 * nt):       # closed, a strip one cell wide, separate triangles
            if boundary <= nt or nt <= 30:
                cases += [(nt, boundary, k, p) for k in (1, 2) for p in (0, 1)]
    cases += [(50000, 3 * 50000, k, p) for k in (1, 2) for p in (0, 1)]
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c in cases) + "\n", capture_output=True,
                         text=True, check=True).stdout.split()
    assert len(out) == len(cases)
    for c, b in zip(cases, out):
        need = _count(c[0], c[0], *c[2:]) if c[1] > c[0] > 30 else _count(*c)
        assert need <= int(b) <= need + 4200, (c, need, int(b))
