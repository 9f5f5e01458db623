"""Cases that a user of this solver runs, from the smallest mesh to the largest.

A case is one call sequence of a user's program through ``native``:

* ``euler``   restart a solver from a stored state, take some SSP-RK3 steps,
              read the state back (``set_state``, ``advance``, ``get_state``);
* ``batch``   the same for several independent solves advanced together;
* ``serve``   hand requests to the server and tick it until all are done;
* ``scalar``  march a scalar solver on by some steps and read the state.

Meshes and states are those of ``workloads`` (vortex, Sedov blast, double Mach
reflection, four-quadrant Riemann problem, forward facing step), with a few
smooth waves of a few per cent laid over the initial data, because a flow that
has run for a while varies in every cell.  FP64 solves return the state as it
is; the mixed form computes in FP32, so its state is returned in FP32.
"""
import functools
import math

import numpy as np
import torch

from paper_2409_09620_gb300 import native as N
from paper_2409_09620_gb300 import workloads as W

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F64 = torch.float64


def listed():
    return [
        # the smallest solve: 2048 cells, P1; every launch of a step counts
        _euler("vortex_2k_p1_fp64", "vortex", 32, 1, "fp64", 64),
        # a small odd-sized request in the mixed form (1058 cells)
        _euler("riemann_1k_p2_mixed", "riemann", 23, 2, "mixed", 64),
        # blast wave, reflecting walls: the middle of the range in FP64
        _euler("sedov_131k_p2_fp64", "sedov", 256, 2, "fp64", 12),
        # unstructured tunnel mesh with a re-entrant corner (72,571 cells)
        _euler("step_73k_p2_fp64", "ffs", 112, 2, "fp64", 16),
        # the other options: component-wise OE, classical decomposition
        _euler("riemann_200k_p1_cw_zxs", "riemann", 316, 1, "fp64", 12, oe=N.OE_CW, decomp=N.DECOMP_ZXS),
        # double Mach reflection on the full grid (1,036,800 cells), both forms
        _euler("dmr_1m_p2_fp64", "dmr", 360, 2, "fp64", 8),
        _euler("dmr_1m_p2_mixed", "dmr", 360, 2, "mixed", 48),
        # the same at half the resolution in P1, mixed (259,200 cells)
        _euler("dmr_259k_p1_mixed", "dmr", 180, 1, "mixed", 48),
        # 16 ragged solves, P1 and P2, 2k-200k cells, advanced together
        {"name": "batch_16_mixed", "kind": "batch", "count": 16, "cmin": 2000, "cmax": 200000, "precision": "mixed",
         "steps": 12, "mesh": 7},
        # six requests of 1k-20k cells through the server
        {"name": "serve_6_mixed", "kind": "serve", "count": 6, "cmin": 1000, "cmax": 20000, "precision": "mixed",
         "steps": 60, "mesh": 11},
        # scalar laws: P3 Burgers (51,200 cells) and P2 convection (204,800 cells)
        {"name": "burgers_51k_p3", "kind": "scalar", "level": 5, "n0": 5, "k": 3, "flux": 1, "steps": 16, "mesh": 31},
        {"name": "linear_205k_p2", "kind": "scalar", "level": 6, "n0": 5, "k": 2, "flux": 0, "steps": 16, "mesh": 31},
    ]


def _euler(name, flow, n, k, precision, steps, oe=N.OE_RI, decomp=N.DECOMP_OPTIMAL, mesh=3):
    c = {"kind": "euler", "flow": flow, "n": n, "k": k, "precision": precision, "steps": steps, "oe": oe,
         "decomp": decomp, "mesh": mesh}
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["euler", "euler", "euler", "euler", "batch", "serve", "scalar"])
    precision = rng.choice(["fp64", "mixed"])
    mesh = rng.randrange(1 << 16)
    if kind == "euler":
        flow = rng.choice(["vortex", "sedov", "riemann", "dmr", "ffs"])
        k = rng.choice([1, 2])
        cells = _log_int(rng, 1000, 700000 if flow != "ffs" else 72000)
        n = {"dmr": math.sqrt(cells / 8.0), "ffs": math.sqrt(cells / 5.8)}.get(flow, math.sqrt(cells / 2.0))
        n = max(8, int(round(n)))
        if flow == "sedov":
            n += n % 2          # a mesh vertex at the blast's origin
        steps = max(4, min(64, int(4e7 // (cells * (8 if precision == "fp64" else 1)))))
        return _euler(None, flow, n, k, precision, steps, oe=rng.choice([N.OE_RI, N.OE_RI, N.OE_CW]),
                      decomp=rng.choice([N.DECOMP_OPTIMAL, N.DECOMP_OPTIMAL, N.DECOMP_ZXS]), mesh=mesh)
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 16), "cmin": 2000, "cmax": rng.choice([20000, 60000, 150000]),
                "precision": precision, "steps": rng.randint(4, 8), "mesh": mesh}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(2, 8), "cmin": 1000, "cmax": rng.choice([5000, 20000]),
                "precision": precision, "steps": rng.randint(20, 50), "mesh": mesh}
    # one uniform refinement multiplies the cells by four: n0 fills the steps between
    return {"kind": "scalar", "level": rng.randint(2, 5), "n0": rng.randint(4, 9), "k": rng.randint(1, 3),
            "flux": rng.randint(0, 1), "steps": rng.randint(8, 24), "mesh": mesh}


# ----------------------------------------------------------------------------
# Inputs: meshes and initial data on the host, coefficients by L2 projection
# ----------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _workload(flow, n, k, mesh):
    """Mesh, boundary data and basic flow: a user's mesh file and set-up."""
    if flow == "vortex":
        return W.vortex_workload(n=n, k=k, seed=mesh)
    if flow == "sedov":
        return W.sedov_workload(n=n, k=k, seed=mesh)
    if flow == "riemann":
        return W.riemann4_workload(n=n, k=k, seed=mesh)
    if flow == "dmr":
        return W.dmr_workload(nx=4 * n, ny=n, k=k, seed=mesh)
    return W.ffs_workload(h=1.0 / n, k=k, seed=mesh)


def _waves(rng, box):
    """A sum of three smooth waves of random direction and phase, at most 1 in magnitude."""
    lx, ly = box[1] - box[0], box[3] - box[2]
    w = [(2 * math.pi * int(rng.integers(1, 5)) / lx, 2 * math.pi * int(rng.integers(1, 5)) / ly,
          float(rng.uniform(0, 2 * math.pi))) for _ in range(3)]

    def f(x, y):
        return sum(torch.sin(a * x + b * y + p) for a, b, p in w) / 3.0
    return f


def _initial(wl, flow, seed):
    """Modal coefficients [4][nb][nt] of the initial data of this seed (on DEV)."""
    rng = np.random.default_rng([int(seed), 17])
    m = wl.mesh
    xy, tri = torch.as_tensor(m.xy, device=DEV), torch.as_tensor(m.tri, device=DEV).long()
    b, w = _rule12()
    p = torch.einsum("mv,kvd->mkd", b, xy[tri])
    x, y = p[..., 0], p[..., 1]
    box = m.box if flow != "ffs" else (0.0, 3.0, 0.0, 1.0)
    f = [_waves(rng, box) for _ in range(4)]
    if flow == "vortex":
        c, s = rng.uniform(0.3, 0.7, 2), rng.uniform(4.5, 5.0)
        u = W.vortex_state(x.cpu().numpy(), y.cpu().numpy(), 0.0, strength=float(s), center=(float(c[0]), float(c[1])))
        u = torch.as_tensor(u, device=DEV)
        rho, vx, vy, pr = _prim(u.movedim(-1, 0))
    elif flow == "sedov":
        u = torch.as_tensor(wl.cell_u0(np.arange(m.nt)), device=DEV)
        rho, vx, vy, pr = (q.expand(12, -1).clone() for q in _prim(u.T))
    elif flow == "riemann":
        q = (x >= 0.5).long() + 2 * (y >= 0.5).long()
        val = [torch.as_tensor(rng.uniform(lo, hi, 4), device=DEV) for lo, hi in
               ((0.1, 2.0), (-1.0, 1.0), (-1.0, 1.0), (0.01, 2.0))]
        rho, vx, vy, pr = (t[q] for t in val)
    elif flow == "dmr":
        behind = x < wl.shock[0] + y / math.sqrt(3.0)
        st = _prim(torch.as_tensor(wl.bc_state[:2], device=DEV).T)   # (post, pre)
        rho, vx, vy, pr = (torch.where(behind, q[0], q[1]) for q in st)
    else:
        rho, vx, vy, pr = (torch.full_like(x, v) for v in (1.4, 3.0, 0.0, 1.0))
    rho, pr = rho * (1 + 0.04 * f[0](x, y)), pr * (1 + 0.04 * f[1](x, y))
    if flow != "sedov":   # the blast starts in gas at rest
        vx, vy = vx + 0.03 * f[2](x, y), vy + 0.03 * f[3](x, y)
    cons = torch.stack([rho, rho * vx, rho * vy, pr / (wl.gamma - 1) + 0.5 * rho * (vx * vx + vy * vy)])
    return _project(cons, (wl.k + 1) * (wl.k + 2) // 2)


def _prim(u, gamma=W.GAMMA):
    v = u[1] / u[0], u[2] / u[0]
    return u[0], v[0], v[1], (gamma - 1) * (u[3] - 0.5 * (u[1] * v[0] + u[2] * v[1]))


def _config(wl, c):
    return N.config_for(wl, precision=N.PREC_MIXED if c["precision"] == "mixed" else N.PREC_FP64,
                        oe=c.get("oe", N.OE_RI), decomp=c.get("decomp", N.DECOMP_OPTIMAL))


def _solves(c):
    """(flow, n, k, mesh seed) of the solves of a batch or of a server's requests."""
    rng = np.random.default_rng([c["mesh"], 5])
    out = []
    for i in range(c["count"]):
        k = int(rng.integers(1, 3))
        cells = math.exp(rng.uniform(math.log(c["cmin"]), math.log(c["cmax"])))
        n = max(4, int(round(math.sqrt(cells / 2.0))))
        flow = "riemann" if c["kind"] == "batch" else ("vortex", "sedov", "riemann")[int(rng.integers(0, 3))]
        out.append((flow, n + (n % 2 if flow == "sedov" else 0), k, c["mesh"] * 100 + i))
    return out


def _scalar_setup(c, seed):
    rng = np.random.default_rng([int(seed), 19])
    m = W.scalar_mesh(c["level"] - 1, n0=c["n0"] * 2, seed=c["mesh"])
    f = _waves(rng, m.box)
    xy, tri = torch.as_tensor(m.xy, device=DEV), torch.as_tensor(m.tri, device=DEV).long()
    p = torch.einsum("mv,kvd->mkd", _rule12()[0], xy[tri])
    s = p[..., 0] + p[..., 1]
    u = 0.5 * torch.sin(2 * math.pi * s + float(rng.uniform(0, 6))) + 0.3 * f(p[..., 0], p[..., 1])
    return m, _project(u[None], (c["k"] + 1) * (c["k"] + 2) // 2)[0]


def _pinned(a):
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory()


# ----------------------------------------------------------------------------
# What a program keeps, and one pass
# ----------------------------------------------------------------------------

def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "euler":
        wl = _workload(c["flow"], c["n"], c["k"], c["mesh"])
        mesh = N.Mesh.from_mesh(wl.mesh)
        s = N.Solver(mesh, _config(wl, c), _initial(wl, c["flow"], seed).cpu().numpy())
        c["solver"], c["start"] = s, _pinned(s.get_state()[0])
        c["out"] = torch.empty_like(c["start"]).pin_memory()
    elif c["kind"] == "batch":
        wls = [(f, _workload(f, n, k, m)) for f, n, k, m in _solves(c)]
        meshes = [N.Mesh.from_mesh(wl.mesh) for _, wl in wls]
        b = N.Batch(meshes, [_config(wl, c) for _, wl in wls],
                    [_initial(wl, f, seed * 100 + i).cpu().numpy() for i, (f, wl) in enumerate(wls)])
        b.set_shape(256, 4, 0)      # each solve's own kernels, side by side
        c["batch"], c["solvers"] = b, [b.solver(i) for i in range(b.n)]
        c["start"] = [_pinned(s.get_state()[0]) for s in c["solvers"]]
        c["out"] = [torch.empty_like(u).pin_memory() for u in c["start"]]
    elif c["kind"] == "serve":
        c["server"] = N.Server(N.PREC_MIXED if c["precision"] == "mixed" else N.PREC_FP64, steps_per_tick=16)
        c["requests"] = []
        for i, (f, n, k, m) in enumerate(_solves(c)):
            wl = _workload(f, n, k, m)
            c["requests"].append((wl.mesh, _config(wl, c), _initial(wl, f, seed * 100 + i).cpu().numpy(),
                                  _end_time(f, n, k, c["steps"])))
    else:
        m, u = _scalar_setup(c, seed)
        cfg = N.make_scalar_config(c["k"], flux=c["flux"])
        c["solver"] = N.ScalarSolver(N.Mesh.from_mesh(m), cfg, u.cpu().numpy())
    return c


def _end_time(flow, n, k, steps):
    """An end time that takes very roughly `steps` steps."""
    alpha = {"vortex": 3.5, "sedov": 1.0e2 * n / 40.0, "riemann": 3.0}[flow]
    return steps * (0.13 if k == 1 else 0.06) * (2.2 if flow == "sedov" else 1.0) / (n * alpha)


def _result(c, u, t):
    """A state as the program keeps it: FP32 for the mixed form."""
    if c["precision"] == "mixed":
        return {"u": torch.as_tensor(u).to(torch.float32), "t": np.float32(t)}
    return {"u": u, "t": np.float64(t)}


def run(state):
    c = state
    if c["kind"] == "euler":
        s = c["solver"]
        s.set_state(c["start"].numpy())
        s.advance(math.inf, max_steps=c["steps"])
        _, t = s.get_state(out=c["out"].numpy())
        return _result(c, c["out"], t)
    if c["kind"] == "batch":
        for s, u in zip(c["solvers"], c["start"]):
            s.set_state(u.numpy())
        c["batch"].advance(max_steps=c["steps"])
        return [_result(c, o, s.get_state(out=o.numpy())[1]) for s, o in zip(c["solvers"], c["out"])]
    if c["kind"] == "serve":
        ids = [c["server"].submit(*r) for r in c["requests"]]
        while any(c["server"].tick()):
            pass
        return [_result(c, c["server"].result(i), c["server"].info(i)["t"]) for i in ids]
    c["solver"].advance(math.inf, max_steps=c["steps"])
    u, t = c["solver"].get_state()
    return {"u": u, "t": np.float64(t)}


# FP64 operations of one cell and stage (an fma is two), and numbers of its state and geometry
FLOPS = {1: 1300.0, 2: 3200.0}
SCALAR_FLOPS = {1: 210.0, 2: 520.0, 3: 1200.0}


def work(case):
    """Bytes: the mesh and the initial state in, the result out, and each stage's
    state in and out once (a stage needs the maxima and means of all cells of the
    one before); operations as the method states them."""
    c = case
    if c["kind"] == "scalar":
        nt = 8 * c["n0"] ** 2 * 4 ** (c["level"] - 1)
        nb, stages = (c["k"] + 1) * (c["k"] + 2) // 2, c["steps"] * (2 if c["k"] == 1 else 3)
        return {"bytes": nt * (8.0 * nb * (2 + 2 * stages) + 60.0), "flops": nt * stages * SCALAR_FLOPS[c["k"]]}
    todo = [(c["flow"], c["n"], c["k"])] if c["kind"] == "euler" else [s[:3] for s in _solves(c)]
    total = {"bytes": 0.0, "flops": 0.0}
    for flow, n, k in todo:
        nt = {"dmr": 8.0 * n * n, "ffs": 5.8 * n * n}.get(flow, 2.0 * n * n)
        nb, stages = (3, 3 * c["steps"]) if k == 1 else (6, 3 * c["steps"])
        s = 4 * nb * 8.0 if c["precision"] == "fp64" else 4 * (8.0 + 4.0 * (nb - 1))
        total["bytes"] += nt * (4 * nb * 16.0 + 60.0 + 2 * s * stages)
        total["flops"] += nt * stages * FLOPS[k]
    return total


# ----------------------------------------------------------------------------
# The same in plain torch, 64 bits
# ----------------------------------------------------------------------------

def exact(case, seed):
    c = dict(case)
    if c["kind"] == "scalar":
        m, u = _scalar_setup(c, seed)
        return _exact_result(*_scalar_march(m, u, c))
    if c["kind"] == "euler":
        wl = _workload(c["flow"], c["n"], c["k"], c["mesh"])
        return _exact_result(*_march(wl, _initial(wl, c["flow"], seed), c, c["steps"], math.inf))
    out = []
    for i, (f, n, k, m) in enumerate(_solves(c)):
        wl = _workload(f, n, k, m)
        serve = c["kind"] == "serve"
        out.append(_exact_result(*_march(wl, _initial(wl, f, seed * 100 + i), c, 1 << 30 if serve else c["steps"],
                                            _end_time(f, n, k, c["steps"]) if serve else math.inf)))
    return out


def _exact_result(u, t):
    return {"u": u, "t": np.float64(t)}


@functools.lru_cache(maxsize=1)
def _rule12():
    a = [(0.063089014491502, 0.063089014491502, 0.873821971016996, 0.050844906370207),
         (0.249286745170910, 0.249286745170910, 0.501426509658180, 0.116786275726379)]
    b = (0.053145049844817, 0.310352451033784, 0.636502499121399, 0.082851075618374)
    pts = [p for q in a for p in ((q[0], q[1], q[2], q[3]), (q[0], q[2], q[1], q[3]), (q[2], q[0], q[1], q[3]))]
    for i, j, l in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        pts.append((b[i], b[j], b[l], b[3]))
    t = torch.tensor(pts, dtype=F64, device=DEV)
    return t[:, :3].contiguous(), t[:, 3].contiguous()


# the basis: coefficients of xi^p eta^q, and int Psi^2 / |K|
_POLY = [{(0, 0): 1},
         {(1, 0): 4, (0, 1): 2, (0, 0): -2},
         {(0, 1): 3, (0, 0): -1},
         {(2, 0): 24, (1, 1): 24, (0, 2): 4, (1, 0): -24, (0, 1): -8, (0, 0): 4},
         {(1, 1): 20, (0, 2): 10, (1, 0): -4, (0, 1): -12, (0, 0): 2},
         {(0, 2): 10, (0, 1): -8, (0, 0): 1},
         {(3, 0): 160, (2, 1): 240, (1, 2): 96, (0, 3): 8, (2, 0): -240, (1, 1): -192, (0, 2): -24, (1, 0): 96,
          (0, 1): 24, (0, 0): -8},
         {(2, 1): 168, (1, 2): 168, (0, 3): 28, (2, 0): -24, (1, 1): -192, (0, 2): -60, (1, 0): 24, (0, 1): 36,
          (0, 0): -4},
         {(1, 2): 84, (0, 3): 42, (1, 1): -48, (0, 2): -66, (1, 0): 4, (0, 1): 26, (0, 0): -2},
         {(0, 3): 35, (0, 2): -45, (0, 1): 15, (0, 0): -1}]
_MASS = [1, 2 / 3, 1 / 2, 16 / 15, 4 / 9, 1 / 3, 16 / 7, 4 / 5, 1 / 3, 1 / 4]


def _psi(nb, x, y, r=0, s=0):
    """d^(r+s) Psi_l / dxi^r deta^s at points (x, y), l = 0..nb-1 first."""
    x, y = torch.as_tensor(x, dtype=F64, device=DEV), torch.as_tensor(y, dtype=F64, device=DEV)
    out = []
    for l in range(nb):
        v = torch.zeros_like(x)
        for (p, q), a in _POLY[l].items():
            if p >= r and q >= s:
                v = v + a * math.perm(p, r) * math.perm(q, s) * x ** (p - r) * y ** (q - s)
        out.append(v)
    return torch.stack(out)


def _project(vals, nb):
    """vals[c][12][nt] at the 12-point rule -> modal coefficients [c][nb][nt]."""
    b, w = _rule12()
    psi = _psi(nb, b[:, 1], b[:, 2]) * w / torch.tensor(_MASS[:nb], dtype=F64, device=DEV)[:, None]
    return torch.einsum("lm,cmk->clk", psi, vals).contiguous()


class _Geo:
    """Adjacency, geometry and point tables of a mesh for degree k."""

    def __init__(self, m, k):
        tri = np.asarray(m.tri, np.int64)
        self.nt, self.k, self.nb = tri.shape[0], k, (k + 1) * (k + 2) // 2
        nt, ca = self.nt, np.asarray(m.canon, np.int64)[tri]
        a, b = ca[:, [1, 2, 0]].T.reshape(-1), ca[:, [2, 0, 1]].T.reshape(-1)      # edge i * nt + K
        key = np.minimum(a, b) * (int(ca.max()) + 1) + np.maximum(a, b)
        o = np.argsort(key, kind="stable")
        other = np.full(3 * nt, -1, np.int64)
        same = key[o[1:]] == key[o[:-1]]
        other[o[1:][same]], other[o[:-1][same]] = o[:-1][same], o[1:][same]
        self.inner = torch.as_tensor(other >= 0, device=DEV).view(3, nt)
        self.other = torch.as_tensor(np.where(other >= 0, other, 0), device=DEV).view(3, nt)
        tag = torch.as_tensor(np.asarray(m.bc, np.int64).T.copy(), device=DEV)
        self.bnd = [(t, (~self.inner & (tag == t)).nonzero(as_tuple=True)) for t in
                    sorted(set(tag[~self.inner].tolist()))]
        v = torch.as_tensor(m.xy, device=DEV)[torch.as_tensor(tri, device=DEV)]          # [nt, 3, 2]
        self.v = v
        j = torch.stack([v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]], dim=-1)                   # d(x, y) / d(xi, eta)
        det = j[:, 0, 0] * j[:, 1, 1] - j[:, 0, 1] * j[:, 1, 0]
        self.area = 0.5 * det
        self.jx, self.jy, self.ex, self.ey = (j[:, 1, 1] / det, -j[:, 0, 1] / det, -j[:, 1, 0] / det, j[:, 0, 0] / det)
        e = torch.stack([v[:, (i + 2) % 3] - v[:, (i + 1) % 3] for i in range(3)])        # [3, nt, 2]
        self.len = e.norm(dim=-1)
        self.nx, self.ny = e[..., 1] / self.len, -e[..., 0] / self.len
        self.h = 2 * self.area / self.len
        g, w = np.polynomial.legendre.leggauss(k + 1)
        self.s = [(1 + q) / 2 for q in g]
        self.w = torch.tensor(w / 2, dtype=F64, device=DEV)
        pts = [((1 - s, s), (0.0, 1 - s), (s, 0.0)) for s in self.s]
        ex = torch.tensor([[pts[q][i][0] for q in range(k + 1)] for i in range(3)], dtype=F64, device=DEV)
        ey = torch.tensor([[pts[q][i][1] for q in range(k + 1)] for i in range(3)], dtype=F64, device=DEV)
        self.edge = _psi(self.nb, ex, ey)                                                 # [nb, 3, Q]
        if k == 1:
            xs, ys, ws = [1 / 6, 2 / 3, 1 / 6], [2 / 3, 1 / 6, 1 / 6], [1 / 3] * 3
        elif k == 2:
            p, q, r, s = 0.445948490915965, 0.108103018168070, 0.091576213509771, 0.816847572980458
            xs, ys, ws = [p, q, p, r, s, r], [q, p, p, s, r, r], [0.223381589678010] * 3 + [0.109951743655322] * 3
        else:
            b12, w12 = _rule12()
            xs, ys, ws = b12[:, 1], b12[:, 2], w12
        self.vol, self.vol_x, self.vol_y = (_psi(self.nb, xs, ys, *d) for d in ((0, 0), (1, 0), (0, 1)))
        self.vw = torch.as_tensor(ws, dtype=F64, device=DEV)
        self.vert = {(r, s): _psi(self.nb, [0.0, 1.0, 0.0], [0.0, 0.0, 1.0], r, s)
                     for r in range(k + 1) for s in range(k + 1 - r)}
        self.imass = 1 / torch.tensor(_MASS[:self.nb], dtype=F64, device=DEV)

    def across(self, t):
        """t[..., 3, Q, nt] at the edge points -> the neighbour's values there."""
        q = t.flip(-2).transpose(-3, -2)
        return q.reshape(*q.shape[:-2], -1)[..., self.other].transpose(-3, -2)

    def vertices_across(self, f):
        """f[..., 3, nt] at the vertices -> own and neighbour's values [..., 2, 3, nt] at the ends of each edge."""
        own = torch.stack([f.roll(-1 - e, dims=-2) for e in (0, 1)], dim=-3)
        jn, nb = self.other // self.nt, self.other % self.nt
        flat = f.reshape(*f.shape[:-2], -1)
        return own, torch.stack([flat[..., ((jn + 2 - e) % 3) * self.nt + nb] for e in (0, 1)], dim=-3)


def _reflect(v, nx, ny):
    mn = 2 * (v[1] * nx + v[2] * ny)
    return torch.stack([v[0], v[1] - mn * nx, v[2] - mn * ny, v[3]])


def _outside(wl, tag, own, mean, x, y, t):
    """Constant exterior state of a boundary tag other than a wall, shaped like own."""
    if tag == 2:
        return mean.expand_as(own)
    bc = torch.as_tensor(wl.bc_state, device=DEV)
    if tag != 7:
        return bc[tag - 3].view(4, *[1] * (own.dim() - 1)).expand_as(own)
    x0, angle, speed, pre, post = wl.shock
    line = x0 + y / math.tan(angle) + t * speed / math.sin(angle)
    return torch.where(x < line, bc[post].view(4, *[1] * x.dim()), bc[pre].view(4, *[1] * x.dim()))


def _flux(u, nx, ny, g):
    p = (g - 1) * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])
    vn = (u[1] * nx + u[2] * ny) / u[0]
    return torch.stack([u[0] * vn, u[1] * vn + p * nx, u[2] * vn + p * ny, (u[3] + p) * vn])


def _speed(u, nx, ny, g):
    p = (g - 1) * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])
    r = ((u[1] * nx + u[2] * ny) / u[0]).abs() + (g * p.clamp(min=0) / u[0]).sqrt()
    return torch.where(u[0] > 0, r, math.inf)


def _edge_points(G, i, K):
    s = torch.tensor(G.s, dtype=F64, device=DEV)
    a, b = G.v[K, (i + 1) % 3], G.v[K, (i + 2) % 3]
    p = a + s[:, None, None] * (b - a)
    return p[..., 0], p[..., 1]


def _alpha(G, wl, U, t):
    tr = torch.einsum("liq,clk->ciqk", G.edge, U)
    best = _speed(tr, G.nx[:, None], G.ny[:, None], wl.gamma).max()
    for tag, (i, K) in G.bnd:
        if tag != 1:
            x, y = _edge_points(G, i, K)
            out = _outside(wl, tag, tr[:, i, :, K].movedim(0, -1), U[:, 0, None, K], x, y, t)
            best = torch.maximum(best, _speed(out, G.nx[i, K], G.ny[i, K], wl.gamma).max())
    return float(best)


def _space(G, wl, U, alpha, t):
    """dt-free right-hand side of every mode, divided by its mass."""
    g = wl.gamma
    u = torch.einsum("lm,clk->cmk", G.vol, U)
    R = torch.einsum("lm,cmk->clk", G.vol_x * G.vw, _flux(u, G.jx, G.jy, g)) + \
        torch.einsum("lm,cmk->clk", G.vol_y * G.vw, _flux(u, G.ex, G.ey, g))
    tr = torch.einsum("liq,clk->ciqk", G.edge, U)
    ot = G.across(tr)
    for tag, (i, K) in G.bnd:
        own = tr[:, i, :, K].movedim(0, -1)                       # [4, Q, edges]
        x, y = _edge_points(G, i, K)
        gh = _reflect(own, G.nx[i, K], G.ny[i, K]) if tag == 1 else _outside(wl, tag, own, U[:, 0, None, K], x, y, t)
        ot[:, i, :, K] = gh.movedim(-1, 0)
    nx, ny = G.nx[:, None], G.ny[:, None]
    fh = 0.5 * (_flux(tr, nx, ny, g) + _flux(ot, nx, ny, g) - alpha * (ot - tr))
    R -= torch.einsum("liq,ciqk->clk", G.edge * G.w, fh * (G.len / G.area)[:, None])
    return R * G.imass[:, None]


def _oe(G, wl, U, dt, t, cw):
    k, nt = G.k, G.nt
    mean = (G.area * U[:, 0]).sum(-1) / G.area.sum()
    d = torch.einsum("lm,clk->cmk", G.vol, U) - mean[:, None, None]
    m2 = (mean[1] ** 2 + mean[2] ** 2).sqrt()
    dm = [(d[q].abs().max(), mean[q].abs()) for q in (1, 2)] if cw else [((d[1] ** 2 + d[2] ** 2).sqrt().max(), m2)] * 2
    D = [(d[0].abs().max(), mean[0].abs()), *dm, (d[3].abs().max(), mean[3].abs())]
    iD = [0.0 if float(a) <= 1e-12 * max(1.0, float(b)) else 1.0 / float(a) for a, b in D]
    # physical derivatives at the vertices, by order
    ref = {rs: torch.einsum("lv,clk->cvk", G.vert[rs], U) for rs in G.vert}
    der = {0: [(1.0, ref[0, 0])],
           1: [(1.0, ref[1, 0] * G.jx + ref[0, 1] * G.ex), (1.0, ref[1, 0] * G.jy + ref[0, 1] * G.ey)]}
    if k == 2:
        def second(a, b, c, e):
            return ref[2, 0] * (a * c) + ref[1, 1] * (a * e + b * c) + ref[0, 2] * (b * e)
        der[2] = [(1.0, second(G.jx, G.ex, G.jx, G.ex)), (2.0, second(G.jx, G.ex, G.jy, G.ey)),
                  (1.0, second(G.jy, G.ey, G.jy, G.ey))]
    nx, ny = G.nx, G.ny
    pairs = {j: [(w, *G.vertices_across(f)) for w, f in der[j]] for j in der}
    for tag, (i, K) in G.bnd:                                      # exterior polynomials at the boundary
        n0, n1 = nx[i, K], ny[i, K]
        r = torch.stack([torch.stack([1 - 2 * n0 * n0, -2 * n0 * n1]), torch.stack([-2 * n0 * n1, 1 - 2 * n1 * n1])])
        own = {j: torch.stack([p[1][:, :, i, K] for p in pairs[j]]) for j in pairs}       # [derivative, 4, 2, edges]
        if tag == 1:
            turn = {0: own[0], 1: torch.einsum("abe,bcve->acve", r, own[1])}
            if k == 2:
                full = torch.stack([torch.stack([own[2][0], own[2][1]]), torch.stack([own[2][1], own[2][2]])])
                full = torch.einsum("abe,bdcve,dfe->afcve", r, full, r)
                turn[2] = torch.stack([full[0, 0], full[0, 1], full[1, 1]])
            out = {j: torch.stack([_reflect(q, n0, n1) for q in turn[j]]) for j in turn}
        else:
            p = torch.stack([G.v[K, (i + 1) % 3], G.v[K, (i + 2) % 3]])
            out = {j: torch.zeros_like(own[j]) for j in own}
            out[0] = _outside(wl, tag, own[0][0], U[:, 0, None, K], p[..., 0], p[..., 1], t)[None]
        for j in pairs:
            for q, f in zip(pairs[j], out[j]):
                q[2][:, :, i, K] = f
    beta = torch.maximum(*[_speed(f, nx, ny, wl.gamma) for f in pairs[0][0][1:]]).amax(0)
    sig = U.new_zeros(4, k + 1, nt)
    for j in range(k + 1):
        J = 0.0
        for w, own, oth in pairs[j]:
            q = own - oth
            if not cw:
                q = torch.stack([q[0], q[1] * nx + q[2] * ny, q[2] * nx - q[1] * ny, q[3]])
            J = J + 0.5 * w * (q * q).sum(1)
        root = J.sqrt()
        if not cw:
            root[1] = root[2] = torch.maximum(root[1], root[2])
        A = (2 * j + 1) / ((2 * k - 1) * math.factorial(j))
        sig[:, j] = (torch.where(root > 0, beta / G.h * A * G.h ** j * root, 0.0)).sum(1)
    scale = torch.tensor(iD, dtype=F64, device=DEV)[:, None, None]
    sig = torch.where(scale > 0, sig * scale, 0.0)
    cum = torch.exp(-dt * torch.cumsum(sig, 1))
    out = U.clone()
    out[:, 1:3] *= cum[:, 1:2]
    if k == 2:
        out[:, 3:6] *= cum[:, 2:3]
    return out


def _extra_points(G, zxs):
    """Basis values [nb, 2, nt] at the limiter's points beside the edge points."""
    if zxs:
        if G.k == 1:
            return G.edge[:, 0, :1, None].expand(-1, 2, G.nt)
        e = -(G.edge * G.w).sum((1, 2)) / 6
        e[0] = 1.0
        return e[:, None, None].expand(-1, 2, G.nt)
    order = torch.argsort(G.len, dim=0, descending=True, stable=True)
    if G.k == 1:
        v = order[:2]
        return _psi(G.nb, (v == 1).to(F64), (v == 2).to(F64))
    l1, l2, l3 = torch.gather(G.len, 0, order)
    r = math.sqrt(3.0)
    lb = (l1 + l2 + l3) / 3
    lh = (l1 ** 2 + l2 ** 2 + l3 ** 2 - 2 / 3 * (l1 * l2 + l2 * l3 + l3 * l1)).sqrt()
    xi, eta = [], []
    for s in (r, -r):
        q = [((6, 6 + 2 * s, 6, 1, -2, -s - 2), 3 * l1 + 3 * l2 + s * (l2 - l3)),
             ((6, 12, 6, -s - 2, -2, s - 2), 6 * l2 + s * (l3 - l1)),
             ((6, 6 - 2 * s, 6, s - 2, -2, 1), 3 * l2 + 3 * l3 + s * (l1 - l2))]
        b = torch.stack([(a[0] * l1 ** 2 + a[1] * l2 ** 2 + a[2] * l3 ** 2 + 2 * (a[3] * l1 * l2 + a[4] * l1 * l3 + a[5] * l2 * l3)
                          + 2 * c * lh) / (18 * (lb + lh) * (l2 + lh)) for a, c in q])
        full = torch.zeros_like(b).scatter_(0, order, b)
        xi.append(full[1])
        eta.append(full[2])
    return _psi(G.nb, torch.stack(xi), torch.stack(eta))


def _limit(G, U, extra):
    a = U[:, 0]
    dev = torch.cat([torch.einsum("liq,clk->ciqk", G.edge[1:], U[:, 1:]).flatten(1, 2),
                     torch.einsum("lpk,clk->cpk", extra[1:], U[:, 1:])], dim=1)
    rho, ie = a[0], a[3] - 0.5 * (a[1] ** 2 + a[2] ** 2) / a[0]
    rmin = (rho + dev[0]).amin(0)
    e1, e2 = rho.clamp(max=1e-13), ie.clamp(max=1e-13)
    th1 = torch.where(rmin < e1, (rho - e1) / (rho - rmin), 1.0)
    w = a[:, None] + dev
    w0 = rho + th1 * dev[0]
    emin = (w[3] - 0.5 * (w[1] ** 2 + w[2] ** 2) / w0).amin(0)
    th2 = torch.where(emin < e2, (ie - e2) / (ie - emin), 1.0)
    out = U.clone()
    out[:, 1:] *= th2
    out[0, 1:] *= th1
    return out


def _march(wl, U, c, steps, t_end):
    k = wl.k
    G = _Geo(wl.mesh, k)
    zxs, cw = c.get("decomp", 0) == N.DECOMP_ZXS, c.get("oe", N.OE_RI) == N.OE_CW
    extra = _extra_points(G, zxs)
    l1, l2, l3 = torch.sort(G.len, dim=0, descending=True)[0]
    lb = (l1 + l2 + l3) / 3
    lh = (l1 ** 2 + l2 ** 2 + l3 ** 2 - 2 / 3 * (l1 * l2 + l2 * l3 + l3 * l1)).clamp(min=0).sqrt()
    C = (1 / (9 * lb) if k == 1 else 1 / (27 * lb)) if zxs else (2 / (3 * (l1 + l2)) if k == 1 else 2 / (9 * lb + 3 * lh))
    cmin = float((C * G.area).min())
    U, t = _limit(G, U, extra), 0.0
    alpha = _alpha(G, wl, U, t)
    for _ in range(steps):
        if t >= t_end:
            break
        dt = cmin / alpha
        last = t + dt >= t_end
        dt = t_end - t if last else dt
        V = U
        for a, b, ci, co in ((0.0, 1.0, 0.0, 1.0), (0.75, 0.25, 1.0, 0.5), (1 / 3, 2 / 3, 0.5, 1.0)):
            V = b * (V + dt * _space(G, wl, V, alpha, t + ci * dt)) + (a * U if a else 0.0)
            V = _limit(G, _oe(G, wl, V, dt, t + co * dt, cw), extra)
            alpha = _alpha(G, wl, V, t + co * dt)
        U, t = V, t_end if last else t + dt
    return U, t


def _scalar_march(m, u, c):
    k = c["k"]
    G = _Geo(m, k)

    def flux(u, nx, ny):
        return u * (nx + ny) if c["flux"] == 0 else 0.5 * u * u * (nx + ny)

    def speed(u):
        s = G.nx + G.ny
        return (s if c["flux"] == 0 else u * s).abs().expand_as(u)

    base = float((G.area / ((2 * k + 1) * G.len.sum(0))).min())
    rk = ((0.0, 1.0), (0.5, 0.5)) if k == 1 else ((0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3))
    deg = [int(j) for j in (0, 1, 1, 2, 2, 2, 3, 3, 3, 3)[:G.nb]]

    def top(u):
        return float(speed(torch.einsum("liq,lk->qik", G.edge, u)).max())

    alpha, t = top(u), 0.0
    for _ in range(c["steps"]):
        dt = base / alpha
        v = u
        for a, b in rk:
            q = torch.einsum("lm,lk->mk", G.vol, v)
            R = torch.einsum("lm,mk->lk", G.vol_x * G.vw, flux(q, G.jx, G.jy)) + \
                torch.einsum("lm,mk->lk", G.vol_y * G.vw, flux(q, G.ex, G.ey))
            tr = torch.einsum("liq,lk->iqk", G.edge, v)
            ot = G.across(tr)
            fh = 0.5 * (flux(tr, G.nx[:, None], G.ny[:, None]) + flux(ot, G.nx[:, None], G.ny[:, None]) - alpha * (ot - tr))
            R -= torch.einsum("liq,iqk->lk", G.edge * G.w, fh * (G.len / G.area)[:, None])
            v = b * (v + dt * R * G.imass[:, None]) + a * u
            mean = float((G.area * v[0]).sum() / G.area.sum())
            dev = float((torch.einsum("lm,lk->mk", G.vol, v) - mean).abs().max())
            if dev > 1e-12 * max(1.0, abs(mean)):
                ref = {rs: torch.einsum("lv,lk->vk", G.vert[rs], v) for rs in G.vert}
                sig = []
                beta = None
                for j in range(k + 1):
                    J = 0.0
                    for p in range(j, -1, -1):       # d^j / dx^p dy^(j-p)
                        co = [torch.ones_like(G.jx)]                            # coefficients of Dxi^r Deta^(n-r)
                        for f in range(j):
                            fa, fb = (G.jx, G.ex) if f < p else (G.jy, G.ey)
                            co = [(fb * co[r] if r < len(co) else 0) + (fa * co[r - 1] if r else 0) for r in range(len(co) + 1)]
                        own, oth = G.vertices_across(sum(co[r] * ref[r, j - r] for r in range(j + 1)))
                        if j == 0:
                            beta = torch.maximum(speed(own), speed(oth)).amax(0)
                        J = J + 0.5 * math.comb(j, p) * ((own - oth) ** 2).sum(0)
                    A = (2 * j + 1) / ((2 * k - 1) * math.factorial(j))
                    sig.append((beta / G.h * A * G.h ** j * J.sqrt()).sum(0) / dev)
                cum = torch.exp(-dt * torch.cumsum(torch.stack(sig), 0))
                v = torch.stack([v[l] if l == 0 else v[l] * cum[deg[l]] for l in range(G.nb)])
            alpha = top(v)
        u, t = v, t + dt
    return u, t
