"""Performance cases of the WENO3 library: what a program that uses it asks of it, over the sizes,
mesh kinds, precisions and options in real use.

A case names a mesh (cell kind, nx x ny base quads, box), the data on it, the solver's options and
one operation of the Python API:

  step       Solver.step, one SSP-RK3 step in place: the inner loop of a simulation
  instances  Solver.step_instances: one step of many independent meshes, a time step for each
  adaptive   Solver.max_dt, then Solver.step with it: a loop whose time step follows the state
  residual   Solver.residual: L(W) alone, for a program with its own time integrator
  monitor    Solver.max_dt and Solver.conservation: what a run logs every so many steps

Meshes and data are seeded: another seed displaces the nodes, splits the quads and draws the states
anew.  An FP32C state U + U_lo lives in one (2, n_cells, n_v) buffer, which is what a step returns.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1712_08317_gb300.api import Mesh, Solver

GAMMA, EPS, THETA, CFL = 1.4, 1e-3, 3.0, 0.4
SPLIT = {"quad": 0.0, "mixed": 0.3, "tri": 1.0}  # share of the base quads cut into two triangles
EXACT_CELLS = 60_000                             # above it the 64-bit reference takes too long


def _case(name, op, kind, nx, ny, box, data, precision, eqn="euler", characteristic=False, linear=False, count=1,
          autotune=False):
    c = {"op": op, "kind": kind, "nx": nx, "ny": ny, "box": box, "data": data, "precision": precision, "eqn": eqn,
         "characteristic": characteristic, "linear": linear, "count": count, "autotune": autotune}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a production run: the mixed low-quality vortex mesh, 1.0M cells, tuned once, thousands of steps
        _case("vortex_1m_fp32c", "step", "mixed", 877, 877, "stretched", "vortex", "fp32c", autotune=True),
        # the same family at a size whose tables are about as large as the L2 cache
        _case("vortex_133k_fp32c", "step", "mixed", 320, 320, "stretched", "vortex", "fp32c"),
        # the density-wave convergence ladder on triangles: its finest and its coarsest level
        _case("wave_51k_tri_fp32c", "step", "tri", 160, 160, "periodic", "wave", "fp32c"),
        _case("wave_800_tri_fp32c", "step", "tri", 20, 20, "periodic", "wave", "fp32c"),
        # scalar advection on 1,600 perturbed quads, the smallest verification run, in FP64
        _case("scalar_1600_quad_fp64", "step", "quad", 40, 40, "periodic", "scalar", "fp64", eqn="scalar"),
        # an FP64 reference run of the low-quality vortex
        _case("vortex_33k_fp64", "step", "mixed", 160, 160, "stretched", "vortex", "fp64"),
        # an FP64 right-hand side for another integrator: a four-quadrant problem with outflow, odd sizes
        _case("riemann_53k_fp64", "residual", "mixed", 223, 183, "outflow", "riemann", "fp64"),
        # a parameter study: 24 ragged instances of all cell kinds in one launch, each with its own time step
        _case("batch_24_fp32c", "instances", "all", 40, 140, "periodic", "wave", "fp32c", count=24, autotune=True),
        # Sod's shock tube in characteristic variables on triangles between reflective walls
        _case("sod_10k_tri_char_fp32c", "step", "tri", 100, 50, "tube", "sod", "fp32c", characteristic=True),
        # double Mach reflection: characteristic variables in FP64, moving inflow states, a partial wall
        _case("dmr_40k_quad_char_fp64", "residual", "quad", 400, 100, "dmr", "dmr", "fp64", characteristic=True),
        # a small FP64 run with a CFL time step from the state at every step
        _case("adaptive_8k_quad_fp64", "adaptive", "quad", 97, 83, "periodic", "wave", "fp64"),
        # the log line of a medium run
        _case("monitor_260k_fp32c", "monitor", "mixed", 449, 447, "periodic", "wave", "fp32c"),
    ]


def draw(rng):
    def size(lo, hi):  # base quads a side, spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["quad", "tri", "mixed"])
    family = rng.choice(["fp32c", "fp32c", "fp64", "scalar", "riemann", "batch", "char", "char64", "adaptive",
                         "monitor"])
    if family == "fp32c":
        n, box = size(8, 620), rng.choice(["periodic", "stretched"])
        n = max(n, 100) if box == "stretched" else n  # the stretched family is unstable on coarse meshes
        return _case(None, "step", kind, n, max(8, n - rng.randrange(8)), box, "vortex" if box == "stretched" else "wave",
                     "fp32c", linear=rng.random() < 0.1, autotune=rng.random() < 0.3)
    if family == "fp64":
        n = size(8, 200)
        return _case(None, "step", kind, n, max(8, n - rng.randrange(8)), "periodic", "wave", "fp64",
                     linear=rng.random() < 0.1)
    if family == "scalar":
        n = size(8, 300)
        return _case(None, "step", kind, n, n, "periodic", "scalar", rng.choice(["fp64", "fp32c"]), eqn="scalar")
    if family == "riemann":
        n = size(8, 200)
        return _case(None, "residual", kind, n, max(8, n - rng.randrange(20)), "outflow", "riemann", "fp64")
    if family == "batch":
        lo = size(8, 40)
        return _case(None, "instances", "all", lo, lo * rng.randrange(2, 5), "periodic", "wave",
                     rng.choice(["fp32c", "fp32c", "fp64"]), count=rng.randrange(3, 20))
    if family == "char":
        n = size(16, 300)
        return _case(None, "step", kind, n, max(8, n // 2), "tube", "sod", "fp32c", characteristic=True)
    if family == "char64":
        n = size(8, 90)
        return _case(None, "residual", "quad", 4 * n, n, "dmr", "dmr", "fp64", characteristic=True)
    if family == "adaptive":
        n = size(8, 150)
        return _case(None, "adaptive", kind, n, n + rng.randrange(8), "periodic", "wave", "fp64")
    n = size(8, 500)
    return _case(None, "monitor", kind, n, n, "periodic", "wave", rng.choice(["fp32c", "fp32c", "fp64"]))


# ------------------------------------------------------------------ meshes and data
class _Box:
    """One mesh: node coordinates, cells (n, 4) counter-clockwise (last id repeated in triangles) and
    their node counts, the boundary description and the solver options that go with it."""

    def __init__(self, kind, nx, ny, box, seed):
        rng = np.random.default_rng(seed)
        self.periodic = box in ("periodic", "stretched")
        self.extent = {"periodic": (2.0, 2.0), "stretched": (10.0, 10.0), "outflow": (1.0, 1.0), "tube": (1.0, 0.5),
                       "dmr": (4.0, 1.0)}[box]
        self.walls, self.wall_from, self.inflow, self.options = (), (0.0, 0.0, 0.0, 0.0), (), {}
        if box == "tube":
            self.walls = (2, 3)
        if box == "dmr":  # a Mach 10 shock at 60 degrees through (1/6, 0) into resting gas
            s, c = math.sin(math.pi / 3), math.cos(math.pi / 3)
            self.walls, self.wall_from, self.inflow = (2,), (0.0, 0.0, 1.0 / 6.0, 0.0), (0, 2, 3)
            self.options = {"inflow_a": (8.0, 8.25 * s, -8.25 * c, 116.5), "inflow_b": (1.4, 0.0, 0.0, 1.0),
                            "inflow_line": (s, -c, s / 6.0, 10.0)}
        X, Y = (e * np.arange(n + 1) / n for e, n in zip(self.extent, (nx, ny)))
        if box == "stretched":  # spacings vary by a factor 10 in x and y, out of phase
            L, a = self.extent[0], 9.0 / 11.0

            def g(s):
                return s - a * L / (2 * math.pi) * np.sin(2 * math.pi * s / L)
            X, Y = g(X), g(Y + L / 4) - g(L / 4)
        X[-1], Y[-1] = self.extent
        delta = 0.4 if box == "stretched" else 0.1
        xx, yy = np.meshgrid(X, Y)
        base = np.stack([xx.ravel(), yy.ravel()], 1)
        i, j = (v.ravel() for v in np.meshgrid(np.arange(nx), np.arange(ny)))
        a = i + (nx + 1) * j
        quads = np.stack([a, a + 1, a + nx + 2, a + nx + 1], 1)
        dx, dy = np.diff(X), np.diff(Y)
        amp = np.zeros((ny + 1, nx + 1, 2))  # interior nodes move by up to delta of the local spacing
        amp[1:-1, 1:-1, 0] = delta * np.minimum(dx[1:], dx[:-1])[None]
        amp[1:-1, 1:-1, 1] = delta * np.minimum(dy[1:], dy[:-1])[:, None]
        amp = amp.reshape(-1, 2)
        self.nodes = base + rng.uniform(-1, 1, base.shape) * amp
        floor = 0.2 * (dx[None] * dy[:, None]).ravel()
        look = np.arange(len(quads))
        while look.size:  # no corner of a quad becomes a sliver: its nodes are drawn again
            p = self.nodes[quads[look]]
            e = np.roll(p, -1, 1) - p
            f = np.roll(e, -1, 1)
            bad = np.unique(quads[look][((e[..., 0] * f[..., 1] - e[..., 1] * f[..., 0]) <= floor[look, None]).any(1)])
            self.nodes[bad] = base[bad] + rng.uniform(-1, 1, (bad.size, 2)) * amp[bad]
            drawn = np.zeros(len(base), bool)
            drawn[bad] = True
            look = np.flatnonzero(drawn[quads].any(1))
        cut = np.arange(len(quads)) < round(SPLIT[kind] * len(quads))  # as many for every seed
        rng.shuffle(cut)
        q = np.where((rng.random(len(quads)) < 0.5)[:, None], quads, np.roll(quads, -1, 1))
        tri = [np.stack([q[:, 0], q[:, k], q[:, k + 1], q[:, k + 1]], 1) for k in (1, 2)]
        self.cells = np.where(cut[:, None, None], np.stack(tri, 1), np.stack([quads, quads], 1)).reshape(-1, 4)
        keep = np.stack([np.ones_like(cut), cut], 1).ravel()
        self.cells, self.count = self.cells[keep], np.where(np.repeat(cut, 2)[keep], 3, 4)

    def handle(self):
        mask = np.arange(4)[None] < self.count[:, None]
        ptr = np.concatenate([[0], np.cumsum(self.count)])
        return Mesh(self.nodes, ptr, self.cells[mask], "periodic" if self.periodic else "outflow", (0.0, 0.0),
                    self.extent, self.walls, self.wall_from, self.inflow)

    def average(self, f):
        """Cell averages of f(x, y) (n_v, ...) by the edge-midpoint rule on each cell's fan of triangles."""
        p = self.nodes[self.cells]
        total, area = 0.0, 0.0
        for k in (1, 2):
            a, b, c = p[:, 0], p[:, k], p[:, k + 1]
            t = 0.5 * ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0]))
            for m in ((a + b) / 2, (b + c) / 2, (c + a) / 2):
                total = total + t / 3 * f(m[:, 0], m[:, 1])
            area = area + t
        return total / area, area

    def stable_dt(self, W, adv=(1.0, 1.0)):
        """CFL min 2 |Omega| / sum over the edges of (|v . n| + c) |l|."""
        p = self.nodes[self.cells]
        _, area = self.average(lambda x, y: np.ones((1, x.size)))
        u, v, c = adv[0], adv[1], 0.0
        if len(W) == 4:
            u, v = W[1] / W[0], W[2] / W[0]
            c = np.sqrt(GAMMA * (GAMMA - 1) * (W[3] - 0.5 * W[0] * (u * u + v * v)) / W[0])
        s = 0.0
        for k in range(4):
            b = np.where((k + 1 < self.count)[:, None], p[:, (k + 1) % 4], p[:, 0])
            d = np.where((k < self.count)[:, None], b - p[:, k], 0.0)
            s = s + np.abs(u * d[:, 1] - v * d[:, 0]) + c * np.hypot(d[:, 0], d[:, 1])
        return CFL * float(np.min(2 * area / s))


def _conservative(r, u, v, p):
    r, u, v, p = np.broadcast_arrays(r, u, v, p)
    return np.stack([r, r * u, r * v, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v)])


def _data(data, box, seed):
    """Cell averages (n_v, n_cells) of the initial state, in input order."""
    rng = np.random.default_rng([seed, 1])
    a, b = rng.uniform(0, 2 * math.pi), rng.uniform(0.1, 0.2)
    if data == "scalar":
        return box.average(lambda x, y: (1 + b * np.sin(math.pi * (x + y) + a))[None])[0]
    if data == "wave":
        return box.average(lambda x, y: _conservative(1 + b * np.sin(math.pi * (x + y) + a), 1.0, 1.0, 1.0))[0]
    if data == "vortex":  # isentropic vortex of strength 25 b near the middle of a uniform flow
        cx, cy = box.extent[0] / 2 + 0.5 * math.cos(a), box.extent[1] / 2 + 0.5 * math.sin(a)

        def f(x, y):
            x, y, s = x - cx, y - cy, 25 * b
            e = np.exp(0.5 * (1 - x * x - y * y))
            T = 1 - (GAMMA - 1) * (s * e) ** 2 / (8 * GAMMA * math.pi ** 2)
            r = T ** (1 / (GAMMA - 1))
            return _conservative(r, 1 - s * e * y / (2 * math.pi), 1 + s * e * x / (2 * math.pi), r * T)
        return box.average(f)[0]
    if data == "riemann":  # four constant states that meet in the middle
        q = np.stack([rng.uniform(0.5, 1.5, 4), rng.uniform(-0.5, 0.5, 4), rng.uniform(-0.5, 0.5, 4),
                      rng.uniform(0.4, 1.5, 4)])
        return box.average(lambda x, y: _conservative(*q[:, (x > 0.5) * 2 + (y > 0.5)]))[0]
    if data == "sod":
        x0, r = 0.5 + 0.1 * (b - 0.15), 0.5 + 0.5 * b
        return box.average(lambda x, y: _conservative(np.where(x < x0, 1.0, 0.125 * r), 0.0, 0.0, np.where(x < x0, 1.0, 0.1)))[0]
    n0, n1, c0, _ = box.options["inflow_line"]
    A, B = (_conservative(*map(np.float64, box.options[k])) for k in ("inflow_a", "inflow_b"))
    return box.average(lambda x, y: np.where(n0 * x + n1 * y < c0, A[:, None], B[:, None]))[0]


def _batch(case):
    """(n, kind) of the n x n meshes of a batch: nx <= n <= ny, part of the case and not of the seed."""
    rng = np.random.default_rng(case["nx"] + 1000 * case["ny"] + case["count"])
    n = np.exp(rng.uniform(math.log(case["nx"]), math.log(case["ny"]), case["count"]))
    return [(int(round(v)), ("quad", "tri", "mixed")[k % 3]) for k, v in enumerate(n)]


def _instances(case, seed):
    """(box, W) of every mesh of a case, in input order."""
    if case["op"] != "instances":
        box = _Box(case["kind"], case["nx"], case["ny"], case["box"], seed)
        return [(box, _data(case["data"], box, seed))]
    boxes = [_Box(kind, n, n, case["box"], seed * 1000 + k) for k, (n, kind) in enumerate(_batch(case))]
    return [(box, _data(case["data"], box, seed * 1000 + k)) for k, box in enumerate(boxes)]


def prepare(case, seed):
    parts = _instances(case, seed)
    meshes = [box.handle() for box, _ in parts]
    mesh = meshes[0] if len(meshes) == 1 else Mesh.concat(meshes)
    sol = Solver(mesh, eqn=case["eqn"], precision=case["precision"], eps=EPS, theta=THETA,
                 characteristic=case["characteristic"], linear=case["linear"], **parts[0][0].options)
    U, lo = sol.to_device(np.concatenate([W for _, W in parts], 1))
    state = U if lo is None else torch.stack([U, lo])
    if lo is not None:
        U, lo = state[0], state[1]
    dt = [box.stable_dt(W) for box, W in parts]
    if case["autotune"]:
        sol.autotune(U, lo)
    return {"op": case["op"], "solver": sol, "state": state, "U": U, "U_lo": lo, "dt": dt[0],
            "dts": torch.tensor(dt, dtype=torch.float64, device="cuda"), "R": torch.empty_like(U)}


def run(s):
    sol, U, lo = s["solver"], s["U"], s["U_lo"]
    if s["op"] == "step":
        sol.step(U, lo, s["dt"])
        return s["state"]
    if s["op"] == "instances":
        sol.step_instances(U, lo, s["dts"])
        return s["state"]
    if s["op"] == "residual":
        return sol.residual(U, lo, s["R"])
    dt = sol.max_dt(U, lo, CFL)
    if s["op"] == "monitor":
        return {"dt": dt, "sums": sol.conservation(U, lo)}
    sol.step(U, lo, float(dt[0]))
    return {"dt": dt, "state": s["state"]}


def _sizes(case):
    """(quads, triangles, faces), boundary faces counted once."""
    base = [(case["nx"] * case["ny"], case["kind"])]
    if case["op"] == "instances":
        base = [(n * n, kind) for n, kind in _batch(case)]
    base = [(n, round(SPLIT[kind] * n)) for n, kind in base]
    return sum(n - s for n, s in base), sum(2 * s for _, s in base), sum(2 * n + s for n, s in base)


def work(case):
    """Tables and state in, state (or residual) out; the arithmetic of the reconstruction, the face
    fluxes and the update, three times in a step."""
    quads, tris, faces = _sizes(case)
    nv, real = (4 if case["eqn"] == "euler" else 1), (8 if case["precision"] == "fp64" else 4)
    state = (quads + tris) * nv * 8  # one double, or two floats
    if case["op"] == "monitor":
        return {"bytes": 2 * state + (quads + tris) * 8 + faces * 24, "flops": (quads + tris) * 40}
    tables = 0
    flops = faces * (2 * 130 if nv == 4 else 8) + (quads + tris) * nv * 20
    for n, M, G in ((quads, 12, 8), (tris, 9, 6)):
        tables += n * (real * (M * G + 4 * M + 2 * G + 1) + 4 * M)
        point = 5 if case["linear"] else 23  # P1 at the point; per sign indicator, weight and two sums
        per_face = M * 7 * 4 + M * 10 if case["characteristic"] else 0  # projection and candidates of each face
        flops += n * nv * (G * M * point + M * 10 + G / 2 * per_face)
    flops *= 1 if case["op"] == "residual" else 3
    return {"bytes": tables + faces * (8 + 3 * real) + state * 2, "flops": flops}


# ------------------------------------------------------------------ the scheme in 64 bits
# Numpy restatement of the scheme (arXiv 1712.08317): stencils with mirror images at boundaries,
# minimum-norm least squares, optimised linear weights, split nonlinear weights, HLLC / upwind, SSP-RK3.
# An image of a cell is (cell, mirror edges m1, m2 (-1: none), vertices, momentum flips).
_RULES = {  # slot: (face of the parent, at its start node, replacement); the replacements 0 come first
    4: {5: (0, 1, 0), 6: (0, 0, 0), 7: (2, 1, 0), 8: (2, 0, 0), 9: (3, 0, 5), 10: (1, 1, 6), 11: (1, 0, 7), 12: (3, 1, 8)},
    3: {4: (0, 1, 0), 5: (1, 1, 0), 6: (2, 1, 0), 7: (2, 0, 4), 8: (0, 0, 5), 9: (1, 0, 6)}}
_SUB = {4: [(1, 2), (2, 3), (3, 4), (4, 1), (1, 5), (1, 6), (3, 7), (3, 8), (4, 9), (2, 10), (2, 11), (4, 12)],
        3: [(1, 2), (2, 3), (3, 1), (1, 4), (2, 5), (3, 6), (3, 7), (1, 8), (2, 9)]}


def _pinv(a):
    flat = a.reshape((-1,) + a.shape[-2:])
    parts = np.array_split(flat, max(1, min(64, len(flat) // 2000)))
    with ThreadPoolExecutor(16) as ex:
        got = list(ex.map(lambda x: np.linalg.pinv(x, rcond=1e-12), parts))
    return np.concatenate(got).reshape(a.shape[:-2] + (a.shape[-1], a.shape[-2]))


class _Exact:
    def __init__(self, box, case):
        self.box, self.case = box, case
        nodes, cells, cnt = box.nodes, box.cells, box.count
        N = self.N = len(cells)
        c = np.arange(N)
        first = np.where(np.arange(4)[None] < cnt[:, None], cells, cells.max() + 1).argmin(1)
        k = np.minimum(np.arange(4)[None], cnt[:, None] - 1)
        self.cells = cells = np.take_along_axis(cells, (k + first[:, None]) % cnt[:, None], 1)
        self.V = nodes[cells]
        key = cells
        if box.periodic:  # nodes a period apart are one node
            grid = np.round(nodes / np.array(box.extent) * 1e8).astype(np.int64) % 10 ** 8
            key = np.unique(grid, axis=0, return_inverse=True)[1].reshape(-1)[cells]
        ends = np.stack([key, np.take_along_axis(key, (np.arange(4)[None] + 1) % cnt[:, None], 1)], 2)
        cc, kk = np.nonzero(np.arange(4)[None] < cnt[:, None])
        e = np.sort(ends[cc, kk], 1)
        order = np.lexsort((e[:, 1], e[:, 0]))
        pair = (e[order[1:]] == e[order[:-1]]).all(1)
        i, j = order[:-1][pair], order[1:][pair]
        self.nb, self.nk = np.full((N, 4), -1), np.full((N, 4), -1)
        self.nb[cc[i], kk[i]], self.nk[cc[i], kk[i]], self.nb[cc[j], kk[j]], self.nk[cc[j], kk[j]] = cc[j], kk[j], cc[i], kk[i]
        m = self.nb
        far = self.V[m, (self.nk + 1) % cnt[m]]
        self.shift = np.where((m >= 0)[..., None], self.V - far, 0.0)
        self.next = np.take_along_axis(self.V, ((np.arange(4)[None] + 1) % cnt[:, None])[..., None], 1)
        d = self.next - self.V
        self.len = np.hypot(d[..., 0], d[..., 1])
        self.normal = np.stack([d[..., 1], -d[..., 0]], -1) / np.where(self.len > 0, self.len, 1)[..., None]
        self.wall, self.inflow = np.full((N, 4), -1), np.zeros((N, 4), bool)  # axis of the reversed momentum
        for side in range(4):
            ax, at = side // 2, box.extent[side // 2] * (side % 2)
            on = (m < 0) & (np.abs(self.V[..., ax] - at) < 1e-9) & (np.abs(self.next[..., ax] - at) < 1e-9)
            on &= np.arange(4)[None] < cnt[:, None]
            along = 0.5 * (self.V + self.next)[..., 1 - ax] >= box.wall_from[side]
            if side in box.walls:
                self.wall[on & along] = ax
            if side in box.inflow:
                self.inflow |= on & ~((side in box.walls) & along)
        near, away = (3 + math.sqrt(3)) / 6, (3 - math.sqrt(3)) / 6
        self.xg = np.stack([near * self.V + away * self.next, away * self.V + near * self.next], 2)  # (N, 4, 2, 2)
        self.area = box.average(lambda x, y: np.ones((1, x.size)))[1]
        self.groups = [self._group(c[cnt == n], n) for n in (4, 3) if (cnt == n).any()]

    def _mirror(self, img, c, k):
        """An image mirrored across the line of edge k of cells c."""
        cell, m1, m2, P, fl = img
        a, t = self.V[c, k], np.stack([-self.normal[c, k, 1], self.normal[c, k, 0]], -1)
        r = P - a[:, None]
        P = a[:, None] + 2 * np.einsum("nvx,nx->nv", r, t)[..., None] * t[:, None] - r
        edge = 4 * c + k
        fl = fl ^ (self.wall[c, k][:, None] == np.arange(2)[None])
        return cell, np.where(m1 < 0, edge, m1), np.where(m1 < 0, m2, edge), P, fl

    def _across(self, c, k, P=None):
        """The image across edge k of cells c, whose own vertices are P (shifted copies of V)."""
        x = self.nb[c, k]
        none = np.full(len(c), -1)
        P = self.V[c] if P is None else P
        real = (np.maximum(x, 0), none, none, self.V[x] + (self.shift[c, k] + P[:, 0] - self.V[c, 0])[:, None],
                np.zeros((len(c), 2), bool))
        ghost = self._mirror((c, none, none, P, np.zeros((len(c), 2), bool)), c, k)
        return self._choose(x >= 0, real, ghost)

    @staticmethod
    def _choose(ok, a, b):
        return tuple(np.where(ok.reshape((-1,) + (1,) * (x.ndim - 1)), x, y) for x, y in zip(a, b))

    def _averages(self, P, cnt, c0, s):
        """Averages of (x, y, x^2, y^2, x y), (x - c0) / s, over polygons (n, 4, 2)."""
        P = (P - c0[:, None]) / s[:, None, None]
        total, area = 0.0, 0.0
        for k in (1, 2):
            a, b, c = P[:, 0], P[:, k], P[:, k + 1]
            t = np.abs((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0])) * (k + 1 < cnt)
            for m in ((a + b) / 2, (b + c) / 2, (c + a) / 2):
                total = total + (t / 3)[:, None] * self._monomials(m)
            area = area + t
        return total / area[:, None]

    @staticmethod
    def _monomials(m):
        x, y = m[..., 0], m[..., 1]
        return np.stack([x, y, x * x, y * y, x * y], -1)

    def _group(self, c, n):
        N, M, G, rules, sub = len(c), (12 if n == 4 else 9), 2 * n, _RULES[n], _SUB[n]
        cnt = self.box.count
        none, noflip = np.full(N, -1), np.zeros((N, 2), bool)
        img = [(c, none, none, self.V[c], noflip)] + [self._across(c, np.full(N, k)) for k in range(n)]
        same = lambda a, b: (a[0] == b[0]) & (a[1] == b[1]) & (a[2] == b[2])  # noqa: E731
        E = [np.ones(N, bool)] * (n + 1)
        for j, (k, start, rep) in rules.items():
            p = img[k + 1]
            kp = self.nk[c, k]
            other = np.where(p[1] < 0, (kp + (1 if start else -1)) % cnt[p[0]], 0)
            child = self._across(p[0], other, p[3])
            turned = self._mirror(self._across(c, np.full(N, (k + (-1 if start else 1)) % n)), c, np.full(N, k))
            child = self._choose(p[1] < 0, child, turned)
            ok = ~np.any([same(child, img[i]) for i in range(n + 1)], 0)
            if rep:
                ok &= ~same(child, img[rep])
            E.append(ok)
            img.append(self._choose(ok, child, img[rep]))
        xg = self.xg[c, :n].reshape(N, G, 2)
        s = np.sqrt(self.area[c])
        c0 = self.V[c].mean(1)
        c0 = c0 + s[:, None] * self._averages(self.V[c], cnt[c], c0, s)[:, :2]
        avg = np.stack([self._averages(i[3], cnt[i[0]], c0, s) for i in img], 1)
        A = (avg[:, 1:] - avg[:, :1]) * np.stack(E[1:], 1)[..., None]
        pG = self._monomials((xg - c0[:, None]) / s[:, None, None]) - avg[:, :1]
        eta = np.einsum("ngk,nkm->ngm", pG, _pinv(A))
        first, second = (np.array([t[i] for t in sub]) for i in (0, 1))
        off = s[:, None, None] * (avg[:, :, :2] - avg[:, :1, :2])
        D = _pinv(np.stack([off[:, first], off[:, second]], 2))  # (N, M, 2, 2): gradient of candidate j
        dG = xg - c0[:, None] - s[:, None, None] * avg[:, :1, :2]
        t = np.einsum("nga,nmab->ngmb", dG, D)
        slot = np.tile(np.arange(M + 1), (N, 1))  # the slot whose image stands in slot j
        for j, (k, start, rep) in rules.items():
            slot[:, j] = np.where(E[j], j, slot[:, rep])
        B = np.zeros((N, G, M + 1, M))
        for j in range(M):
            B[np.arange(N), :, slot[:, first[j]], j] += t[:, :, j, 0]
            B[np.arange(N), :, slot[:, second[j]], j] += t[:, :, j, 1]
            B[:, :, 0, j] += 1 - t[:, :, j].sum(-1)
        Bi = _pinv(B)
        solve = lambda e: np.einsum("ngmr,ngr->ngm", Bi, np.concatenate([1 - e.sum(-1, keepdims=True), e], -1))  # noqa: E731
        a = np.abs(solve(eta))
        d = np.ones_like(a)
        if n == 4:
            d[..., 4:] = 1 / np.maximum(1, a[..., 4:])
        else:
            for i, j in ((3, 7), (4, 8), (5, 6)):
                d[..., i] = d[..., j] = 1 / np.maximum(1, np.maximum(a[..., i], a[..., j]))
        gam = solve(np.einsum("ngk,ngkm->ngm", pG, _pinv(d[..., None] * A[:, None])) * d)
        gam = gam / gam.sum(-1, keepdims=True)
        cell, flip = np.stack([i[0] for i in img], 1), np.stack([i[4] for i in img], 1)
        return {"c": c, "n": n, "first": first, "second": second, "D": D, "dG": dG, "gam": gam, "cell": cell, "flip": flip}

    def _points(self, g, dU, pts):
        """Increments (fields, N, len(pts)) over the cell value from the stencil differences dU (fields, N, M + 1)."""
        grad = np.einsum("nmab,vnmb->vnma", g["D"], np.stack([dU[:, :, g["first"]], dU[:, :, g["second"]]], -1))
        P = np.einsum("vnma,nga->vngm", grad, g["dG"][:, pts])
        gam = g["gam"][None][:, :, pts]
        if self.case["linear"]:
            return (gam * P).sum(-1)
        beta = (self.area[g["c"]][None, :, None] * (grad ** 2).sum(-1))[:, :, None]
        plus = 0.5 * (gam + THETA * np.abs(gam))
        out = 0.0
        for w, sign in ((plus, 1), (plus - gam, -1)):
            sig = w.sum(-1, keepdims=True)
            w = w / sig
            q = w * beta
            al = w / (beta * (1 + q + q * q) + EPS) ** 2
            out = out + sign * sig[..., 0] * (al * P).sum(-1) / al.sum(-1)
        return out

    def _frame(self, g, W, k):
        """Right eigenvectors (N, 4, 4) of the normal flux Jacobian at the Roe average across face k."""
        Wn = self._flipped(W[:, g["cell"][:, k + 1]], g["flip"][:, k + 1])
        r, u, v, p = zip(*(self._primitive(w) for w in (W[:, g["c"]], Wn)))
        H = [(w[3] + q) / w[0] for w, q in zip((W[:, g["c"]], Wn), p)]
        s = [np.sqrt(x) for x in r]
        u, v, H = ((s[0] * x[0] + s[1] * x[1]) / (s[0] + s[1]) for x in (u, v, H))
        kin = 0.5 * (u * u + v * v)
        a = np.sqrt((GAMMA - 1) * (H - kin))
        nx, ny = self.normal[g["c"], k].T
        qn, qt, one, zero = u * nx + v * ny, v * nx - u * ny, np.ones_like(u), np.zeros_like(u)
        rows = [[one, one, zero, one], [u - a * nx, u, -ny, u + a * nx], [v - a * ny, v, nx, v + a * ny],
                [H - a * qn, kin, qt, H + a * qn]]
        return np.stack([np.stack(x, -1) for x in rows], -2)

    @staticmethod
    def _flipped(W, flip):
        if len(W) == 1:
            return W
        return np.stack([W[0], np.where(flip[..., 0], -W[1], W[1]), np.where(flip[..., 1], -W[2], W[2]), W[3]])

    @staticmethod
    def _primitive(W):
        u, v = W[1] / W[0], W[2] / W[0]
        return W[0], u, v, (GAMMA - 1) * (W[3] - 0.5 * W[0] * (u * u + v * v))

    def residual(self, W):
        Wg = np.zeros((len(W), self.N, 4, 2))
        for g in self.groups:
            c, n = g["c"], g["n"]
            W0 = W[:, c]
            dW = self._flipped(W[:, g["cell"]], g["flip"]) - W0[:, :, None]
            for k in range(n):
                if self.case["characteristic"]:
                    R = self._frame(g, W, k)
                    inc = self._points(g, np.einsum("nfv,vns->fns", np.linalg.inv(R), dW), [2 * k, 2 * k + 1])
                    inc = np.einsum("nvf,fng->vng", R, inc)
                else:
                    inc = self._points(g, dW, [2 * k, 2 * k + 1])
                Wg[:, c, k] = W0[:, :, None] + inc
        cc, kk = np.nonzero((np.arange(4)[None] < self.box.count[:, None]) & ((self.nb < 0) | (self.nb > np.arange(self.N)[:, None])))
        x, n = self.nb[cc, kk], self.normal[cc, kk]
        L = Wg[:, cc, kk]
        R = np.where((x >= 0)[None, :, None], Wg[:, np.maximum(x, 0), self.nk[cc, kk]][..., ::-1], L)
        nx, ny = n[:, 0][:, None], n[:, 1][:, None]
        if len(W) == 1:
            an = nx + ny  # the default velocity (1, 1)
            F = an * np.where(an >= 0, L, R)
        else:
            mn = 2 * (L[1] * nx + L[2] * ny)
            wall = (self.wall[cc, kk] >= 0)[:, None]
            R[1], R[2] = np.where(wall, L[1] - mn * nx, R[1]), np.where(wall, L[2] - mn * ny, R[2])
            if self.inflow.any():
                n0, n1, c0, _ = self.box.options["inflow_line"]
                A, B = (_conservative(*map(np.float64, self.box.options[q])) for q in ("inflow_a", "inflow_b"))
                xg = self.xg[cc, kk]
                behind = n0 * xg[..., 0] + n1 * xg[..., 1] < c0  # at t = 0
                R = np.where(self.inflow[cc, kk][:, None], np.where(behind, A[:, None, None], B[:, None, None]), R)
            F = self._hllc(L, R, nx, ny)
        F = 0.5 * self.len[cc, kk] * F.sum(-1)
        out = np.zeros_like(W)
        inner = x >= 0
        np.subtract.at(out, (slice(None), cc), F)
        np.add.at(out, (slice(None), x[inner]), F[:, inner])
        return out / self.area

    def _hllc(self, WL, WR, nx, ny):
        sides = []
        for W in (WL, WR):
            W = np.stack([W[0], W[1] * nx + W[2] * ny, W[2] * nx - W[1] * ny, W[3]])
            r, u, v, p = self._primitive(W)
            F = np.stack([W[1], W[1] * u + p, W[2] * u, (W[3] + p) * u])
            sides.append((W, r, u, v, p, F, np.sqrt(GAMMA * p / r), (W[3] + p) / r, np.sqrt(r)))
        (_, rl, ul, vl, pl, FL, al, hl, sl), (_, rr, ur, vr, pr, FR, ar, hr, sr) = sides
        u, v, H = ((sl * x + sr * y) / (sl + sr) for x, y in ((ul, ur), (vl, vr), (hl, hr)))
        a = np.sqrt((GAMMA - 1) * (H - 0.5 * (u * u + v * v)))
        SL, SR = np.minimum(ul - al, u - a), np.maximum(ur + ar, u + a)
        S = (pr - pl + rl * ul * (SL - ul) - rr * ur * (SR - ur)) / (rl * (SL - ul) - rr * (SR - ur))
        star = []
        for (W, r, u, v, p, F, _, _, _), SK in zip(sides, (SL, SR)):
            f = r * (SK - u) / (SK - S)
            star.append(F + SK * (np.stack([f, f * S, f * v, f * (W[3] / r + (S - u) * (S + p / (r * (SK - u))))]) - W))
        F = np.where(SL >= 0, FL, np.where(S >= 0, star[0], np.where(SR > 0, star[1], FR)))
        return np.stack([F[0], F[1] * nx - F[2] * ny, F[1] * ny + F[2] * nx, F[3]])

    def step(self, W, dt):
        W1 = W + dt * self.residual(W)
        W2 = 0.75 * W + 0.25 * (W1 + dt * self.residual(W1))
        return W / 3 + 2 / 3 * (W2 + dt * self.residual(W2))


def exact(case, seed):
    quads, tris, _ = _sizes(case)
    if quads + tris > EXACT_CELLS and case["op"] != "monitor":
        return None
    parts = _instances(case, seed)
    if case["op"] == "monitor":
        sums = [(W * box.average(lambda x, y: np.ones((1, x.size)))[1]).sum(1) for box, W in parts]
        return {"dt": np.array([box.stable_dt(W) for box, W in parts]), "sums": np.stack(sums)}
    dt = [box.stable_dt(W) for box, W in parts]
    schemes = [_Exact(box, case) for box, _ in parts]
    out = [s.residual(W) if case["op"] == "residual" else s.step(W, h) for s, (_, W), h in zip(schemes, parts, dt)]
    meshes = [box.handle() for box, _ in parts]  # only for the order in which the library keeps the cells
    perm = (meshes[0] if len(meshes) == 1 else Mesh.concat(meshes)).perm
    W = np.concatenate(out, 1)[:, perm].T
    if case["precision"] == "fp32c" and case["op"] != "residual":
        hi = W.astype(np.float32).astype(np.float64)
        W = np.stack([hi, W - hi])
    return {"dt": np.array(dt), "state": W} if case["op"] == "adaptive" else W
