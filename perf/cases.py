"""The workloads this solver is timed on: whole calls a user makes through
``solver.Solver``, ``solver.Batch`` and ``serve.Server``.

A case is a dict of plain values.  ``kind`` says what the call is:

  solve     one board: zero the state, advance ``steps`` leapfrog steps, read
            every probe's spectrum and trace, and the E_z plane through the
            dielectric
  snapshot  one board: advance in ``shots`` equal parts and read the E_z plane
            through the dielectric after each (the data of Figs. 3-4)
  fields    one board: advance, read the probes and all six field volumes
  sweep     one board, new materials: replace the material volume (the host
            rebuilds the coefficient ids), advance, read the spectra
  batch     several uneven boards stepped together, spectra and traces of each
  served    a burst of requests through the solve server: boards are created,
            stepped in one mix, retired; the spectra of each

Boards are stacks of planes (``geometry`` "stack"), the paper's Table 1 board
with its resistive voltage source ("table1"), random-material grids ("random")
or closed cavities with PMC side walls ("cavity").  ``total`` is the run length
N of the spectrum; a pass advances the first ``steps`` of it, as a user's
program does that works a long run in windows.  Probes lie near the sources,
where a window's wave has arrived.
"""
import math

import numpy as np
import torch

from paper_1008_2602_gb300 import serve, solver
from paper_1008_2602_gb300 import workloads as W

MM, PS = 1e-3, 1e-12
C0 = 299792458.0
MU0 = 4.0e-7 * math.pi
EPS0 = 1.0 / (MU0 * C0 * C0)
ETA0 = MU0 * C0


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _stack(name, kind, bx, by, pairs, diel, core, air_xy, air_z, upml_xy, upml_z, dxy_mm, dz_mm, steps, total, probes,
           sources=1, fmax_ghz=10.0, precision="fp32", sheet=1, shots=0):
    return dict(name=name, kind=kind, geometry="stack", bx=bx, by=by, pairs=pairs, diel=diel, core=core,
                air_xy=air_xy, air_z=air_z, upml_xy=upml_xy, upml_z=upml_z, dxy_mm=dxy_mm, dz_mm=dz_mm, steps=steps,
                total=total, probes=probes, sources=sources, fmax_ghz=fmax_ghz, precision=precision, sheet=sheet,
                shots=shots)


def _multilayer(name, kind, scale, steps, precision="fp32"):
    return _stack(name, kind, 800 // scale, 600 // scale, 4, 6, 8, 28, 10, 12, 12, 0.25, 0.1, steps, 50000, 64,
                  sources=4, precision=precision)


def listed():
    return [
        # the animation frames of the paper's 100 x 60 x 0.8 mm board: a few steps between two reads of a plane
        _stack("snapshot_72x52x20", "snapshot", 50, 30, 1, 2, 0, 3, 3, 8, 6, 2.0, 0.4, 40, 40, 1, fmax_ghz=0.0, sheet=0,
               shots=4),
        # the resonance run of Table 1 (voltage source), first 1500 of its 30000 steps, every bin up to Nyquist
        dict(name="table1_38x33x20", kind="solve", geometry="table1", air=3, upml=6, steps=1500, total=1500,
             precision="fp32"),
        # a small plane pair solved from start to spectrum: 2000 steps, bins up to Nyquist
        _stack("small_56x48x30", "solve", 32, 24, 1, 4, 0, 4, 4, 8, 8, 1.0, 0.25, 2000, 2000, 4, fmax_ghz=0.0),
        # mixed materials cell by cell (16-bit coefficient ids), odd extents, kappa grading, all fields read back
        dict(name="random_97x61x43", kind="fields", geometry="random", nx=97, ny=61, nz=43, upml=5, n_mat=3,
             kappa=5.0, steps=150, total=150, precision="fp32"),
        # the cavity model of a plane pair: PMC side walls, PEC planes, no UPML
        dict(name="cavity_181x131x6", kind="solve", geometry="cavity", nx=181, ny=131, nz=6, eps=4.0, dxy_mm=0.5,
             dz_mm=0.2, steps=600, total=600, precision="fp32"),
        # a 100 x 80 mm plane pair, 16 probes, a window of its 20000 steps
        _stack("realistic_232x192x39", "solve", 200, 160, 1, 5, 0, 6, 6, 10, 10, 0.5, 0.2, 400, 20000, 16, sources=3),
        # the multilayer board (four plane pairs, 64 probes) at quarter, half and full extent
        _multilayer("multilayer_280x230x100", "solve", 4, 200),
        _multilayer("multilayer_480x380x100_fp16", "solve", 2, 100, precision="fp16"),
        _multilayer("multilayer_880x680x100", "solve", 1, 100),
        # a material study: each window of the half-extent board starts from a new material volume
        _multilayer("sweep_480x380x100", "sweep", 2, 60),
        # uneven boards solved together
        dict(name="batch_24", kind="batch", set=4, boards=24, size_lo=20.0, size_hi=120.0, steps=100, total=5000,
             precision="fp32"),
        # a burst of requests of mixed size and length through the server
        dict(name="served_10", kind="served", set=5, requests=10, median=4e5, most=4e6, steps_lo=200, steps_hi=900, chunk=200,
             precision="fp32"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["snapshot", "fields", "sweep", "batch", "served", "table1", "cavity", "cavity"])
    if kind == "batch":
        n = _logint(rng, 3, 24)
        lo = rng.uniform(10.0, 60.0)
        return dict(kind="batch", set=rng.randrange(1 << 20), boards=n, size_lo=lo, size_hi=lo + rng.uniform(10.0, 60.0), steps=_logint(rng, 40, 100),
                    total=5000, precision=rng.choice(["fp32", "fp32", "fp16"]))
    if kind == "served":
        lo = _logint(rng, 50, 300)
        return dict(kind="served", set=rng.randrange(1 << 20), requests=_logint(rng, 2, 12), median=float(_logint(rng, 150_000, 500_000)), most=4e6,
                    steps_lo=lo, steps_hi=lo + _logint(rng, 50, 600), chunk=rng.choice([100, 200, 250]),
                    precision=rng.choice(["fp32", "fp32", "fp16"]))
    if kind == "table1":
        n = _logint(rng, 200, 2000)
        return dict(kind="solve", geometry="table1", air=rng.randint(2, 9), upml=rng.randint(4, 10), steps=n, total=n,
                    precision="fp32")
    if kind == "cavity":
        nx, ny, nz = _logint(rng, 20, 600), _logint(rng, 20, 500), rng.randint(2, 24)
        steps = int(max(20, min(1000, 4e8 / (nx * ny * nz))))
        return dict(kind="solve", geometry="cavity", nx=nx, ny=ny, nz=nz, eps=rng.uniform(2.0, 5.0),
                    dxy_mm=rng.choice([0.5, 1.0]), dz_mm=rng.choice([0.2, 0.25]), steps=steps, total=steps,
                    precision="fp32")
    if kind == "fields":
        u = rng.randint(2, 6)
        nx, ny, nz = (_logint(rng, 2 * u + 12, 140) for _ in range(3))
        steps = rng.randint(20, 200)
        return dict(kind="fields", geometry="random", nx=nx, ny=ny, nz=nz, upml=u, n_mat=3,
                    kappa=rng.choice([1.0, 1.0, 5.0]), steps=steps, total=steps, precision="fp32")
    # a stack of planes: sides, stack, cell sizes and run length over the whole range
    bx = _logint(rng, 20, 800)
    by = max(16, min(600, int(bx * rng.uniform(0.5, 1.0))))
    pairs, diel, core = rng.randint(1, 4), rng.randint(2, 8), rng.randint(4, 8)
    air_xy, air_z = _logint(rng, 3, 28), rng.randint(3, 10)
    ux, uz = rng.randint(6, 12), rng.randint(6, 12)
    nz = 2 * (uz + air_z) + pairs * (diel + 2) + (pairs - 1) * core
    cells = (bx + 2 * (air_xy + ux)) * (by + 2 * (air_xy + ux)) * nz
    most = 2000 if kind == "solve" else 200
    steps = int(max(24, min(most, rng.uniform(0.3, 1.0) * 5e9 / cells)))
    shots = rng.randint(2, 8) if kind == "snapshot" else 0
    if shots:
        steps = shots * max(5, min(50, steps // shots))
    whole = cells < 500_000 and kind == "solve"
    precision = rng.choice(["fp32", "fp16"]) if cells > 1_000_000 and kind == "solve" else "fp32"
    return _stack("", kind, bx, by, pairs, diel, core, air_xy, air_z, ux, uz, rng.choice([0.25, 0.5, 1.0]),
                  rng.choice([0.1, 0.2, 0.25]), steps, steps if whole or shots else 20000, _logint(rng, 1, 64),
                  sources=rng.randint(1, 4), fmax_ghz=10.0, precision=precision, shots=shots)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ports(p, rng, n_src, n_prb, steps):
    """Pulsed E_z sources at seeded edges between the planes, and E_z probes within the reach of ``steps`` steps."""
    i0, i1, j0, j1 = p.board
    h = (p.dx, p.dy, p.dz)
    cdt = C0 * p.dt if p.dt > 0 else p.courant / math.sqrt(sum(1.0 / v ** 2 for v in h))
    reach = [max(1, int(0.4 * steps * cdt / (2.15 * v))) for v in h[:2]]
    src, prb = [], []
    for _ in range(n_src):
        k0, k1 = p.dielectric_k[int(rng.integers(len(p.dielectric_k)))]
        src.append((int(rng.integers(i0 + 1, i1)), int(rng.integers(j0 + 1, j1)), int(rng.integers(k0, k1)), 2))
    for t in range(n_prb):
        i, j, k, _ = src[t % n_src]
        k0, k1 = next(q for q in p.dielectric_k if q[0] <= k < q[1])
        lo, hi = [max(i0 + 1, i - reach[0]), max(j0 + 1, j - reach[1])], [min(i1, i + reach[0] + 1), min(j1, j + reach[1] + 1)]
        prb.append((int(rng.integers(lo[0], hi[0])), int(rng.integers(lo[1], hi[1])), int(rng.integers(k0, k1)), 2))
    return W.add_ports(p, src, prb, J0=1e6 * float(rng.uniform(0.5, 2.0)))


def _problem(case, seed):
    rng = np.random.default_rng(seed)
    g = case["geometry"]
    if g == "table1":
        p = W.table1_board(n_steps=case["total"], air=(case["air"],) * 3, upml=(case["upml"],) * 3)
        prm = np.array(p.vsource_params)
        prm[:, 0] = rng.uniform(1.0, 10.0)
        return p.replace(eps_r=np.array([1.0, rng.uniform(3.5, 4.6)]), vsource_params=prm)
    if g == "random":
        p = W.random_problem(int(rng.integers(1 << 30)), case["nx"], case["ny"], case["nz"], upml=case["upml"],
                             n_mat=case["n_mat"], n_steps=case["total"])
        return p.replace(upml_kappa_max=case["kappa"])
    if g == "cavity":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        d = (case["dxy_mm"] * MM, case["dxy_mm"] * MM, case["dz_mm"] * MM)
        walls = (W.WALL_PMC,) * 4 + (W.WALL_PEC,) * 2
        p = W.box(nx, ny, nz, d=d, eps_r=case["eps"] * float(rng.uniform(0.9, 1.1)), walls=walls)
        at = [(int(rng.integers(nx)), int(rng.integers(ny)), int(rng.integers(nz)), 2) for _ in range(5)]
        return W.add_ports(p, at[:1], at[1:], J0=1e6 * float(rng.uniform(0.5, 2.0)), n_steps=case["total"])
    layers = []
    for q in range(case["pairs"]):
        layers += [("pec", 0, 0), ("diel", case["diel"], float(rng.uniform(3.5, 4.6))), ("pec", 0, 0)]
        if q < case["pairs"] - 1:
            layers.append(("diel", case["core"], float(rng.uniform(3.5, 4.6))))
    p, _ = W.pcb_stack(board_cells=(case["bx"], case["by"]), layers=layers,
                       air=(case["air_xy"], case["air_xy"], case["air_z"]),
                       upml=(case["upml_xy"], case["upml_xy"], case["upml_z"]),
                       d=(case["dxy_mm"] * MM, case["dxy_mm"] * MM, case["dz_mm"] * MM), sheet_thickness=case["sheet"])
    f = case["fmax_ghz"] * 1e9
    return _ports(p, rng, case["sources"], case["probes"], case["steps"]).replace(n_steps=case["total"], f_max=f if f > 0 else None)


def _swept(case, p, seed):
    """Another material volume of the same board: the dielectric layers trade places."""
    rng = np.random.default_rng(seed + 7919)
    perm = np.arange(len(p.eps_r), dtype=np.uint8)
    perm[1:] = rng.permutation(perm[1:])
    return perm[p.mat]


def _reseeded(p, rng, steps):
    """The same board with other permittivities and ports."""
    eps = np.concatenate([[1.0], rng.uniform(3.5, 4.6, len(p.eps_r) - 1)])
    return _ports(p.replace(eps_r=eps), rng, len(p.sources), len(p.probes), steps)


def _batch_problems(case, seed):
    rng = np.random.default_rng(seed)
    ps = W.batch_boards(seed=case["set"], n_boards=case["boards"], n_steps=case["total"],
                        size_mm=(case["size_lo"], case["size_hi"]))
    return [_reseeded(p, rng, case["steps"]) for p in ps]


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    r = W.request_stream(seed=case["set"], n_requests=case["requests"], median_cells=case["median"],
                         max_cells=case["most"], steps=(case["steps_lo"], case["steps_hi"]))
    for q in r:
        q.arrival = 0.0   # one burst: the server's schedule then depends on the requests alone
        q.problem = _reseeded(q.problem, rng, q.problem.n_steps)
    return r


def _plane(p):
    return p.dielectric_k[0][0] if p.dielectric_k else p.nz // 2


def prepare(case, seed):
    kind = case["kind"]
    if kind == "served":
        return dict(case=case, requests=_requests(case, seed))
    if kind == "batch":
        sols = [solver.Solver(p, precision=case["precision"]) for p in _batch_problems(case, seed)]
        return dict(case=case, batch=solver.Batch(), solvers=sols)
    p = _problem(case, seed)
    state = dict(case=case, solver=solver.Solver(p, precision=case["precision"]))
    if kind == "sweep":
        state["mat"] = _swept(case, p, seed)
    state["plane"] = _plane(p)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "served":
        backend = serve.CudaBackend(precision=case["precision"])
        try:
            res = serve.Server(backend, hbm_budget=64 << 30, max_boards=64, chunk=case["chunk"]).run(state["requests"])
        finally:
            backend.close()
        return [r.spectra for r in sorted(res, key=lambda r: r.rid)]
    if kind == "batch":
        b, sols = state["batch"], state["solvers"]
        for s in sols:
            s.reset()
            b.add(s, case["steps"])
        b.step(case["steps"])
        b.sync()
        out = [(s.spectra(), s.traces()) for s in sols]
        for s in sols:
            b.remove(s)
        return out
    s = state["solver"]
    if kind == "sweep":
        s.set_materials(state["mat"])
        s.step(case["steps"])
        return s.spectra()
    s.reset()
    if kind == "snapshot":
        out = []
        for _ in range(case["shots"]):
            s.step(case["steps"] // case["shots"])
            out.append(s.plane(2, state["plane"]))
        return out
    s.step(case["steps"])
    out = [s.spectra(), s.traces()]
    return out + ([s.field(c) for c in range(6)] if kind == "fields" else [s.plane(2, state["plane"])])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _cells(case):
    if case["geometry"] == "table1":
        a = 2 * (case["air"] + case["upml"])
        return (20 + a) * (15 + a) * (2 + a)
    if case["geometry"] != "stack":
        return case["nx"] * case["ny"] * case["nz"]
    xy = 2 * (case["air_xy"] + case["upml_xy"])
    nz = (2 * (case["air_z"] + case["upml_z"]) + case["pairs"] * (case["diel"] + 2 * case["sheet"])
          + (case["pairs"] - 1) * case["core"])
    return (case["bx"] + xy) * (case["by"] + xy) * nz


def work(case):
    """Per cell and step: six components read and six written in the storage
    type and one coefficient id; two differences, two products and two sums
    per component (seven operations)."""
    es = 2 if case["precision"] == "fp16" else 4
    if case["kind"] == "served":
        updates = float(sum(r.problem.cells * r.problem.n_steps for r in _requests(case, 1)))
    elif case["kind"] == "batch":
        updates = float(sum(p.cells for p in _batch_problems(case, 1))) * case["steps"]
    else:
        updates = float(_cells(case)) * case["steps"]
    return {"bytes": updates * (12 * es + 1), "flops": updates * 42.0}


# ---------------------------------------------------------------------------
# the same numbers in 64 bits
# ---------------------------------------------------------------------------

def _factors(n, d, dlo, dhi, p, dt, half, dev):
    """D/B recurrence factors of one axis at its integer or half positions."""
    x = np.arange(n if half else n + 1) + (0.5 if half else 0.0)
    sig, kap = np.zeros_like(x), np.ones_like(x)
    for depth, rho in ((dlo, (dlo - x) / max(dlo, 1)), (dhi, (x - (n - dhi)) / max(dhi, 1))):
        if depth:
            r = np.where(rho > 0, np.abs(rho) ** p.upml_m, 0.0)
            sig += -(p.upml_m + 1.0) * math.log(p.upml_R0) / (2.0 * ETA0 * depth * d) * r
            kap += (p.upml_kappa_max - 1.0) * r
    q = sig * dt / (2.0 * EPS0)
    return [torch.tensor(v, device=dev) for v in ((kap - q) / (kap + q), 1.0 / (kap + q), kap + q, kap - q)]


class _Yee:
    """Yee leapfrog with D and B everywhere, 64 bits, plain torch."""

    def __init__(self, p, mat=None):
        self.p = p
        dev = self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        n = (p.nx, p.ny, p.nz)
        d = (p.dx, p.dy, p.dz)
        self.dt = p.dt if p.dt > 0 else p.courant / (C0 * math.sqrt(sum(1.0 / v ** 2 for v in d)))
        self.S = [C0 * self.dt / v for v in d]
        # factors by axis and position, shaped to broadcast over [z, y, x]
        shape = ((1, 1, -1), (1, -1, 1), (-1, 1, 1))
        self.cw = [[[f.view(shape[w]) for f in _factors(n[w], d[w], p.upml_depth[2 * w], p.upml_depth[2 * w + 1], p,
                                                        self.dt, half, dev)] for half in (False, True)] for w in range(3)]
        full = lambda half: tuple(n[w] + (0 if half[w] else 1) for w in (2, 1, 0))  # noqa: E731
        self.E, self.H, self.ce = [], [], []
        eps = torch.tensor(np.asarray(p.eps_r, np.float64), device=dev)[
            torch.from_numpy(np.ascontiguousarray(p.mat if mat is None else mat)).to(dev).long()]
        for w in range(3):
            self.E.append(torch.zeros(full([a == w for a in range(3)]), dtype=torch.float64, device=dev))
            self.H.append(torch.zeros(full([a != w for a in range(3)]), dtype=torch.float64, device=dev))
            self.ce.append(self._edge_coefficients(eps, w))
        del eps
        self.D = [torch.zeros_like(v) for v in self.E]
        self.B = [torch.zeros_like(v) for v in self.H]
        self.step_no = 0
        self.src = []
        for (i, j, k, w), (J0, t0, tau) in zip(np.asarray(p.sources).reshape(-1, 4),
                                               np.asarray(p.source_params).reshape(-1, 3)):
            self.src.append((int(w), (int(k), int(j), int(i)), float(J0), float(t0), float(tau), None))
        for (i, j, k, w), (V0, t0, tau, Rs) in zip(np.asarray(p.vsources).reshape(-1, 4),
                                                   np.asarray(p.vsource_params).reshape(-1, 4)):
            area = p.dx * p.dy * p.dz / d[int(w)]
            ce = float(self.ce[int(w)][int(k), int(j), int(i)])
            beta = self.dt * d[int(w)] * ce / (2.0 * EPS0 * float(Rs) * area)
            gam = self.dt * ce / (EPS0 * float(Rs) * area)
            self.src.append((int(w), (int(k), int(j), int(i)), float(V0), float(t0), float(tau), (beta, gam)))
        self.prb = []
        for w in range(3):
            at = [(t, (q[2] * self.E[w].shape[1] + q[1]) * self.E[w].shape[2] + q[0])
                  for t, q in enumerate(np.asarray(p.probes).reshape(-1, 4).tolist()) if q[3] == w]
            if at:
                self.prb.append((w, torch.tensor([a for a, _ in at], device=dev), torch.tensor([b for _, b in at], device=dev)))

    def _edge_coefficients(self, eps, w):
        """1 / eps_r of the E_w edges: mean over the cells that share one, 0 on conductors."""
        p = self.p
        s, c = eps, torch.ones_like(eps)
        for a in range(3):
            if a == w:
                continue
            pad = [0] * 6
            pad[2 * a] = pad[2 * a + 1] = 1
            s, c = torch.nn.functional.pad(s, pad), torch.nn.functional.pad(c, pad)
            m = s.shape[2 - a]
            s = s.narrow(2 - a, 0, m - 1) + s.narrow(2 - a, 1, m - 1)
            c = c.narrow(2 - a, 0, m - 1) + c.narrow(2 - a, 1, m - 1)
        ce = c / s
        for i0, i1, j0, j1, k0, k1 in np.asarray(p.pec_boxes).reshape(-1, 6).tolist():
            hi = [i1 + 1, j1 + 1, k1 + 1]
            hi[w] -= 1
            ce[k0:hi[2], j0:hi[1], i0:hi[0]] = 0.0
        for a in range(3):
            if a != w:
                for side in (0, 1):
                    if p.walls[2 * a + side] == W.WALL_PEC:
                        ce.select(2 - a, -1 if side else 0).zero_()
        return ce

    def _add_diff(self, out, h, axis, s):
        """out += s dH/d(axis) on nodes; PMC walls mirror H oddly, PEC walls hold E at zero."""
        a = 2 - axis
        m = out.shape[a]
        inner = out.narrow(a, 1, m - 2)
        inner.add_(h.narrow(a, 1, m - 2), alpha=s).sub_(h.narrow(a, 0, m - 2), alpha=s)
        if self.p.walls[2 * axis] == W.WALL_PMC:
            out.select(a, 0).add_(h.select(a, 0), alpha=2.0 * s)
        if self.p.walls[2 * axis + 1] == W.WALL_PMC:
            out.select(a, m - 1).sub_(h.select(a, m - 2), alpha=2.0 * s)

    def step(self):
        for w in range(3):
            b, c = (w + 1) % 3, (w + 2) % 3
            t = torch.diff(self.E[c], dim=2 - b).mul_(-self.S[b])
            t.add_(torch.diff(self.E[b], dim=2 - c), alpha=self.S[c])
            self._update(self.H[w], self.B, w, t, self.cw[b][1], self.cw[c][1], self.cw[w][0], None)
        for w in range(3):
            b, c = (w + 1) % 3, (w + 2) % 3
            old = [float(self.E[w][at]) if v else 0.0 for (u, at, _, _, _, v) in self.src if u == w]
            t = torch.zeros_like(self.E[w])
            self._add_diff(t, self.H[c], b, self.S[b])
            self._add_diff(t, self.H[b], c, -self.S[c])
            self._update(self.E[w], self.D, w, t, self.cw[b][0], self.cw[c][0], self.cw[w][1], self.ce[w])
            time = (self.step_no + 0.5) * self.dt
            for (u, at, a0, t0, tau, v), e0 in zip([s for s in self.src if s[0] == w], old):
                f = (time - t0) / tau
                f = a0 * f * math.exp(-f * f)
                if v is None:
                    self.E[w][at] -= self.ce[w][at] * (self.dt / EPS0 * f)
                else:
                    self.E[w][at] = (self.E[w][at] - v[0] * e0 - v[1] * f) / (1.0 + v[0])
        self.step_no += 1

    @staticmethod
    def _update(f, aux, w, curl, a, b, c, ce):
        new = curl.mul_(a[1]).addcmul_(aux[w], a[0])
        t = new * c[2]
        t.addcmul_(aux[w], c[3], value=-1.0)
        t.mul_(b[1])
        if ce is not None:
            t.mul_(ce)
        f.mul_(b[0]).add_(t)
        aux[w] = new

    def run(self, n, traces=None):
        for _ in range(n):
            self.step()
            if traces is not None:
                for w, which, at in self.prb:
                    traces[which, self.step_no - 1] = self.E[w].reshape(-1)[at]

    def spectra(self, traces):
        N = self.p.n_steps
        Q = N // 2 + 1
        if self.p.f_max:
            Q = min(Q, int(math.floor(self.p.f_max * N * self.dt + 1e-9)) + 1)
        n = torch.arange(traces.shape[1], device=self.dev, dtype=torch.int64)
        out = torch.zeros((traces.shape[0], Q), dtype=torch.complex128, device=self.dev)
        for q in range(0, Q, 256):
            qs = torch.arange(q, min(q + 256, Q), device=self.dev, dtype=torch.int64)
            ph = (-2.0 * math.pi / N) * ((qs[None, :] * n[:, None]) % N).double()
            out[:, q:q + 256] = self.dt * torch.complex(traces @ torch.cos(ph), traces @ torch.sin(ph))
        return out

    def field(self, c):
        f, scale = (self.E[c], 1.0) if c < 3 else (self.H[c - 3], 1.0 / ETA0)
        p = self.p
        out = torch.zeros((p.nz + 1, p.ny + 1, p.nx + 1), dtype=torch.float64, device=self.dev)
        out[:f.shape[0], :f.shape[1], :f.shape[2]] = f * scale
        return out


def _solved(p, steps, mat=None):
    y = _Yee(p, mat)
    tr = torch.zeros((len(np.asarray(p.probes).reshape(-1, 4)), steps), dtype=torch.float64, device=y.dev)
    y.run(steps, tr)
    return y, y.spectra(tr), tr


def exact(case, seed):
    kind = case["kind"]
    if kind == "served":
        return [_solved(r.problem, r.problem.n_steps)[1] for r in sorted(_requests(case, seed), key=lambda r: r.rid)]
    if kind == "batch":
        return [_solved(p, case["steps"])[1:] for p in _batch_problems(case, seed)]
    p = _problem(case, seed)
    if kind == "sweep":
        return _solved(p, case["steps"], _swept(case, p, seed))[1]
    if kind == "snapshot":
        y, out = _Yee(p), []
        for _ in range(case["shots"]):
            y.run(case["steps"] // case["shots"])
            out.append(y.field(2)[_plane(p)].clone())
        return out
    y, sp, tr = _solved(p, case["steps"])
    return [sp, tr] + ([y.field(c) for c in range(6)] if kind == "fields" else [y.field(2)[_plane(p)].clone()])
