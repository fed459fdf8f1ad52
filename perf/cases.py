"""Performance cases of the dual-porosity simulator: what a user of the library
has it do, through the Python binding (``paper_1808_04338_gb300.dpsim``), from
a 600-cell parity problem to the 200x200x50 field (8M unknowns).

Kinds of case ("kind"):
  advance   one backward-Euler timestep from a given state (sim_advance)
  run       a simulation period with its own timestep control (sim_run)
  assembly  Jacobian and residual at an iterate (sim_assemble), handed out
            whole, as a program with its own solver takes them
  solve     one Newton linear solve and update (sim_assemble, sim_solve_step)
  ensemble  many realisations of uneven size advanced in lockstep (Batch)
  serve     a server started, realisations registered, a timestep of each
            requested and its state fetched (Server): what a cold request costs

Cases with an FP32 or BF16 preconditioner use the report options with the
Newton tolerance at 1e-9 instead of 1e-6, so that the state a pass ends on is
that of the equations and not of the path the iteration took to its tolerance.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import dp_inputs as di
from paper_1808_04338_gb300 import dpsim

DAY = di.DAY
# Newton iterations and FGMRES iterations a solve that work() counts (rounded
# from what these workloads take, whatever the code does)
NEWTON, KRYLOV = 5, 8


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the parity configuration, the smallest call: latency and launches
        dict(name="tiny_step", kind="advance", base="tiny", nx=10, ny=10, nz=3, mode="parity",
             precision=0, schur=0, days=1.0, flooded=False, gravity=False, capillary=False),
        # the paper's Example 2 over its first 15 days (steps of 1, 2, 4, 8 days): gravity,
        # oil-rate producers reaching their pressure limit, many small solves
        dict(name="example2_run", kind="run", base="example2", nx=10, ny=10, nz=3, mode="parity",
             precision=0, schur=0, days=15.0),
        # the layered 200k-cell configuration, plain FP64, with a waterflood under way
        dict(name="layered_step", kind="advance", base="layered", nx=100, ny=100, nz=10,
             mode="parity", precision=0, schur=0, days=5.0, flooded=True, gravity=False,
             capillary=False),
        # a ragged mid-size model with capillary curves, BF16 coarse levels
        dict(name="ragged_step_bf16", kind="advance", base="layered", nx=93, ny=71, nz=17,
             mode="report", precision=2, schur=0, days=5.0, flooded=True, gravity=False,
             capillary=True),
        # the headline field: first 5-day step, FP32 preconditioner
        dict(name="field_step", kind="advance", base="field", nx=200, ny=200, nz=50,
             mode="report", precision=1, schur=0, days=5.0, flooded=False, gravity=False,
             capillary=False),
        # the same with the matrix cells eliminated exactly
        dict(name="field_step_eliminated", kind="advance", base="field", nx=200, ny=200, nz=50,
             mode="report", precision=1, schur=1, days=5.0, flooded=False, gravity=False,
             capillary=False),
        # Jacobian and residual of the field at a Newton iterate
        dict(name="field_assembly", kind="assembly", base="field", nx=200, ny=200, nz=50,
             days=5.0, gravity=False, capillary=False),
        # the same call on a small ragged model with every term of the equations
        dict(name="capillary_assembly", kind="assembly", base="example1", nx=61, ny=43, nz=27,
             days=1.0, gravity=True, capillary=True),
        # one linear solve of a mid-size field in plain FP64 to a tight tolerance
        dict(name="solve_fp64", kind="solve", base="field", nx=121, ny=113, nz=37, precision=0,
             schur=0, eta=1e-8, days=5.0),
        # sixteen realisations of the ensemble (4k to 240k cells) in lockstep
        dict(name="ensemble_step", kind="ensemble", members=16, first=0, stride=4, precision=1,
             days=5.0),
        # eight realisations served from cold by four workers
        dict(name="serve_cold", kind="serve", members=8, smallest=23, ratio=1.23, nz=10,
             workers=4, precision=1, days=5.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    """nx, ny, nz of about log-uniform size between lo and hi locations, nx and ny at least
    16 where the size allows, often odd, aspect ratios as reservoir grids have them."""
    n = _log(rng, lo, hi)
    nz = max(1, round(n ** (1.0 / 3.0) * _log(rng, 0.2, 0.7)))
    side = math.sqrt(n / nz)
    a = _log(rng, 0.6, 1.6)
    return max(9, round(side * a)), max(9, round(side / a)), nz


def draw(rng):
    kind = rng.choice(["advance", "advance", "advance", "advance", "assembly", "assembly",
                       "solve", "run", "ensemble", "serve"])
    if kind == "advance":
        mode = rng.choice(["parity", "report", "report"])
        nx, ny, nz = _grid(rng, 300, 1.0e5) if mode == "parity" else _grid(rng, 2000, 1.8e6)
        # gravity on thin grids, with a flood under way (in thick ones the hydrostatic upstream
        # directions flip from one Newton iterate to the next and the timestep is cut)
        gravity = nz <= 8 and rng.random() < 0.6
        return dict(kind=kind, base=rng.choice(["layered", "field"])
                    if min(nx, ny) >= 16 and not gravity else "layered", nx=nx, ny=ny, nz=nz, mode=mode,
                    precision=0 if mode == "parity" else rng.choice([1, 1, 2]),
                    schur=rng.choice([0, 0, 1]), days=rng.choice([1.0, 2.0, 5.0]),
                    flooded=rng.random() < 0.5 or gravity, gravity=gravity,
                    capillary=nx * ny * nz < 250000 and rng.random() < 0.3)
    if kind == "assembly":
        nx, ny, nz = _grid(rng, 300, 2.0e6)
        return dict(kind=kind, base=rng.choice(["layered", "example1", "example2"]), nx=nx,
                    ny=ny, nz=nz, days=rng.choice([1.0, 5.0]), gravity=rng.random() < 0.5,
                    capillary=rng.random() < 0.4)
    if kind == "solve":
        nx, ny, nz = _grid(rng, 1000, 5.0e5)
        return dict(kind=kind, base="layered", nx=nx, ny=ny, nz=nz,
                    precision=rng.choice([0, 0, 1]), schur=rng.choice([0, 1]),
                    eta=1e-8, days=rng.choice([1.0, 5.0]))
    if kind == "run":
        nx, ny, nz = _grid(rng, 100, 4000)
        return dict(kind=kind, base=rng.choice(["example1", "example2"]), nx=nx, ny=ny, nz=nz,
                    mode="parity", precision=0, schur=0, days=rng.choice([3.0, 7.0, 15.0]))
    if kind == "ensemble":
        stride = rng.choice([3, 5, 7])
        return dict(kind=kind, members=rng.randint(3, 64 // stride - 1),
                    first=rng.randint(0, stride), stride=stride, precision=rng.choice([1, 2]),
                    days=rng.choice([2.0, 5.0]))
    return dict(kind=kind, members=rng.randint(3, 7), smallest=rng.randint(15, 31),
                ratio=round(rng.uniform(1.05, 1.22), 3), nz=rng.randint(5, 10),
                workers=rng.choice([2, 4]), precision=rng.choice([0, 1]),
                days=rng.choice([1.0, 5.0]))


# ----------------------------------------------------------------- inputs

def _problem(case, seed):
    """The realisation of a case: the repository's synthetic workloads at the
    case's grid, drawn from the seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    base = case["base"]
    if base == "tiny":
        prob = di.tiny(seed)
    elif base == "layered":
        prob = di.layered(nx, ny, nz, seed)
    elif base == "field":
        prob = di.field8m(nx, ny, nz, seed)
    else:   # the paper's examples have one permeability: a field around it
        prob = di.paper_example(int(base[-1]), grid=None if (nx, ny, nz) == (10, 10, 3)
                                else (nx, ny, nz))
        n = prob.n_loc
        prob.kf = prob.kf * np.exp(0.4 * di.normals(seed, 0, n))
        prob.km = prob.km * np.exp(0.2 * di.normals(seed, 2, n))
    if "gravity" in case:
        prob.g = 9.80665 if case["gravity"] else 0.0
        if case["gravity"]:   # oil at rest: the column's own weight
            k = np.repeat(np.arange(nz), 2 * nx * ny)
            prob.p0 = prob.p0 + prob.rho_o_ref * prob.g * prob.dz * k
    if case.get("capillary"):
        s = np.linspace(prob.swc, 1.0 - prob.sor, 9)
        for name, p_entry in (("pc_f", 0.5), ("pc_m", 4.0)):
            setattr(prob, name, np.stack([s, p_entry * di.PSI * (1.0 - (s - s[0]) /
                                                                 (s[-1] - s[0])) ** 2], 1))
    return prob


def _flood(prob, seed, reach=1.0):
    """Pressure and saturation (fracture, matrix interleaved) of a waterflood
    under way: water and pressure around the injectors, a pressure sink around
    the producers, the matrix lagging behind its fracture."""
    nx, ny, nz = prob.nx, prob.ny, prob.nz
    i, j = np.arange(nx)[None, :], np.arange(ny)[:, None]
    span = reach * max(1.5, 0.18 * math.hypot(nx, ny) / math.sqrt(max(len(prob.wells) - 1, 1)))
    inj, prod = np.zeros((ny, nx)), np.zeros((ny, nx))
    for w in prob.wells:
        bell = np.exp(-((i - w.i) ** 2 + (j - w.j) ** 2) / span ** 2)
        if w.kind == di.WELL_RATE_INJ:
            inj = inj + bell
        else:
            prod = prod + bell
    inj, prod = np.minimum(inj, 1.0), np.minimum(prod, 1.0)
    layer = 1.0 - 0.3 * di.splitmix64_uniform(seed, 6, np.arange(nz))[:, None, None]
    p = np.array(prob.p0).reshape(nz, ny, nx, 2)
    sw = np.array(prob.sw0).reshape(nz, ny, nx, 2)
    top = 1.0 - prob.sor
    p[..., 0] += 20.0 * di.PSI * (layer * (inj - prod))
    p[..., 1] += 16.0 * di.PSI * (layer * (inj - prod))
    sw[..., 0] += (0.9 * top - sw[..., 0]) * (layer * inj)
    sw[..., 1] += (0.5 * top - sw[..., 1]).clip(0.0) * (layer * inj)
    return p.reshape(-1), sw.reshape(-1)


def _options(case):
    if case.get("mode") == "parity":
        return dpsim.options("parity", precision=case["precision"], schur=case["schur"])
    if case["kind"] == "solve":
        return dpsim.options("report", precision=case["precision"], schur=case["schur"],
                             eta_mode=0, eta_fixed=case["eta"])
    kw = dict(cluster_rows=-1) if case["kind"] == "ensemble" else {}
    return dpsim.options("report", precision=case["precision"], schur=case.get("schur", 0),
                         newton_tol=1e-9, **kw)


def _device(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


class _Members:
    """Realisations advanced together, each on its own stream; released in
    order (batch, realisations, streams)."""

    def __init__(self, probs, opts):
        self.streams = [dpsim.OwnedStream() for _ in probs]
        self.sims = [dpsim.Sim(p, opts, stream=s.torch) for p, s in zip(probs, self.streams)]
        self.own = dpsim.OwnedStream()
        self.batch = dpsim.Batch(self.sims, stream=self.own.torch)
        self.x0 = [_device(p.p0, p.sw0, p.bhp0) for p in probs]
        self.out = [[torch.empty_like(t) for t in x] for x in self.x0]
        torch.cuda.synchronize()

    def __del__(self):
        self.batch.close()
        for s in self.sims:
            s.close()
        for s in self.streams + [self.own]:
            s.close()


def _ensemble(case, seed):
    probs = []
    for k in range(case["members"]):
        p = di.ensemble_member(case["first"] + k * case["stride"])
        p.kf = np.exp(math.log(100.0) + di.normals(seed * 64 + k, 0, p.n_loc)) * di.MD
        probs.append(p)
    return probs


def _served(case, seed):
    probs = []
    for k in range(case["members"]):
        n = round(case["smallest"] * case["ratio"] ** k)
        probs.append(di.layered(n, n + 1, case["nz"], seed * 64 + k))
    return probs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        probs = _ensemble(case, seed)
        return dict(kind=kind, members=_Members(probs, _options(case)),
                    dts=[case["days"] * DAY] * len(probs))
    if kind == "serve":
        return dict(kind=kind, probs=_served(case, seed), opts=_options(case),
                    workers=case["workers"], dt=case["days"] * DAY)
    prob = _problem(case, seed)
    if case.get("flooded"):
        prob.p0, prob.sw0 = _flood(prob, seed)
    if kind == "assembly":
        sim = dpsim.Sim(prob, dpsim.options("parity"))
        # x^n is the problem's state, the iterate a flood a little ahead of it
        p, sw = _flood(prob, seed)
        sim.set_state(p, sw, prob.bhp0)
        sim.set_iterate(*_flood(prob, seed, 1.05), prob.bhp0 * 1.001)
        return dict(kind=kind, sim=sim, dt=case["days"] * DAY,
                    val=torch.empty((sim.nnzb, 2, 2), dtype=torch.float64, device="cuda"),
                    res=torch.empty(2 * sim.nb, dtype=torch.float64, device="cuda"))
    sim = dpsim.Sim(prob, _options(case))
    x0 = _device(prob.p0, prob.sw0, prob.bhp0)
    return dict(kind=kind, sim=sim, x0=x0, out=[torch.empty_like(t) for t in x0],
                dt=case["days"] * DAY)


# -------------------------------------------------------------------- run

def _state(sim, out):
    sim.get_state_ptr(*[t.data_ptr() for t in out])
    return {"p": out[0], "sw": out[1], "bhp": out[2]}


def run(state):
    kind = state["kind"]
    if kind == "ensemble":
        m = state["members"]
        for s, x in zip(m.sims, m.x0):
            s.set_state_device(*x)
        rc, _, _ = m.batch.advance(state["dts"])
        return {"rc": rc, "states": [_state(s, o) for s, o in zip(m.sims, m.out)]}
    if kind == "serve":
        srv = dpsim.Server(state["workers"], 64 << 30, state["opts"])
        ids = [srv.add(p) for p in state["probs"]]
        rcs = [srv.wait(t).status for t in [srv.submit(r, state["dt"]) for r in ids]]
        out = {"rc": rcs, "states": [srv.state(r) for r in ids]}
        srv.close()
        return out
    sim = state["sim"]
    if kind == "assembly":
        sim.assemble(state["dt"])
        rc = dpsim.load().sim_get_jacobian(sim.h, None, None,
                                           ctypes.c_void_p(state["val"].data_ptr()),
                                           ctypes.c_void_p(state["res"].data_ptr()))
        return {"rc": rc, "jacobian": state["val"], "residual": state["res"]}
    sim.set_state_device(*state["x0"])
    if kind == "advance":
        rc, _ = sim.advance(state["dt"])
    elif kind == "run":
        rc, st = sim.run(state["dt"], DAY, 20.0 * DAY, 0.01 * DAY)
        return {"rc": rc, "steps": st.steps, **_state(sim, state["out"])}
    else:
        sim.assemble(state["dt"])
        rc, _ = sim.solve_step()
    return {"rc": rc, **_state(sim, state["out"])}


# ------------------------------------------------------------------- work

def _sizes(case):
    """(locations, blocks of the solver's matrix, block rows) without the wells."""
    n = case["nx"] * case["ny"] * case["nz"]
    faces = 3 * n - case["nx"] * case["ny"] - case["ny"] * case["nz"] - case["nx"] * case["nz"]
    if case.get("schur"):
        return n, n + 2 * faces, n
    return n, 4 * n + 2 * faces, 2 * n


def work(case):
    """Per pass: every assembly reads the state and the rock and writes the blocks and the
    residual; every solve reads the blocks once for its factor and once an FGMRES iteration in
    FP64 and, in the preconditioner's precision, the factor and the operator of its two stage
    residuals; a new basis vector is read and written; each block product is 8 flops."""
    kind = case["kind"]
    if kind in ("ensemble", "serve"):
        probs = ([(lambda n, z: (n, n, z))(round(20 + 60 * r / 63.0), round(5 + 15 * r / 63.0))
                  for r in range(case["first"], case["first"] + case["members"] * case["stride"],
                                 case["stride"])] if kind == "ensemble" else
                 [(m, m + 1, case["nz"]) for m in
                  (round(case["smallest"] * case["ratio"] ** k) for k in range(case["members"]))])
        parts = [work(dict(kind="advance", nx=a, ny=b, nz=c, precision=case["precision"],
                           schur=0)) for a, b, c in probs]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    n, nnz, nb = _sizes(case)
    _, nnz_full, _ = _sizes(dict(case, schur=0))
    asm = {"bytes": 2 * n * 16 + 4 * n * 8 + nnz_full * 32 + 2 * n * 16,
           "flops": 60.0 * 4 * n + 60.0 * 2 * n}
    if kind == "assembly":
        return {k: float(v) for k, v in asm.items()}
    small = 4 if case["precision"] else 8
    krylov = nnz * (32 + 4) + nnz * (2 * 4 + 2) * small + 2 * nb * 16
    krylov_flops = 8.0 * nnz * 3 + 4.0 * 2 * nb * KRYLOV
    solves = {"solve": 1, "run": 4 * NEWTON}.get(kind, NEWTON)
    if kind == "run" and case["days"] < 15.0:
        solves = round(NEWTON * math.log2(case["days"] + 1))
    its = KRYLOV * (2 if case.get("mode") == "parity" or kind == "solve" else 1)
    return {"bytes": float(solves * (asm["bytes"] + 2 * nnz * 32 + its * krylov)),
            "flops": float(solves * (asm["flops"] + 8.0 * nnz * 4 + its * krylov_flops))}


# ------------------------------------------------------------------ exact
# The model restated in plain torch, 64 bits: residual and Jacobian by
# connection, derivatives by automatic differentiation of each connection's
# flux, and for problems of a few hundred cells Newton's method with a dense
# solve.

def _table(points, s):
    """The piecewise linear capillary pressure, constant outside its points."""
    if points is None:
        return torch.zeros_like(s)
    t = torch.as_tensor(points, dtype=torch.float64, device=s.device)
    k = (torch.searchsorted(t[:, 0].contiguous(), s.detach(), right=True) - 1).clamp(0, len(t) - 2)
    line = t[k, 1] + (t[k + 1, 1] - t[k, 1]) * ((s - t[k, 0]) / (t[k + 1, 0] - t[k, 0]))
    line = torch.where(s.detach() <= t[0, 0], t[0, 1], line)
    return torch.where(s.detach() >= t[-1, 0], t[-1, 1], line)


def _fluid(prob, p, s):
    """Densities and mobilities, (oil, water)."""
    rho = (prob.rho_o_ref * (1.0 + prob.c_o * (p - prob.p_ref)),
           prob.rho_w_ref * (1.0 + prob.c_w * (p - prob.p_ref)))
    S = (s - prob.swc) / (1.0 - prob.swc - prob.sor)
    S = torch.where(S <= 0.0, torch.zeros_like(S), torch.where(S >= 1.0, torch.ones_like(S), S))
    return rho, ((1.0 - S) ** 2 / prob.mu_o, S ** 2 / prob.mu_w)


def _slopes(outs, ins):
    """d outs[k] / d ins[l] where every element depends on its own inputs only."""
    return [[g if g is not None else torch.zeros_like(x) for g, x in
             zip(torch.autograd.grad(o.sum(), ins, retain_graph=True, allow_unused=True), ins)]
            if o.requires_grad else [torch.zeros_like(x) for x in ins] for o in outs]


class _Plain:
    def __init__(self, prob, device):
        self.prob = prob
        f = dict(dtype=torch.float64, device=device)
        nx, ny, nz = prob.nx, prob.ny, prob.nz
        n = prob.n_loc
        loc = torch.arange(n, device=device).reshape(nz, ny, nx)
        kf = torch.as_tensor(prob.kf, **f)
        a, b, T, dz = [], [], [], []
        for la, lb, area, dist, gz in (
                (loc[:, :, :-1], loc[:, :, 1:], prob.dy * prob.dz, prob.dx, 0.0),
                (loc[:, :-1], loc[:, 1:], prob.dx * prob.dz, prob.dy, 0.0),
                (loc[:-1], loc[1:], prob.dx * prob.dy, prob.dz, -prob.dz)):
            la, lb = la.reshape(-1), lb.reshape(-1)
            a.append(2 * la)
            b.append(2 * lb)
            T.append(2.0 * area * kf[la] * kf[lb] / (dist * (kf[la] + kf[lb])))
            dz.append(torch.full((len(la),), gz, **f))
        all_loc = torch.arange(n, device=device)
        self.V = prob.dx * prob.dy * prob.dz
        a.append(2 * all_loc)
        b.append(2 * all_loc + 1)
        T.append(prob.sigma * torch.as_tensor(prob.km, **f) * self.V)
        dz.append(torch.zeros(n, **f))
        self.a, self.b, self.T, self.dz = (torch.cat(v) for v in (a, b, T, dz))
        self.phi = torch.stack([torch.as_tensor(prob.phi_f, **f),
                                torch.as_tensor(prob.phi_m, **f)], 1).reshape(-1)
        cells, wells, wi = [], [], []
        for w, W in enumerate(prob.wells):
            r_e = 0.28 * math.sqrt(prob.dx ** 2 + prob.dy ** 2) / 2.0
            for k in range(W.k_top, W.k_bot + 1):
                q = W.i + nx * (W.j + ny * k)
                cells.append(2 * q)
                wells.append(w)
                wi.append(W.wi if W.wi > 0.0 else 2.0 * math.pi * float(prob.kf[q]) * prob.dz /
                          (math.log(r_e / W.rw) + W.skin))
        self.cell = torch.tensor(cells, device=device)
        self.well = torch.tensor(wells, device=device)
        self.wi = torch.tensor(wi, **f)
        self.kind = torch.tensor([w.kind for w in prob.wells], device=device)
        self.target = torch.tensor([w.target for w in prob.wells], **f)
        # positions of every block in the matrix with sorted columns
        self.nc, self.nb = 2 * n, 2 * n + len(prob.wells)
        rows = torch.cat([torch.arange(self.nb, device=device), self.a, self.b, self.cell,
                          self.nc + self.well])
        cols = torch.cat([torch.arange(self.nb, device=device), self.b, self.a,
                          self.nc + self.well, self.cell])
        order = torch.argsort(rows * self.nb + cols)
        self.pos = torch.empty_like(order)
        self.pos[order] = torch.arange(len(order), device=device)
        self.rows, self.cols = rows[order], cols[order]

    def mass(self, p, s):
        P = self.prob
        rho, _ = _fluid(P, p, s)
        v = self.V * self.phi * (1.0 + P.c_rock * (p - P.p_ref_rock))
        return v * rho[0] * (1.0 - s), v * rho[1] * s

    def assemble(self, x, mass_old, dt):
        """(blocks [nnz, 2, 2], residual [2 nb]) at x = (p, s, bhp)."""
        P = self.prob
        p, s, bhp = x
        val = torch.zeros((len(self.rows), 2, 2), dtype=torch.float64, device=p.device)
        res = torch.zeros((self.nb, 2), dtype=torch.float64, device=p.device)
        diag, ab, ba, cw, wc = torch.split(self.pos, [self.nb, len(self.a), len(self.a),
                                                      len(self.cell), len(self.cell)])
        blk = lambda sl, i, j: torch.stack([torch.stack([sl[0][i], sl[0][j]], -1),  # noqa: E731
                                            torch.stack([sl[1][i], sl[1][j]], -1)], -2)
        grad = lambda v: v.detach().clone().requires_grad_(True)  # noqa: E731
        # accumulation
        pc, sc = grad(p), grad(s)
        m = [(new - old) / dt for new, old in zip(self.mass(pc, sc), mass_old)]
        val[diag[:self.nc]] += blk(_slopes(m, [pc, sc]), 0, 1)
        res[:self.nc] += torch.stack(m, 1).detach()
        # fluxes, upstream weighted; the curves by continuum
        ins = [grad(v) for v in (p[self.a], s[self.a], p[self.b], s[self.b])]
        (ra, la), (rb, lb) = _fluid(P, ins[0], ins[1]), _fluid(P, ins[2], ins[3])
        face = (self.b % 2) == 0
        cap_a = _table(P.pc_f, ins[1])
        cap_b = torch.where(face, _table(P.pc_f, ins[3]), _table(P.pc_m, ins[3]))
        flux = []
        for k in range(2):
            pot = (ins[0] - ins[2]) - 0.5 * (ra[k] + rb[k]) * (P.g * self.dz)
            if k == 1:
                pot = pot - (cap_a - cap_b)
            up = torch.where(pot.detach() >= 0.0, ra[k] * la[k], rb[k] * lb[k])
            flux.append(self.T * up * pot)
        sl = _slopes(flux, ins)
        A, B = blk(sl, 0, 1), blk(sl, 2, 3)
        val[ab] += B
        val[ba] -= A
        val.index_add_(0, diag[self.a], A)
        val.index_add_(0, diag[self.b], -B)
        F = torch.stack(flux, 1).detach()
        res.index_add_(0, self.a, F)
        res.index_add_(0, self.b, -F)
        # wells
        ins = [grad(v) for v in (p[self.cell], s[self.cell], bhp[self.well])]
        rho, lam = _fluid(P, ins[0], ins[1])
        kind, dp = self.kind[self.well], ins[2] - ins[0]
        inj = kind == di.WELL_RATE_INJ
        zero = torch.zeros_like(dp)
        q = [torch.where(inj, zero, self.wi * rho[0] * lam[0] * dp),
             self.wi * rho[1] * torch.where(inj, lam[0] + lam[1], lam[1]) * dp]
        sl = _slopes(q, ins)
        val.index_add_(0, diag[self.cell], -blk(sl, 0, 1))
        for k in range(2):
            val[cw, k, 0] = -sl[k][2]
        res.index_add_(0, self.cell, -torch.stack(q, 1).detach())
        row = torch.where(inj, self.wi * (lam[0] + lam[1]) * dp,
                          torch.where(kind == di.WELL_OIL_RATE, q[0], zero))
        sl = _slopes([row], ins)
        val[wc, 0, 0], val[wc, 0, 1] = sl[0][0], sl[0][1]
        sign = torch.where(self.kind == di.WELL_OIL_RATE, 1.0, -1.0)
        wr = sign * self.target + torch.where(self.kind == di.WELL_BHP, bhp, 0.0)
        wr = wr.index_add(0, self.well, row.detach())
        wd = torch.where(self.kind == di.WELL_BHP, 1.0, 0.0).to(torch.float64)
        wd = wd.index_add(0, self.well, sl[0][2])
        val[diag[self.nc:], 0, 0], val[diag[self.nc:], 1, 1] = wd, 1.0
        res[self.nc:, 0] = wr
        return val, res.reshape(-1)

    def step(self, x, dt):
        """The state one backward-Euler step later, by dense Newton; None if it
        does not converge."""
        old = [m.detach() for m in self.mass(x[0], x[1])]
        n, prev = 2 * self.nb, None
        for _ in range(40):
            val, res = self.assemble(x, old, dt)
            J = torch.zeros((self.nb, self.nb, 2, 2), dtype=torch.float64, device=res.device)
            J[self.rows, self.cols] = val
            J = J.permute(0, 2, 1, 3).reshape(n, n)
            scale = J.abs().amax(1)
            y = torch.linalg.solve(J / scale[:, None], -(res / scale))
            y = y.reshape(self.nb, 2)
            size = float((y[:self.nc, 0].abs().max() / x[0].abs().max()).clamp_min(
                y[:self.nc, 1].abs().max()))
            x = (x[0] + y[:self.nc, 0], x[1] + y[:self.nc, 1].clamp(-0.2, 0.2),
                 x[2] + y[self.nc:, 0])
            if size < 1e-13 or (prev is not None and size < 1e-10 and size >= 0.5 * prev):
                return x
            prev = size
        return None


def exact(case, seed):
    if case["kind"] not in ("assembly", "advance"):
        return None
    if case["kind"] == "advance" and case["nx"] * case["ny"] * case["nz"] > 600:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f = dict(dtype=torch.float64, device=dev)
    prob = _problem(case, seed)
    m = _Plain(prob, dev)
    dt = case["days"] * DAY
    if case["kind"] == "assembly":
        old = [torch.as_tensor(v, **f) for v in _flood(prob, seed)]
        p, s = (torch.as_tensor(v, **f) for v in _flood(prob, seed, 1.05))
        val, res = m.assemble((p, s, torch.as_tensor(prob.bhp0 * 1.001, **f)),
                              [v.detach() for v in m.mass(*old)], dt)
        return {"rc": None, "jacobian": val, "residual": res}
    p, s = _flood(prob, seed) if case.get("flooded") else (prob.p0, prob.sw0)
    x = m.step(tuple(torch.as_tensor(v, **f) for v in (p, s, prob.bhp0)), dt)
    return None if x is None else {"rc": None, "p": x[0], "sw": x[1], "bhp": x[2]}
