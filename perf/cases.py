"""What a user of the tent-pitched Trefftz-DG solver has it do, as cases that
can be timed: sweeps of a front to the final time in one to three space
dimensions, with one or many right-hand sides, in both precisions, the energy
balance, the reverse sweep and the wave-speed gradient.

A case names a mesh (kind, n or h), a degree p, a final time T, the number of
right-hand sides, the precision, the walls and the task:

  sweep     set_state, advance to T, get_state
  balance   the same, and the energy with the energy lost in the tents
  adjoint   TentSweep forward and its backward pass (gradient with respect to
            the initial front)
  gradient  forward sweep, misfit, reverse sweep with dJ/dc per element

exact() is the method written down a second time in plain torch binary64,
all tents of a level at once: pitching (Section 2.2), the Trefftz space of
eq. (3.1), the tent system of eq. (4.1) with the Section 5 recovery terms and
the interface terms of eq. (2.5); gradients by automatic differentiation.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_1907_02367_gb300 as tp
from paper_1907_02367_gb300 import inputs

ALPHA = BETA = 0.5


def _case(name, mesh, size, p, T, nrhs, precision, walls="wave", task="sweep"):
    c = dict(mesh=mesh, size=size, p=p, T=T, nrhs=nrhs, precision=precision, walls=walls, task=task)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest user call: a 1+1D plane wave with boundary data on 16 elements; launches and latency
        _case("interval_p3_fp64", "interval", 16, 3, 1.0, 1, "fp64"),
        # the long-time energy study (Section 6.5): five elements, high degree, a long chain of tiny tents, energy out
        _case("interval_p6_balance", "interval", 5, 6, 20.0, 1, "fp64", "rest", "balance"),
        # the 2+1D standing wave on 968 triangles, one column, in both precisions: the everyday sweep
        _case("square_p4_fp64", "square", 22, 4, 1.0, 1, "fp64", "rest"),
        _case("square_p4_mixed", "square", 22, 4, 1.0, 1, "mixed", "rest"),
        # an odd small mesh with Neumann walls on one side, three columns, energy balance tracked
        _case("square_p3_neumann", "square", 13, 3, 0.7, 3, "fp64", "neumann", "balance"),
        # two materials on a graded mesh (Section 6.7), interface tents of twice the unknowns, uneven patches, p = 5
        _case("inclusion_p5_mixed", "inclusion", 0.05, 5, 0.1, 1, "mixed", "rest"),
        # the singular solution on the corner-graded L-shape (Section 6.6), Dirichlet data on the outer walls
        _case("lshape_p3_fp64", "lshape", 0.3, 3, 0.4, 1, "fp64"),
        # 3+1D, one column
        _case("cube_p3_mixed", "cube", 6, 3, 0.6, 1, "mixed", "rest"),
        # 3+1D with 64 pulses sharing the tent matrices, binary64
        _case("cube_p3_64rhs_fp64", "cube", 5, 3, 0.6, 64, "fp64", "pulses"),
        # and in the mixed precision, the large one: the benchmark's sweep on a smaller cube
        _case("cube_p3_64rhs_mixed", "cube", 10, 3, 0.6, 64, "mixed", "pulses"),
        # inversion for the initial state: forward and backward through the autograd function, four pulses
        _case("square_p4_adjoint", "square", 12, 4, 0.4, 4, "fp64", "pulses", "adjoint"),
        # inversion for the wave speed: four pulses over a disc of another speed, mixed forward, checkpoints every 8 levels
        _case("disc_p4_gradient", "disc", 14, 4, 0.3, 4, "mixed", "pulses", "gradient"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same families, sizes over their whole range."""
    kind = rng.choice(["interval", "balance", "square", "square", "inclusion", "lshape", "cube", "pulses", "adjoint",
                       "gradient"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "interval":
        n = round(_log(rng, 3, 64))
        return _case(None, "interval", n, rng.randint(2, 8), round(_log(rng, 8, 64) / n, 3), rng.choice([1, 1, 2, 5]), prec)
    if kind == "balance":
        return _case(None, "interval", rng.randint(3, 9), rng.randint(2, 8), round(_log(rng, 2, 20), 2), 1, prec, "rest",
                     "balance")
    if kind == "square":
        n = round(_log(rng, 4, 24))
        return _case(None, "square", n, rng.randint(2, 5), round(_log(rng, 0.1, min(1.0, 22 / n)), 3),
                     rng.choice([1, 1, 1, 2, 3, 6]), prec, rng.choice(["rest", "neumann", "wave"]),
                     rng.choice(["sweep", "balance"]))
    if kind == "inclusion":
        h = 0.0
        while h == 0.0 or _kappa("inclusion", h) < 0.2:   # (some sizes leave slivers where the rings meet the grid)
            h = round(rng.uniform(0.05, 0.15), 3)
        return _case(None, "inclusion", h, rng.randint(2, 5), round(rng.uniform(0.01, 0.1) * min(1.0, h / 0.07), 3), 1, prec,
                     "rest")
    if kind == "lshape":
        return _case(None, "lshape", round(rng.uniform(0.28, 0.45), 3), rng.randint(2, 5), round(rng.uniform(0.1, 0.4), 3), 1,
                     prec)
    if kind == "cube":
        return _case(None, "cube", rng.randint(2, 7), rng.randint(1, 3), round(_log(rng, 0.1, 0.6), 3), rng.choice([1, 1, 2]),
                     prec, "rest")
    if kind == "pulses":
        return _case(None, "cube", rng.randint(2, 9 if prec == "mixed" else 5), rng.randint(2, 3), round(_log(rng, 0.1, 0.6), 3),
                     rng.choice([16, 32, 48, 64, 64]), prec, "pulses")
    if kind == "adjoint":
        return _case(None, "square", rng.randint(3, 12), rng.randint(2, 4), round(_log(rng, 0.1, 0.4), 3),
                     rng.choice([1, 2, 4, 7]), prec, "pulses", "adjoint")
    mesh = rng.choice(["disc", "square"])
    return _case(None, mesh, rng.randint(5, 14), rng.randint(2, 4), round(_log(rng, 0.08, 0.3), 3),
                 rng.choice([1, 2, 4] if mesh == "disc" else [1, 4, 16]), prec, "pulses", "gradient")


# ---------------------------------------------------------------------------
# meshes and data
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _mesh(kind, size):
    if kind == "interval":
        return inputs.mesh_interval(size)
    if kind == "square":
        return inputs.mesh_square(size, 0.2, seed=2)
    if kind == "inclusion":
        return inputs.mesh_inclusion_graded(h_max=size)
    if kind == "lshape":
        return inputs.mesh_lshape(size)
    if kind == "disc":
        m = inputs.mesh_square(size, 0.2, seed=13)
        cen = m.coords[m.elems].mean(axis=1)
        m.c[:] = np.where(np.linalg.norm(cen - 0.5, axis=1) < 0.2, 1.5, 1.0)
        return m
    return inputs.mesh_cube(size, 0.1, seed=4)


@functools.lru_cache(maxsize=None)
def _kappa(kind, size):
    return inputs.pitch_kappa(_mesh(kind, size))


@functools.lru_cache(maxsize=None)
def _walls(kind, size):
    """Neumann on the wall x_1 = 0, Dirichlet elsewhere."""
    return inputs.boundary_marker(_mesh(kind, size), lambda x: x[0] < 1e-12)


@functools.lru_cache(maxsize=64)
def _tents(kind, size, T):
    m = _mesh(kind, size)
    return tp.Tents(m.coords, m.elems, m.c, _kappa(kind, size), T)


def _marker(case):
    return _walls(case["mesh"], case["size"]) if case["walls"] == "neumann" else None


class _Wave:
    """U of a case and seed, per right-hand side, with v = dU/dt and sigma = -grad U: values (n_points, n + 2)."""

    def __init__(self, case, seed):
        self.kind, self.dim = case["walls"], _mesh(case["mesh"], case["size"]).dim
        self.lshape = case["mesh"] == "lshape"
        rng = np.random.default_rng([seed, 17])
        R = case["nrhs"]
        self.amp, self.phase = rng.uniform(0.5, 1.5, R), rng.uniform(0.0, 2.0 * math.pi, R)
        d = rng.normal(size=(R, self.dim))
        self.dir = d / np.linalg.norm(d, axis=1, keepdims=True)
        self.k = rng.uniform(2.0, 5.0, R)
        self.cen, self.wid = rng.uniform(0.25, 0.75, (R, self.dim)), rng.uniform(0.08, 0.15, R)

    def at(self, r, x, t):
        """x: (N, dim), t: number or (N,), numpy or torch; the same kind out."""
        back = (lambda a: a) if torch.is_tensor(x) else (lambda a: a.numpy())
        x = torch.as_tensor(x, dtype=torch.float64)
        t = torch.as_tensor(t, dtype=torch.float64, device=x.device).expand(x.shape[0])
        if self.lshape:
            f = inputs.bessel_corner_solution()(x.cpu().numpy(), (t + self.phase[r] / 10.0).cpu().numpy())
            return back(self.amp[r] * torch.as_tensor(f, device=x.device))
        if self.kind == "pulses":
            d = x - torch.as_tensor(self.cen[r], device=x.device)
            u = self.amp[r] * torch.exp(-(d * d).sum(1) / self.wid[r] ** 2)
            return back(torch.cat([u[:, None], torch.zeros_like(u)[:, None], (2.0 / self.wid[r] ** 2) * d * u[:, None]], 1))
        if self.kind == "rest":   # standing wave, v = 0 on the walls of the unit cube
            s, c = torch.sin(math.pi * x), torch.cos(math.pi * x)
            w = math.sqrt(self.dim) * math.pi
            ct, st = torch.cos(w * t + self.phase[r]), torch.sin(w * t + self.phase[r])
            prod = s.prod(1)
            cols = [ct * prod, -w * st * prod]
            for m in range(self.dim):
                o = torch.ones_like(prod)
                for j in range(self.dim):
                    o = o * (c[:, j] if j == m else s[:, j])
                cols.append(-math.pi * ct * o)
            return back(self.amp[r] * torch.stack(cols, 1))
        ph = self.k[r] * (x @ torch.as_tensor(self.dir[r], device=x.device) - t) + self.phase[r]   # plane wave
        cols = [torch.sin(ph), -self.k[r] * torch.cos(ph)]
        cols += [-self.k[r] * float(self.dir[r][m]) * torch.cos(ph) for m in range(self.dim)]
        return back(self.amp[r] * torch.stack(cols, 1))

    @property
    def homogeneous(self):
        return self.kind in ("rest", "pulses")

    def boundary(self, r, xt, nrm, neumann):
        """g_D = v, or g_N = sigma . n where `neumann`."""
        f = self.at(r, xt[:, :-1], xt[:, -1])
        gN = (f[:, 2:] * nrm).sum(1)
        return torch.where(neumann, gN, f[:, 1]) if torch.is_tensor(f) else np.where(neumann, gN, f[:, 1])


# ---------------------------------------------------------------------------
# the framework's calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    m, wave = _mesh(case["mesh"], case["size"]), _Wave(case, seed)
    s = tp.Solver(m.coords, m.elems, m.c, case["p"], case["T"], _kappa(case["mesh"], case["size"]), nrhs=case["nrhs"],
                  tents=_tents(case["mesh"], case["size"], case["T"]), precision=case["precision"],
                  bnd_type=_marker(case), track_dissipation=case["task"] == "balance",
                  ckpt_stride=8 if case["task"] == "gradient" else 0,
                  # (the gradient takes its columns in one group: 16 of them fit split over two CTAs)
                  rhs_split=2 if case["task"] == "gradient" and case["nrhs"] == 16 else 0)
    x = torch.as_tensor(s.front_points()[0], device="cuda")
    front0 = torch.empty(s.front_shape(), dtype=torch.float64, device="cuda")
    for r in range(case["nrhs"]):
        front0[r] = wave.at(r, x, 0.0).view(front0.shape[1:])
    g = None
    if not wave.homogeneous and s.n_bnd:
        xt = s.boundary_points()
        nrm, kind = s.boundary_kinds()
        g = torch.as_tensor(np.stack([wave.boundary(r, xt, nrm, kind == 1) for r in range(case["nrhs"])]), device="cuda")
    state = dict(task=case["task"], solver=s, front0=front0, g=g)
    if case["task"] in ("adjoint", "gradient"):   # the recorded front that the misfit compares with
        state["target"] = 0.9 * front0.flip(2).contiguous()
    return state


def run(state):
    s, task = state["solver"], state["task"]
    if task == "adjoint":
        f0 = state["front0"].detach().requires_grad_(True)
        out = tp.TentSweep.apply(f0, s)
        grad, = torch.autograd.grad(out, f0, out.detach() - state["target"])
        return {"front": out.detach(), "grad_front0": grad}
    s.set_state(state["front0"], state["g"])
    s.advance()
    front, tau = s.get_state()
    if task == "gradient":
        dc = torch.empty(s.n_elem, dtype=torch.float64, device="cuda")
        lam0 = s.adjoint(front - state["target"], dJ_dc=dc)
        return {"front": front, "grad_front0": lam0, "grad_c": dc}
    out = {"front": front, "tau": tau}
    if task == "balance":
        out["energy"] = s.energy_and_dissipation()
    return out


def work(case):
    """Flops of the tent systems (assembly of one matrix per tent, moments, solve
    and outflow per right-hand side) and the front read and written once."""
    m = _mesh(case["mesh"], case["size"])
    n, p, R = m.dim, case["p"], case["nrhs"]
    nb, Q, C = math.comb(p + n, n) + math.comb(p - 1 + n, n), (p + 1) ** n, n + 2
    coef = _trefftz(n, p)[1]
    basis = coef.shape[1] - 1 + int(np.count_nonzero(coef)) + (n + 1) * nb
    v = _tents(case["mesh"], case["size"], case["T"]).export()["vert"]
    star = np.bincount(m.elems.reshape(-1), minlength=m.n_vert)[v].astype(np.float64)
    solve = nb ** 3 / 3.0 + nb * nb * R
    tents = star * Q * (3 * basis + C * nb * (nb + 1) / 2 + 2 * C * nb * R) + solve
    sweeps = {"adjoint": 2, "gradient": 3}.get(case["task"], 1)
    front = R * m.n_elem * Q * C * 8
    return {"bytes": float(2 * front * min(sweeps, 2) + m.coords.nbytes + m.elems.nbytes + 12 * len(v)),
            "flops": 2.0 * sweeps * float(tents.sum())}


# ---------------------------------------------------------------------------
# the method in plain torch
# ---------------------------------------------------------------------------
def exact(case, seed):
    m, wave = _mesh(case["mesh"], case["size"]), _Wave(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    grads = case["task"] in ("adjoint", "gradient")
    M = _Method(m, case["p"], case["T"], _kappa(case["mesh"], case["size"]), _marker(case), dev)
    if len(M.levels) > 2500:
        return None
    f0 = torch.stack([wave.at(r, M.front_x.reshape(-1, m.dim), 0.0).view(m.n_elem, M.Q, -1) for r in range(case["nrhs"])])
    target = 0.9 * f0.flip(2)
    c = torch.as_tensor(m.c, dtype=torch.float64, device=dev).clone()
    if grads:
        f0.requires_grad_(True)
        c.requires_grad_(True)
    front, D = M.sweep(f0, c, wave, case["task"] == "balance")
    if grads:
        g0, gc = torch.autograd.grad(front, (f0, c), front.detach() - target)
        out = {"front": front.detach(), "grad_front0": g0}
        return out if case["task"] == "adjoint" else dict(out, grad_c=gc)
    out = {"front": front, "tau": torch.full((m.n_vert,), case["T"], dtype=torch.float64, device=dev)}
    if case["task"] == "balance":
        E = 0.5 * (M.front_w * (front[..., 1] ** 2 / c[:, None] ** 2 + (front[..., 2:] ** 2).sum(-1))).sum((1, 2))
        out["energy"] = torch.stack([E, D], 1)
    return out


@functools.lru_cache(maxsize=None)
def _trefftz(n, p):
    """Exponents (t, x_1..x_n) of the monomials, and the coefficients of the
    c = 1 Trefftz polynomials sum_j t^(2j+s) / (2j+s)! Lap^j x^b, s = 0, 1."""
    exps = [e for e in itertools.product(range(p + 1), repeat=n + 1) if sum(e) <= p]
    where = {e: i for i, e in enumerate(exps)}
    rows = []
    for s in (0, 1):
        for b in itertools.product(range(p + 1), repeat=n):
            if sum(b) > p - s:
                continue
            row, lap, k = np.zeros(len(exps)), {b: 1.0}, s
            while lap:
                for e, v in lap.items():
                    row[where[(k,) + e]] += v / math.factorial(k)
                nxt = {}
                for e, v in lap.items():
                    for d in range(n):
                        if e[d] >= 2:
                            f = e[:d] + (e[d] - 2,) + e[d + 1:]
                            nxt[f] = nxt.get(f, 0.0) + v * e[d] * (e[d] - 1)
                lap, k = nxt, k + 2
            rows.append(row)
    return np.array(exps), np.array(rows)


def _simplex_rule(n, m):
    """Collapsed Gauss-Jacobi rule, m points per direction, as barycentric
    coordinates (Q, n+1) and weights summing to 1/n!; the first coordinate's
    points outermost."""
    dirs = []
    for d in range(n):
        a = n - 1 - d   # weight (1 - s)^a on [0, 1]: Golub-Welsch for Jacobi (a, 0)
        k = np.arange(1, m)
        diag = np.array([(-a * a) / ((2 * i + a) * (2 * i + a + 2)) if (2 * i + a) else -a / (a + 2.0) for i in range(m)])
        off = np.sqrt(4 * k * (k + a) * k * (k + a) / ((2 * k + a) ** 2 * (2 * k + a + 1) * (2 * k + a - 1)))
        x, V = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
        dirs.append(((1 + x) / 2, V[0] ** 2 / (a + 1)))
    pts, w = [], []
    for idx in itertools.product(range(m), repeat=n):
        rest, lam, wt = 1.0, [], 1.0
        for d, i in enumerate(idx):
            lam.append(rest * dirs[d][0][i])
            rest *= 1.0 - dirs[d][0][i]
            wt *= dirs[d][1][i]
        pts.append([1.0 - sum(lam)] + lam)
        w.append(wt)
    return np.array(pts), np.array(w)


class _Method:
    """The tent sweep of a mesh, every tent of a level at once."""

    def __init__(self, m, p, T, kappa, marker, dev):
        self.dev, self.n, self.p, self.T = dev, m.dim, p, T
        n, NV = m.dim, m.dim + 1
        exps, coef = _trefftz(n, p)
        self.exps, self.nb = exps, len(coef)
        where = {tuple(e): i for i, e in enumerate(exps.tolist())}
        der = []
        for d in range(n + 1):
            D = np.zeros_like(coef)
            for i, e in enumerate(exps.tolist()):
                if e[d]:
                    D[:, where[tuple(e[:d] + [e[d] - 1] + e[d + 1:])]] += e[d] * coef[:, i]
            der.append(D)
        up = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
        self.coef, self.der = up(coef.T), [up(D.T) for D in der]
        bary, wref = _simplex_rule(n, p + 1)
        self.bary, self.wref, self.Q = up(bary), up(wref), len(wref)
        self.X, self.el = up(m.coords), up(m.elems.astype(np.int64))
        XE = self.X[self.el]
        self.einv = torch.linalg.inv(XE[:, 1:] - XE[:, :1])              # gradient = einv @ increments
        self.det = torch.linalg.det(XE[:, 1:] - XE[:, :1]).abs()
        self.front_x = torch.einsum("qi,kid->kqd", self.bary, XE)
        self.front_w = self.wref * self.det[:, None]
        # stars, neighbours, boundary and interface facets of every vertex, padded with -1
        el, c = m.elems.tolist(), m.c
        star, nbr, owner = [[] for _ in range(m.n_vert)], [set() for _ in range(m.n_vert)], {}
        for k, vs in enumerate(el):
            for o, v in enumerate(vs):
                star[v].append(k)
                nbr[v].update(vs)
                owner.setdefault(tuple(sorted(vs[:o] + vs[o + 1:])), []).append((k, o))
        for v in range(m.n_vert):
            nbr[v].discard(v)
        kinds = [[[] for _ in range(m.n_vert)] for _ in range(3)]        # Dirichlet, Neumann, interface
        fac = []
        for f, own in owner.items():
            k, o = min(own)
            if len(own) == 2 and c[own[0][0]] == c[own[1][0]]:
                continue
            kind = 2 if len(own) == 2 else int(marker[k, o]) if marker is not None else 0
            fx, out = m.coords[list(f)], m.coords[el[k][o]]
            e = fx[1:] - fx[0]
            nrm = fx[0] - out if n == 1 else np.linalg.svd(e)[2][-1]
            nrm = nrm / np.linalg.norm(nrm) * (1.0 if np.dot(nrm, fx[0] - out) > 0 else -1.0)
            for v in f:
                kinds[kind][v].append(len(fac))
                fac.append(([w for w in f if w != v], nrm, k, max(own)[0]))
        pad = lambda ls: np.array([list(a) + [-1] * (max(map(len, ls)) - len(a)) for a in ls], dtype=np.int64)  # noqa: E731
        self.star, nbrp = up(pad(star)), pad([sorted(a) for a in nbr])
        self.kinds = [up(pad(ls)) if any(ls) else None for ls in kinds]
        if fac:
            self.fw = up(np.array([f[0] for f in fac], dtype=np.int64).reshape(len(fac), n - 1))
            self.fn, self.fk, self.fm = (up(np.array([f[i] for f in fac])) for i in (1, 2, 3))
        # materials of a patch: the distinct speeds of the mesh
        speeds = sorted(set(c.tolist()))
        self.ng = len(speeds)
        self.grp = up(np.array([speeds.index(s) for s in c.tolist()], dtype=np.int64))
        self.levels = self._pitch(m, nbrp, owner, kappa, T)
        self.nbr, self.cmax = up(nbrp), up(np.array([max(c[k] for k in s) for s in star]))

    @staticmethod
    def _pitch(m, nbr, owner, kappa, T):
        nv, has = m.n_vert, nbr >= 0
        cE = {}
        for k, vs in enumerate(m.elems.tolist()):
            for a, b in itertools.permutations(vs, 2):
                cE[a, b] = max(cE.get((a, b), 0.0), m.c[k])
        delta = np.full(nbr.shape, np.inf)
        for v in range(nv):
            for j, w in enumerate(nbr[v]):
                if w >= 0:
                    s = 0.0
                    for q in (m.coords[v] - m.coords[w]) ** 2:
                        s = s + q
                    delta[v, j] = kappa * math.sqrt(s) / cE[v, w]
        tau, last, tents = np.zeros(nv), np.zeros(nv, dtype=np.int64), []
        while True:
            tn = np.where(has, tau[nbr], np.inf)
            cand = np.nonzero((tau < T) & (tau <= tn.min(1)))[0]
            if not len(cand):
                break
            blocked, pick = np.zeros(nv, dtype=bool), []
            for v in cand:
                if not blocked[v]:
                    pick.append(v)
                    blocked[nbr[v][has[v]]] = True
            pick = np.array(pick)
            top = np.minimum(T, (tn[pick] + delta[pick]).min(1))
            lev = 1 + np.maximum(last[pick], np.where(has[pick], last[nbr[pick]], 0).max(1))
            tents.append((pick, tau[pick], top, lev))
            tau[pick], last[pick] = top, lev
        v, b, t, L = (np.concatenate(a) for a in zip(*tents))
        order = np.argsort(L, kind="stable")
        cuts = np.searchsorted(L[order], np.arange(1, L.max() + 2))
        return [(v[order[i:j]], b[order[i:j]], t[order[i:j]]) for i, j in zip(cuts[:-1], cuts[1:])]

    def _basis(self, xh, th):
        """U, dU/dt^, dU/dx^_m at reference points (..., n) and (...,)."""
        pw = [[torch.ones_like(th)] for _ in range(self.n + 1)]
        for d in range(self.n + 1):
            z = th if d == 0 else xh[..., d - 1]
            for _ in range(self.p):
                pw[d].append(pw[d][-1] * z)
        mono = torch.stack([functools.reduce(torch.mul, [pw[d][e] for d, e in enumerate(ex)]) for ex in self.exps.tolist()], -1)
        return mono @ self.coef, [mono @ D for D in self.der]

    def _fields(self, x, t, c, g, tent):
        """Values (B, points, C, ng nb) of the fields of every unknown at points
        of material g and speed c (per point) of each tent."""
        xv, tc, h = tent
        sh = (len(h),) + (1,) * (x.dim() - 2)
        hh = h.view(sh)
        U, D = self._basis((x - xv.view(sh + (self.n,))) / hh[..., None], c * (t - tc.view(sh)) / hh)
        F = torch.stack([U, D[0] * (c / hh)[..., None]] + [-D[1 + d] / hh[..., None] for d in range(self.n)], -2)
        if self.ng > 1:
            one = torch.nn.functional.one_hot(g, self.ng).to(F.dtype).expand(x.shape[:-1] + (self.ng,))
            F = (one[..., None, :, None] * F[..., :, None, :]).flatten(-2)
        return F.flatten(1, -3)

    def sweep(self, front, c, wave, balance):
        n, Q, R = self.n, self.Q, front.shape[0]
        tau = torch.zeros(len(self.X), dtype=torch.float64, device=self.dev)
        lost = torch.zeros(R, dtype=torch.float64, device=self.dev)
        for v, tb, tt in self.levels:
            v, tb, tt = (torch.as_tensor(a, device=self.dev) for a in (v, tb, tt))
            front, D = self._level(front, c, tau, v, tb, tt, wave, balance)
            tau = tau.index_put((v,), tt)
            lost = lost + D
        return front, lost

    def _level(self, front, c, tau, v, tb, tt, wave, balance):
        n, Q, B, R = self.n, self.Q, len(v), front.shape[0]
        nbr = self.nbr[v]
        # tent scale: the anisotropic diameter of its vertices (eq. 3.3)
        ok = torch.cat([torch.ones(B, 2, dtype=torch.bool, device=self.dev), nbr >= 0], 1)
        px = torch.cat([self.X[v][:, None].expand(B, 2, n), self.X[nbr.clamp(min=0)]], 1)
        pt = torch.cat([tb[:, None], tt[:, None], tau[nbr.clamp(min=0)]], 1)
        d2 = ((px[:, :, None] - px[:, None]) ** 2).sum(-1) + (self.cmax[v].view(B, 1, 1) * (pt[:, :, None] - pt[:, None])) ** 2
        h = torch.where(ok[:, :, None] & ok[:, None], d2, 0.0).amax((1, 2)).sqrt()
        tent = (self.X[v], 0.5 * (tb + tt), h)
        st = self.star[v]
        st = st[:, (st >= 0).any(0)]
        live, k = st >= 0, st.clamp(min=0)
        top_t = tau.index_put((v,), tt)                                # tents of a level do not share elements
        T0, T1 = tau[self.el[k]], top_t[self.el[k]]                    # (B, P, n+1)
        g0, g1 = (torch.einsum("bpdi,bpi->bpd", self.einv[k], t[..., 1:] - t[..., :1]) for t in (T0, T1))
        x, w = self.front_x[k], (self.front_w[k] * live[..., None]).flatten(1)
        ck = c[k][..., None].expand(k.shape + (Q,))
        gk = self.grp[k][..., None].expand_as(ck)
        t0, t1 = (torch.einsum("qi,bpi->bpq", self.bary, t) for t in (T0, T1))
        F0, F1 = self._fields(x, t0, ck, gk, tent), self._fields(x, t1, ck, gk, tent)
        ic2 = (1.0 / ck ** 2).flatten(1)
        rep = lambda g: g[:, :, None].expand(k.shape + (Q, n)).flatten(1, 2)  # noqa: E731

        def dual(F, g):   # (U, v, sigma) -> the face form's dual values (0, c^-2 v - sigma.g, sigma - v g)
            V, S = F[:, :, 1:2], F[:, :, 2:]
            return torch.cat([0.0 * V, ic2[..., None, None] * V - (S * g[..., None]).sum(2, keepdim=True),
                              S - V * g[..., None]], 2)

        flat = lambda F: F.flatten(1, 2)  # noqa: E731  (B, points C, N)
        W = w[..., None, None]
        A = flat(F1).transpose(1, 2) @ flat(W * dual(F1, rep(g1)))
        A = A + F0[:, :, 0].transpose(1, 2) @ (w[..., None] * F0[:, :, 0])
        fb = front[:, k].permute(1, 2, 3, 4, 0).flatten(1, 2)           # (B, points, C, R)
        data = torch.cat([fb[:, :, :1], dual(fb, rep(g0))[:, :, 1:]], 2)
        b = flat(F0).transpose(1, 2) @ flat(W * data)
        N = A.shape[1]
        have = (torch.nn.functional.one_hot(self.grp[k], self.ng) * live[..., None]).amax(1)
        A = A + torch.diag_embed((1.0 - have).repeat_interleave(self.nb, 1))
        faces = []
        for kind in range(3):
            if self.kinds[kind] is None:
                continue
            f = self.kinds[kind][v]
            if not bool((f >= 0).any()):
                continue
            there, f = f >= 0, f.clamp(min=0)
            X = torch.cat([self.X[v][:, None, None].expand(f.shape + (2, n)), self.X[self.fw[f]]], 2)
            Tm = torch.cat([tb[:, None, None].expand(f.shape + (1,)), tt[:, None, None].expand(f.shape + (1,)), tau[self.fw[f]]], 2)
            E = torch.cat([X, Tm[..., None]], -1)
            E = E[:, :, 1:] - E[:, :, :1]
            wf = (self.wref * torch.linalg.det(E @ E.transpose(-1, -2)).abs().sqrt()[..., None] * there[..., None]).flatten(1)
            xf, tf = torch.einsum("qi,bfid->bfqd", self.bary, X), torch.einsum("qi,bfi->bfq", self.bary, Tm)
            nr = self.fn[f][:, :, None].expand(xf.shape).flatten(1, 2)

            def side(e):
                F = self._fields(xf, tf, c[e][..., None].expand(tf.shape), self.grp[e][..., None].expand(tf.shape), tent)
                return F[:, :, 0], F[:, :, 1], (F[:, :, 2:] * nr[..., None]).sum(2)

            U, V, S = side(self.fk[f])
            wq = wf[..., None]
            if kind == 2:
                _, Vm, Sm = side(self.fm[f])
                jv, js, av, as_ = V - Vm, S - Sm, 0.5 * (V + Vm), 0.5 * (S + Sm)
                A = A + js.transpose(1, 2) @ (wq * (av + BETA * js)) + jv.transpose(1, 2) @ (wq * (as_ + ALPHA * jv))
                faces.append((kind, wf, jv, js, None))
                continue
            G = torch.zeros(R, B, wf.shape[1], dtype=torch.float64, device=self.dev)
            if not wave.homogeneous:
                xt = torch.cat([xf, tf[..., None]], -1).reshape(-1, n + 1)
                yes = torch.full((len(xt),), kind == 1, device=self.dev)
                G = torch.stack([wave.boundary(r, xt, nr.reshape(-1, n), yes) for r in range(R)]).view(G.shape)
            Gt = (G * wf).permute(1, 2, 0)
            if kind == 0:
                A = A + V.transpose(1, 2) @ (wq * (S + ALPHA * V))
                b = b + (ALPHA * V - S).transpose(1, 2) @ Gt
            else:
                A = A + S.transpose(1, 2) @ (wq * (V + BETA * S))
                b = b + (BETA * S - V).transpose(1, 2) @ Gt
            faces.append((kind, wf, V, S, G.permute(1, 2, 0)))
        e = A.diagonal(dim1=1, dim2=2).abs().rsqrt().detach()
        As, bs = A * e[:, :, None] * e[:, None], b * e[:, :, None]
        y = torch.linalg.solve(As, bs)
        if not A.requires_grad:
            for _ in range(2):
                y = y + torch.linalg.solve(As, bs - As @ y)
        z = y * e[:, :, None]                                          # (B, N, R)
        out = (flat(F1) @ z).view(B, len(k[0]), Q, n + 2, R)[live].permute(3, 0, 1, 2)
        D = torch.zeros(R, dtype=torch.float64, device=self.dev)
        if balance:
            u0 = (flat(F0) @ z).view(B, -1, n + 2, R)
            du, gg = u0 - fb, rep(g0)[..., None]
            q = ic2[..., None] * du[:, :, 1] ** 2 + (du[:, :, 2:] ** 2).sum(2) - 2.0 * du[:, :, 1] * (du[:, :, 2:] * gg).sum(2)
            D = D + (w[..., None] * (0.5 * q + du[:, :, 0] * u0[:, :, 0])).sum((0, 1))
            for kind, wf, V, S, G in faces:
                a, s = V @ z, S @ z
                val = (ALPHA * a * a + BETA * s * s if kind == 2 else ALPHA * a * a - G * (ALPHA * a - s) if kind == 0
                       else BETA * s * s - G * (BETA * s - a))
                D = D + (wf[..., None] * val).sum((0, 1))
        return front.index_put((torch.arange(R, device=self.dev)[:, None], k[live][None]), out), D
