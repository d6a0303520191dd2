"""The work that is measured: what programs have this framework do.

Each case is one call sequence of a user's program through the public entry
points of ``paper_2607_20704_gb300.amr`` (``Mesh``, ``Particles``), on the
recipes of ``paper_2607_20704_gb300.inputs``:

``solve``     a resident mesh takes a new state from pinned host memory, advances
              some coarse steps (CFL step, W-cycle over the levels) and its state
              goes back to pinned host memory: one request of a solve loop
``ensemble``  the same for a handle of several meshes advanced together
``substeps``  a program that drives the level steps itself: the time step, then
              every level in W-cycle order
``adaptive``  a mesh is created from host arrays and regridded before each of a
              few coarse steps; the resulting octs and states are read back
``gravity``   multigrid potential of the base level or of every level, read back
``deposit``   particles resident on the device are sorted and deposited on a
              uniform grid, and the density is taken as a device tensor
``levels``    particles in device arrays are deposited onto every level of a mesh

The mesh of a case is fixed by the case; the seed gives the state on it (the
recipe's state with seeded density noise, pressures and velocities kept) or
the particles.  ``exact`` evaluates the same definitions in 64 bits with plain
torch on dense arrays (per level, cut to the level's bounding box).
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2607_20704_gb300 import amr, inputs

DEV = "cuda"
F64 = torch.float64
_STREAM = []


def stream():
    """One stream for all handles, as a program with one compute queue has."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest calls: a mesh of a few hundred octs, where launches and latency count
        dict(name="small_random_fp64", kind="solve", mesh="random", levelmin=3, levelmax=6, shape=1.0,
             precision=8, steps=6),
        # the shock tube with one refined slab, ten coarse steps
        dict(name="sod_fp64", kind="solve", mesh="sod", levelmin=6, levelmax=7, shape=1.0, precision=8, steps=10),
        # the blast with three refined levels (the benchmark's mesh), each precision
        dict(name="sedov_fp64", kind="solve", mesh="sedov", levelmin=7, levelmax=10, shape=1.0, precision=8,
             steps=3),
        dict(name="sedov_fp32", kind="solve", mesh="sedov", levelmin=7, levelmax=10, shape=1.0, precision=4,
             steps=12),
        # one level of 256^3 cells: the setting of uniform-grid rates, the largest state
        dict(name="uniform_fp32", kind="solve", mesh="uniform", levelmin=8, levelmax=8, shape=1.0, precision=4,
             steps=6),
        # a parameter study: many small blasts in one handle
        dict(name="ensemble_fp32", kind="ensemble", mesh="sedov", levelmin=5, levelmax=7, shape=1.5, precision=4,
             members=24, steps=6),
        # clustered densities, the program steps the levels itself
        dict(name="clustered_substeps_fp64", kind="substeps", mesh="lognormal", levelmin=6, levelmax=9, shape=1.0,
             precision=8, steps=2),
        # a blast whose mesh follows it
        dict(name="adaptive_fp64", kind="adaptive", mesh="sedov", levelmin=6, levelmax=9, shape=1.0, precision=8,
             steps=6),
        # self-gravity on every level of a clustered mesh
        dict(name="gravity_levels", kind="gravity", mesh="lognormal", levelmin=7, levelmax=9, shape=1.0,
             precision=8, cycles=4, levels=True),
        # particle mass on a grid with as many cells as particles: the quick and the reproducible way
        dict(name="deposit_atomic_fp32", kind="deposit", grid=256, lattice=256, algo="atomic", precision=4),
        dict(name="deposit_segment_fp64", kind="deposit", grid=128, lattice=128, algo="segment", precision=8),
        # particle mass on the levels of a clustered mesh
        dict(name="deposit_levels_fp64", kind="levels", mesh="lognormal", levelmin=7, levelmax=9, shape=1.0,
             lattice=160, precision=8),
    ]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "ensemble", "substeps", "adaptive", "gravity",
                       "deposit", "deposit", "levels"])
    prec = rng.choice([4, 8])
    shape = round(rng.uniform(0.7, 1.3), 3)
    if kind == "solve":
        mesh = rng.choice(["random", "sod", "sedov", "uniform", "lognormal"])
        lo, hi = {"random": (3, 5), "sod": (4, 6), "sedov": (4, 7), "uniform": (4, 7), "lognormal": (4, 7)}[mesh]
        lmin = rng.randint(lo, hi)
        extra = {"sod": 1, "uniform": 0}.get(mesh, rng.randint(1, 2 if mesh == "lognormal" else 3))
        top = {4: 40, 5: 24, 6: 10, 7: 3}.get(lmin, 40)
        return dict(kind=kind, mesh=mesh, levelmin=lmin, levelmax=lmin + extra, shape=shape, precision=prec,
                    steps=rng.randint(1, top))
    if kind == "ensemble":
        lmin = rng.randint(4, 5)
        return dict(kind=kind, mesh=rng.choice(["sod", "sedov"]), levelmin=lmin, levelmax=lmin + 1, shape=shape,
                    precision=prec, members=rng.randint(3, 41), steps=rng.randint(1, 6))
    if kind == "substeps":
        lmin = rng.randint(4, 6)
        return dict(kind=kind, mesh=rng.choice(["lognormal", "random"]), levelmin=lmin,
                    levelmax=lmin + rng.randint(1, 2), shape=shape, precision=prec, steps=rng.randint(1, 4))
    if kind == "adaptive":
        lmin = rng.randint(4, 6)
        return dict(kind=kind, mesh="sedov", levelmin=lmin, levelmax=lmin + rng.randint(1, 3), shape=shape,
                    precision=8, steps=rng.randint(1, 6))
    if kind == "gravity":
        lmin = rng.randint(4, 8)
        return dict(kind=kind, mesh="lognormal", levelmin=lmin, levelmax=min(lmin + 2, 9), shape=shape,
                    precision=prec, cycles=rng.randint(1, 6), levels=lmin < 8)
    if kind == "deposit":
        return dict(kind=kind, grid=2 ** rng.randint(5, 8), lattice=int(math.exp(rng.uniform(math.log(21), math.log(230)))),
                    algo=rng.choice(["atomic", "segment"]), precision=prec)
    lmin = rng.randint(4, 7)
    return dict(kind=kind, mesh="lognormal", levelmin=lmin, levelmax=lmin + 2, shape=shape,
                lattice=int(math.exp(rng.uniform(math.log(21), math.log(150)))), precision=prec)


# ---------------------------------------------------------------------------
# meshes and states
# ---------------------------------------------------------------------------
def hilbert(x, y, z, bits):
    """3-D Hilbert index, x most significant (Skilling 2004): the order in
    which a level's octs are kept."""
    a = [np.asarray(t, np.int64).copy() for t in (x, y, z)]
    for b in range(bits - 1, 0, -1):
        m = (1 << b) - 1
        for d in range(3):
            up = ((a[d] >> b) & 1).astype(bool)
            t = np.where(up, 0, (a[0] ^ a[d]) & m)
            a[0] ^= np.where(up, m, t)
            if d:
                a[d] ^= t
    a[1] ^= a[0]
    a[2] ^= a[1]
    g = np.zeros_like(a[2])
    for b in range(bits - 1, 0, -1):
        g ^= np.where((a[2] >> b) & 1, (1 << b) - 1, 0)
    h = np.zeros_like(g)
    for b in range(bits - 1, -1, -1):
        for t in a:
            h = (h << 1) | (((t ^ g) >> b) & 1)
    return h


def _blast_on_grid(level):
    """Unit density at rest, unit energy in a ball of two cells' radius."""
    r0 = 2.0 / (1 << level)

    def fn(x, y, z):
        r2 = (x - 0.5) ** 2 + (y - 0.5) ** 2 + (z - 0.5) ** 2
        p = np.where(r2 < r0 * r0, (2.0 / 3.0) / (4.0 / 3.0 * np.pi * r0 ** 3), 1e-5)
        zero = 0.0 * x
        return 1.0 + zero, zero, zero, zero, p
    return inputs.uniform_grid(level, fn, gamma=5.0 / 3.0)


@functools.lru_cache(maxsize=3)
def _problem(mesh, lmin, lmax, shape):
    """The recipe's mesh and state, octs in mesh order (level, Hilbert)."""
    if mesh == "random":
        p = inputs.random_mesh(lmin, lmax, 5, radius=0.2 * shape)
    elif mesh == "sod":
        p = inputs.sod(lmin, lmax, slab=(0.5 - 0.05 * shape, 0.5 + 0.05 * shape))
    elif mesh == "sedov":
        p = inputs.sedov(lmin, lmax, radii={l: 0.03 * shape * 2.0 ** (lmax - l) for l in range(lmin + 1, lmax + 1)})
    elif mesh == "uniform":
        p = _blast_on_grid(lmin)
    else:  # the smoothed, isothermal variant: well posed over many steps
        p = inputs.lognormal(lmin, lmax - lmin, threshold=4.0 * shape, smooth=1.0, isothermal=0.01)
    h = np.zeros(p.n_oct, np.int64)
    for l in range(lmin, lmax + 1):
        s = p.level == l
        h[s] = hilbert(p.i[s], p.j[s], p.k[s], l - 1)
    o = np.lexsort((h, p.level))
    cells = (8 * o[:, None] + np.arange(8)[None, :]).ravel()
    p.level, p.i, p.j, p.k = p.level[o], p.i[o], p.j[o], p.k[o]
    p.U = np.ascontiguousarray(p.U[:, cells])
    p.levelmax = max(lmax, int(p.level.max())) if mesh != "lognormal" else lmax
    return p


def _mesh_of(case):
    return _problem(case["mesh"], case["levelmin"], case["levelmax"], case["shape"])


def _state(p, seed):
    """The recipe's state with 1 % seeded density noise (pressures and
    velocities kept), split cells holding the mean of their children."""
    f = 1.0 + 0.01 * np.random.default_rng(seed).standard_normal(p.U.shape[1]).clip(-3, 3)
    U = p.U.copy()
    ek = 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0]
    U[:4] *= f
    U[4] += ek * (f - 1.0)
    lv = p.level
    for l in range(int(lv.max()), p.levelmin, -1):
        s = np.flatnonzero(lv == l)
        c0 = np.flatnonzero(lv == l - 1)
        code = lambda i, j, k: (i.astype(np.int64) << 40) | (j.astype(np.int64) << 20) | k.astype(np.int64)  # noqa: E731
        cc = code(p.i[c0], p.j[c0], p.k[c0])
        order = np.argsort(cc)
        f_oct = c0[order[np.searchsorted(cc[order], code(p.i[s] >> 1, p.j[s] >> 1, p.k[s] >> 1))]]
        fc = (p.i[s] & 1) + 2 * (p.j[s] & 1) + 4 * (p.k[s] & 1)
        kids = U.reshape(5, -1, 8)[:, s]
        acc = kids[:, :, 0].copy()
        for c in range(1, 8):
            acc += kids[:, :, c]
        U.reshape(5, -1, 8)[:, f_oct, fc] = acc / 8.0
    return U


def _pinned(a):
    t = torch.empty(a.shape, dtype=F64, pin_memory=True).numpy()
    t[:] = a
    return t


def _w_cycle(levels, l=None):
    l = levels[0] if l is None else l
    finer = _w_cycle(levels, l + 1) * 2 if l < levels[-1] else []
    return finer + [l]


def _particles(case, seed):
    return inputs.particles(case.get("grid", 2 ** case.get("levelmin", 7)), "cosmo", seed, lattice=case["lattice"])


def prepare(case, seed):
    kind, s = case["kind"], {"case": case, "kind": case["kind"]}
    prec = case["precision"]
    if kind == "deposit":
        ps = _particles(case, seed)
        s["parts"] = amr.Particles(*ps.args(), precision=prec, stream=stream())
        return s
    p = _mesh_of(case)
    if kind == "adaptive":
        s["args"] = (p.level, p.i, p.j, p.k, _state(p, seed))
        s["params"] = p.params()
        return s
    members = case.get("members", 1)
    states = [_state(p, seed * 1000 + q) for q in range(members)]
    mem = [dict(level=p.level, i=p.i, j=p.j, k=p.k, U=U, **p.params()) for U in states]
    s["mesh"] = amr.Mesh(members=mem, precision=prec, stream=stream())
    s["levels"] = s["mesh"].levels()
    if kind in ("solve", "ensemble", "substeps"):
        s["in"] = [_pinned(U) for U in states]
        s["out"] = [_pinned(np.zeros_like(U)) for U in states]
    if kind == "levels":
        dt = F64 if prec == 8 else torch.float32
        s["parts"] = [torch.from_numpy(a).to(device=DEV, dtype=dt) for a in _particles(case, seed).args()[1:]]
    return s


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "deposit":
        s["parts"].sort()
        s["parts"].deposit(case["algo"])
        with torch.cuda.stream(stream()):  # the program's own copy: the view ends with the handle's next deposit
            return s["parts"].rho_device().clone()
    if kind == "adaptive":
        # the launch shape is given, as a program that creates many meshes gives it
        with amr.Mesh(*s["args"], **s["params"], precision=case["precision"], stream=stream(), tile=128, schedule=0,
                      nsubgrid=0, refine_grad_rho=0.1, refine_grad_p=0.1, regrid_every_step=True) as m:
            m.advance(case["steps"])
            return {l: m.read(l) for l in m.levels()}
    m = s["mesh"]
    if kind == "gravity":
        if case["levels"]:
            m.poisson_levels(1.0, case["cycles"], residuals=False)
            return [m.read_phi_level(l) for l in s["levels"]]
        m.poisson(1.0, case["cycles"], residuals=False)
        return m.read_phi()
    if kind == "levels":
        counts = m.cic_deposit_levels_device(*s["parts"])
        return counts, [m.particle_rho(l) for l in s["levels"]]
    for q, U in enumerate(s["in"]):
        if len(s["in"]) > 1:
            m.select(q)
        m.load_state_async(U)
    dts = []
    if kind == "substeps":
        for _ in range(case["steps"]):
            dt = m.cfl_dt()
            for l in _w_cycle(s["levels"]):
                m.step_level(l, dt * 0.5 ** (l - s["levels"][0]))
            dts.append(dt)
    else:
        m.advance(case["steps"])
    for q, out in enumerate(s["out"]):
        if len(s["out"]) > 1:
            m.select(q)
        m.store_state_async(out)
    return s["out"] + dts


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how far correct results may differ
# ---------------------------------------------------------------------------
FLOPS_PER_UPDATE = 445  # primitives, predictor, three Riemann solves and the update of a cell


def work(case):
    w = case["precision"]
    if case["kind"] == "deposit":
        n, cells = case["lattice"] ** 3, case["grid"] ** 3
        # the sort writes the particles once more; 8 products and 8 sums per particle
        return {"bytes": (3 * 4 * w + 8) * n + w * cells, "flops": 40 * n}
    p = _mesh_of(case)
    noct = {l: int(np.count_nonzero(p.level == l)) for l in range(p.levelmin, int(p.level.max()) + 1)}
    cells = 8 * p.n_oct
    if case["kind"] == "levels":
        n = case["lattice"] ** 3
        return {"bytes": 4 * w * n + (w + 8) * cells, "flops": 40 * n}
    if case["kind"] == "gravity":
        c = cells if case["levels"] else 8 * noct[p.levelmin]
        # per V-cycle and cell: 4 sweeps of 8, residual and restriction 10, prolongation 6, the coarse grids an
        # eighth of it again; the density read and the potential written once
        return {"bytes": (8 + w) * c, "flops": 55.0 * c * case["cycles"]}
    leaf = {l: 8 * n - noct.get(l + 1, 0) for l, n in noct.items()}
    upd = sum(n << (l - p.levelmin) for l, n in leaf.items()) * case["steps"] * case.get("members", 1)
    host = 80 * cells * case.get("members", 1)
    return {"bytes": 10 * w * upd + host, "flops": FLOPS_PER_UPDATE * upd}


def tolerance(case):
    """About four times what the path shows against ``exact`` over the listed
    cases and drawn ones: hydro 4.5e-16 in FP64 (more for other orders of the
    same sums, which shocks carry on over hundreds of level steps) and 6.5e-7
    in FP32; the potential 2e-14 (FP32 densities 3.3e-9); deposits 1.9e-15 and
    1.8e-6."""
    kind, fp32 = case["kind"], case["precision"] == 4
    if kind == "gravity":
        return {"rel": 2e-8, "max": 2e-7} if fp32 else {"rel": 1e-13, "max": 4e-13}
    if kind in ("deposit", "levels"):
        return {"rel": 8e-6, "max": 4e-5} if fp32 else {"rel": 1e-14, "max": 4e-14}
    return {"rel": 3e-6, "max": 3e-5} if fp32 else {"rel": 1e-14, "max": 1e-12}


# ---------------------------------------------------------------------------
# the definitions in 64 bits
# ---------------------------------------------------------------------------
class _Level:
    """One level on dense arrays [z, y, x] over the bounding box of its cells
    and a margin of at least four cells (the whole periodic box along an axis
    that the cells nearly fill); rolls wrap, which in a cut box touches the
    margin only."""

    def __init__(self, level, i, j, k):
        self.l, self.side = level, 1 << level
        c = np.arange(8)
        xyz = [(2 * t.astype(np.int64)[:, None] + b[None, :]).ravel()
               for t, b in ((i, c & 1), (j, (c >> 1) & 1), (k, (c >> 2) & 1))]
        self.lo, self.n = [0] * 3, [self.side] * 3
        for d, t in enumerate(xyz):
            lo, hi = (int(t.min()) - 4) & ~1, (int(t.max()) + 6) & ~1
            if hi - lo < self.side:
                self.lo[d], self.n[d] = lo, hi - lo
        self.at = torch.from_numpy(self.index(*xyz)).to(DEV)  # place of every cell, octs in the given order
        shape = tuple(self.n[::-1])
        self.ex = torch.zeros(shape, dtype=torch.bool, device=DEV)
        self.ex.view(-1)[self.at] = True
        self.split = torch.zeros_like(self.ex)
        self.U = torch.zeros((5,) + shape, dtype=F64, device=DEV)
        self.R = torch.zeros_like(self.U)
        self.octs = (i, j, k)

    def index(self, x, y, z):
        q = [(t - lo) % self.side for t, lo in zip((x, y, z), self.lo)]
        return (q[2] * self.n[1] + q[1]) * self.n[0] + q[0]

    def into(self, fine, step):
        """Index tensors of this level's cells under the fine level's cells
        (step 1) or under its aligned blocks of eight (step 2)."""
        out = []
        for d in (2, 1, 0):
            f = (fine.lo[d] + torch.arange(0, fine.n[d], step, device=DEV)) % fine.side
            q = ((f >> 1) - self.lo[d]) % self.side
            out.append(q.clamp(max=self.n[d] - 1))  # only margins are ever clamped
        return out[0][:, None, None], out[1][None, :, None], out[2][None, None, :]

    def get(self):
        return self.U.view(5, -1)[:, self.at]


def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


def _blocks_mean(t):
    """Mean over aligned blocks of eight, children summed in child order."""
    s = None
    for cz, cy, cx in itertools.product(range(2), range(2), range(2)):
        v = t[..., cz::2, cy::2, cx::2]
        s = v.clone() if s is None else s + v
    return s / 8.0


class _Amr:
    def __init__(self, p, U):
        self.g, self.cfl, self.sr, self.sc = p.gamma, p.cfl, 1e-10, 1e-10
        self.lmin, self.lmax = p.levelmin, p.levelmax
        self.build({l: (p.i[p.level == l], p.j[p.level == l], p.k[p.level == l])
                    for l in range(p.levelmin, int(p.level.max()) + 1)})
        U = torch.from_numpy(U).to(DEV)
        at = 0
        for L in self.lv.values():
            L.U.view(5, -1)[:, L.at] = U[:, at:at + L.at.numel()]
            at += L.at.numel()

    def build(self, octs):
        self.lv = {l: _Level(l, *o) for l, o in octs.items()}
        for l in list(self.lv)[1:]:
            self.lv[l - 1].split[self.lv[l - 1].into(self.lv[l], 2)] |= self.lv[l].ex[::2, ::2, ::2]
        for l in list(self.lv)[1:]:
            self.lv[l - 1].split &= self.lv[l - 1].ex

    def full(self, l):
        """The level's values, those of the covering coarser cell elsewhere."""
        L = self.lv[l]
        if l == self.lmin:
            return L.U
        C = self.lv[l - 1]
        return torch.where(L.ex, L.U, self.full(l - 1)[(slice(None),) + C.into(L, 1)])

    def children(self, l):
        """Minmod prolongation of level l-1 onto level l."""
        A = self.full(l - 1)
        L, C = self.lv[l], self.lv[l - 1]
        idx = (slice(None),) + C.into(L, 1)
        out = A[idx].clone()
        for d, ax in ((0, 3), (1, 2), (2, 1)):
            s = _minmod(torch.roll(A, -1, ax) - A, A - torch.roll(A, 1, ax))[idx]
            q = (L.lo[d] + torch.arange(L.n[d], device=DEV)) & 1
            sh = [1, 1, 1, 1]
            sh[ax] = -1
            out += (0.5 * q.to(F64) - 0.25).view(sh) * s
        return out

    def prim(self, U):
        r = U[0].clamp(min=self.sr)
        v = U[1:4] / r
        p = (self.g - 1) * (U[4] - 0.5 * r * (v * v).sum(0))
        p = torch.maximum(p, r * (self.sc ** 2 / self.g))
        return torch.stack([r, v[0], v[1], v[2], p])

    def hllc(self, qL, qR, d):
        g = self.g
        for q in (qL, qR):
            q[0].clamp_(min=self.sr)
            q[4] = torch.maximum(q[4], q[0] * (self.sc ** 2 / g))
        rl, ul, pl, rr, ur, pr = qL[0], qL[1 + d], qL[4], qR[0], qR[1 + d], qR[4]
        c = torch.sqrt(torch.maximum(g * pl / rl, g * pr / rr))
        sl, sr = torch.minimum(ul, ur) - c, torch.maximum(ul, ur) + c
        rcl, rcr = rl * (ul - sl), rr * (sr - ur)
        us = (rcr * ur + rcl * ul + (pl - pr)) / (rcl + rcr)
        ps = (rcr * pl + rcl * pr + rcl * rcr * (ul - ur)) / (rcl + rcr)
        left = (sl > 0) | (us > 0)
        q = torch.where(left, qL, qR)
        e = q[4] / (g - 1) + 0.5 * q[0] * (q[1:4] ** 2).sum(0)
        sk, star = torch.where(left, sl, sr), torch.where(left, sl <= 0, sr > 0)
        u, p, r = q[1 + d], q[4], q[0]
        rs = torch.where(star, r * (sk - u) / (sk - us), r)
        es = torch.where(star, ((sk - u) * e - p * u + ps * us) / (sk - us), e)
        uo, po = torch.where(star, us, u), torch.where(star, ps, p)
        m = rs * uo
        F = torch.stack([m, m * q[1], m * q[2], m * q[3], (es + po) * uo])
        F[1 + d] = m * uo + po
        return F

    def step(self, l, dt):
        L = self.lv[l]
        V = L.U if l == self.lmin else torch.where(L.ex, L.U, self.children(l))
        W = self.prim(V)
        dtdx = dt * 2.0 ** l
        dW = [_minmod(torch.roll(W, -1, ax) - W, W - torch.roll(W, 1, ax)) for ax in (3, 2, 1)]
        r, p = W[0], W[4]
        src = torch.zeros_like(W)
        for d in range(3):
            u, dw = W[1 + d], dW[d]
            src -= u * dw
            src[0] -= r * dw[1 + d]
            src[1 + d] -= dw[4] / r
            src[4] -= self.g * p * dw[1 + d]
        Ws = W + 0.5 * dtdx * src
        del src, W, V
        dU = torch.zeros_like(L.U)
        leaf = L.ex & ~L.split
        for d, ax in ((0, 3), (1, 2), (2, 1)):
            F = self.hllc(Ws + 0.5 * dW[d], torch.roll(Ws - 0.5 * dW[d], -1, ax), d)
            exn, spn = torch.roll(L.ex, -1, ax - 1), torch.roll(L.split, -1, ax - 1)
            F = torch.where((L.ex | exn) & ~L.split & ~spn, F, torch.zeros_like(F))
            dU += torch.roll(F, 1, ax) - F
            if l > self.lmin:  # coarse-fine faces: the cell without an oct on one side
                plus = torch.where(L.ex & ~exn, F, torch.zeros_like(F))
                minus = torch.where(~L.ex & exn, F, torch.zeros_like(F))
                self.reflux(l, dtdx * (torch.roll(plus, 1, ax) - minus))
        L.U = torch.where(leaf, (L.U + dtdx * dU) + L.R, L.U)
        L.R.zero_()
        if l > self.lmin:
            C = self.lv[l - 1]
            iz, iy, ix = C.into(L, 2)
            m = L.ex[::2, ::2, ::2]
            at = ((iz * C.n[1] + iy) * C.n[0] + ix)[m]
            C.U.view(5, -1)[:, at] = _blocks_mean(L.U)[:, m]

    def reflux(self, l, D):
        L, C = self.lv[l], self.lv[l - 1]
        s = _blocks_mean(D)
        m = (s != 0).any(0)
        iz, iy, ix = C.into(L, 2)
        at = ((iz * C.n[1] + iy) * C.n[0] + ix)[m]
        C.R.view(5, -1).index_add_(1, at, s[:, m])

    def dt(self):
        out = math.inf
        for l, L in self.lv.items():
            W = self.prim(L.U)
            c = torch.sqrt(self.g * W[4] / W[0])
            v = (W[1:4].abs() + c).sum(0)[L.ex & ~L.split]
            if v.numel():
                out = min(out, self.cfl * 2.0 ** -l / float(v.max()) * 2.0 ** (l - self.lmin))
        return out

    def advance(self, n, regrid=None):
        dts = []
        for _ in range(n):
            if regrid:
                self.regrid(regrid)
            dt = self.dt()
            for l in _w_cycle(list(self.lv)):
                self.step(l, dt * 0.5 ** (l - self.lmin))
            dts.append(dt)
        return dts

    def regrid(self, thr):
        flag = {}
        for l, L in self.lv.items():
            W = self.prim(self.full(l))[[0, 4]]
            f = torch.zeros_like(L.ex)
            for ax in (1, 2, 3):
                for s in (1, -1):
                    b = torch.roll(W, s, ax)
                    f |= (2 * (W - b).abs() > thr * (W.abs() + b.abs())).any(0)
            f = self.widen(f & L.ex) & L.ex
            flag[l] = f if l < self.lmax else torch.zeros_like(f)
        for l in sorted(flag, reverse=True):
            if l == self.lmin or not bool(flag[l].any()):
                continue
            C, L = self.lv[l - 1], self.lv[l]
            w = self.widen(flag[l])
            need = w[::2, ::2, ::2].clone()
            for cz, cy, cx in itertools.product(range(2), range(2), range(2)):
                need |= w[cz::2, cy::2, cx::2]
            iz, iy, ix = C.into(L, 2)
            flag[l - 1].view(-1)[((iz * C.n[1] + iy) * C.n[0] + ix)[need]] = True
        old, octs = self.lv, {self.lmin: self.lv[self.lmin].octs}
        for l in range(self.lmin, self.lmax):
            if l not in old:
                break
            f = flag[l] & old[l].ex
            if not bool(f.any()):
                break
            z, y, x = [t.cpu().numpy() for t in torch.nonzero(f, as_tuple=True)]
            x, y, z = [(t + lo) % old[l].side for t, lo in zip((x, y, z), old[l].lo)]
            o = np.argsort(hilbert(x, y, z, l))
            octs[l + 1] = (x[o], y[o], z[o])
        self.build(octs)
        for l, L in self.lv.items():
            if l == self.lmin:
                L.U = old[l].U
                continue
            L.U = torch.where(L.ex, self.children(l), L.U)
            if l in old:
                i, j, k = [np.asarray(t, np.int64) for t in old[l].octs]
                c = np.arange(8)
                xyz = [(2 * t[:, None] + b[None, :]).ravel() for t, b in
                       ((i, c & 1), (j, (c >> 1) & 1), (k, (c >> 2) & 1))]
                inside = np.ones(xyz[0].shape, bool)
                for t, lo, n in zip(xyz, L.lo, L.n):
                    inside &= (t - lo) % L.side < n
                at = torch.from_numpy(L.index(*[t[inside] for t in xyz])).to(DEV)
                src = old[l].get()[:, torch.from_numpy(inside).to(DEV)]
                keep = L.ex.view(-1)[at]
                L.U.view(5, -1)[:, at[keep]] = src[:, keep]
        for l in sorted(self.lv, reverse=True)[:-1]:
            C, L = self.lv[l - 1], self.lv[l]
            iz, iy, ix = C.into(L, 2)
            m = L.ex[::2, ::2, ::2]
            C.U.view(5, -1)[:, ((iz * C.n[1] + iy) * C.n[0] + ix)[m]] = _blocks_mean(L.U)[:, m]

    @staticmethod
    def widen(f):
        for ax in range(3):
            f = f | torch.roll(f, 1, ax) | torch.roll(f, -1, ax)
        return f

    def state(self):
        return torch.cat([L.get() for L in self.lv.values()], 1).cpu().numpy()


def _nbsum(p):
    s = None
    for ax in (2, 1, 0):
        t = torch.roll(p, 1, ax) + torch.roll(p, -1, ax)
        s = t if s is None else s + t
    return s


def _prolonged(ec, n):
    """Trilinear prolongation (weights 27, 9, 3, 1 over 64)."""
    for ax in range(3):
        a, b = torch.roll(ec, 1, ax), torch.roll(ec, -1, ax)
        ec = torch.stack([0.75 * ec + 0.25 * a, 0.75 * ec + 0.25 * b], ax + 1).flatten(ax, ax + 1)
    return ec


def _parity(n):
    a = torch.arange(n, device=DEV)
    return (a[:, None, None] + a[None, :, None] + a[None, None, :]) & 1


def _v_cycle(e, f, dx, masks, nbnd, bs, k, bottom):
    """One V-cycle on MG level k, in place; masks None: the periodic box."""
    n = e.shape[0]
    par = _parity(n)
    diag = 6.0 if masks is None else (6 + nbnd[k]).to(F64)

    def sweeps(q):
        for _ in range(q):
            for colour in (0, 1):
                new = (_nbsum(e) + (bs if k == 0 else 0.0) - dx * dx * f) / diag
                m = par == colour
                e.copy_(torch.where(m if masks is None else m & masks[k], new, e))
    if k == bottom:
        sweeps(8)
        return
    sweeps(2)
    r = f - (_nbsum(e) + (bs if k == 0 else 0.0) - diag * e) / (dx * dx)
    if masks is not None:
        r = torch.where(masks[k], r, torch.zeros_like(r))
    fc = _blocks_mean(r)
    ec = torch.zeros_like(fc)
    _v_cycle(ec, fc, 2 * dx, masks, nbnd, bs, k + 1, bottom)
    up = _prolonged(ec, n)
    e += up if masks is None else torch.where(masks[k], up, torch.zeros_like(up))
    sweeps(2)


def _gravity(case, p, U):
    box = {}
    at = 0
    for l in range(p.levelmin, int(p.level.max()) + 1):
        s = p.level == l
        n = 1 << l
        c = np.arange(8)
        x, y, z = [(2 * t[s].astype(np.int64)[:, None] + b[None, :]).ravel()
                   for t, b in ((p.i, c & 1), (p.j, (c >> 1) & 1), (p.k, (c >> 2) & 1))]
        ix = torch.from_numpy((z * n + y) * n + x).to(DEV)
        rho = torch.zeros(n ** 3, dtype=F64, device=DEV)
        rho[ix] = torch.from_numpy(U[0, at:at + ix.numel()]).to(DEV)
        ex = torch.zeros(n ** 3, dtype=torch.bool, device=DEV)
        ex[ix] = True
        box[l] = (ix, rho.view(n, n, n), ex.view(n, n, n))
        at += ix.numel()
    l0 = p.levelmin
    mean = box[l0][1].mean()
    f = box[l0][1] - mean
    phi = {l0: torch.zeros_like(f)}
    for _ in range(case["cycles"]):
        _v_cycle(phi[l0], f, 2.0 ** -l0, None, None, 0.0, 0, l0 - 1)
    phi[l0] -= phi[l0].mean()
    out = [phi[l0].view(-1)[box[l0][0]].cpu().numpy()]
    if not case["levels"]:
        return out[0]
    for l in list(box)[1:]:
        _, rho, ex = box[l]
        up = phi[l - 1]
        for ax in range(3):
            up = up.repeat_interleave(2, ax)
        # the coarser potential where it exists at level l-1; boundary faces always see such a cell
        masks, nbnd = [ex], []
        for k in range(1, l - l0 + 1):
            m = masks[-1]
            masks.append(m.view(m.shape[0] // 2, 2, m.shape[1] // 2, 2, m.shape[2] // 2, 2).any(5).any(3).any(1))
        for m in masks:
            nbnd.append(6 - sum(torch.roll(m, s, ax).int() for ax in range(3) for s in (1, -1)))
        bs = torch.zeros_like(rho)
        for ax in range(3):
            for s in (1, -1):
                bs += torch.where(torch.roll(ex, s, ax), torch.zeros_like(up), up + torch.roll(up, s, ax))
        e = torch.where(ex, up, torch.zeros_like(up))
        f = rho - mean
        for _ in range(case["cycles"]):
            _v_cycle(e, f, 2.0 ** -l, masks, nbnd, bs, 0, l - l0)
        phi[l] = e
        out.append(e.view(-1)[box[l][0]].cpu().numpy())
    return out


def _cic(n, x, y, z, m):
    """Cloud-in-Cell density on a periodic n^3 grid, flat (x fastest)."""
    rho = torch.zeros(n ** 3, dtype=F64, device=DEV)
    i, w = [], []
    for t in (x, y, z):
        s = t * n - 0.5
        fl = torch.floor(s)
        i.append(fl.to(torch.int64))
        w.append((1.0 - (s - fl), s - fl))
    for c in range(8):
        b = (c & 1, (c >> 1) & 1, c >> 2)
        q = [(i[d] + b[d]) % n for d in range(3)]
        rho.index_add_(0, q[0] + n * (q[1] + n * q[2]), m * w[0][b[0]] * w[1][b[1]] * w[2][b[2]] * float(n) ** 3)
    return rho


def exact(case, seed):
    kind = case["kind"]
    if kind in ("deposit", "levels"):
        ps = _particles(case, seed)
        x, y, z, m = [torch.from_numpy(a).to(DEV) for a in ps.args()[1:]]
        if case["precision"] == 4:  # the positions that the framework is given or keeps
            x, y, z, m = [t.float().double() for t in (x, y, z, m)]
        if kind == "deposit":
            return _cic(case["grid"], x, y, z, m)
        p = _mesh_of(case)
        counts, out = np.zeros(16, np.int64), []
        top = int(p.level.max())
        for l in range(p.levelmin, top + 1):
            counts[l] = x.numel()
            s, n = p.level == l, 1 << l
            c = np.arange(8)
            q = [torch.from_numpy((2 * t[s].astype(np.int64)[:, None] + b[None, :]).ravel()).to(DEV)
                 for t, b in ((p.i, c & 1), (p.j, (c >> 1) & 1), (p.k, (c >> 2) & 1))]
            out.append(_cic(n, x, y, z, m)[q[0] + n * (q[1] + n * q[2])].cpu().numpy())
            if l < top:  # the next list: particles whose cell here is split
                fin = p.level == l + 1
                sp = torch.zeros(n ** 3, dtype=torch.bool, device=DEV)
                k = [torch.from_numpy(t[fin].astype(np.int64)).to(DEV) for t in (p.i, p.j, p.k)]
                sp[k[0] + n * (k[1] + n * k[2])] = True
                h = [torch.floor(t * n).to(torch.int64) for t in (x, y, z)]
                keep = sp[h[0] + n * (h[1] + n * h[2])]
                x, y, z, m = [t[keep] for t in (x, y, z, m)]
        return counts, out
    p = _mesh_of(case)
    if kind == "gravity":
        U = _state(p, seed * 1000)
        return _gravity(case, p, U.astype(np.float32).astype(np.float64) if case["precision"] == 4 else U)
    if kind == "adaptive":
        a = _Amr(p, _state(p, seed))
        a.advance(case["steps"], regrid=0.1)
        out = {}
        for l, L in a.lv.items():
            i, j, k = [np.asarray(t, np.int64) for t in L.octs]
            key = (np.uint64(l) << np.uint64(60)) | ((i << 40) | (j << 20) | k).astype(np.uint64)
            out[l] = (key, L.get().cpu().numpy())
        return out
    outs, dts = [], []
    for q in range(case.get("members", 1)):
        a = _Amr(p, _state(p, seed * 1000 + q))
        dts = a.advance(case["steps"])
        outs.append(a.state())
    return outs + (dts if kind == "substeps" else [])
