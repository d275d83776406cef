"""Performance cases of the nested-mesh solver: what its users' programs run.

Three forms, all through the public binding (ctypes over the C ABI):

* ``run``: one hierarchy (a context).  A pass advances it some coarse steps, reads the
  force on the perturber and the simulated time, and reads every field of every level
  into pinned host memory.
* ``pool``: many independent hierarchies stepped together, read the same way; with
  ``batches`` > 1 the pass steps in batches and reads every run's force history after
  each, as the request server does.
* ``operators``: what a restart does around the stepping: load a checkpoint, fill the
  boundaries, CommUp and CommMean on every level, the time step, the force, and the
  whole padded arrays back.

Inputs: the uniform wind of the workloads plus a smooth seeded perturbation of all five
fields (1 % amplitude), a function of position, so that the levels agree where they
overlap.  Results of the FP32 state are returned as float32, of the FP64 state as
float64.  ``exact`` is the same scheme in plain torch float64 over whole padded arrays.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_1812_03191_gb300 import binding, inputs

FIELDS = ("rho", "e", "vx", "vy", "vz")
AMP = 1e-2
FLOPS_PER_CELL = 600  # plain arithmetic of one level step per cell (three sweeps, two kicks)


def _run(name, precision, levels, nx, ny, nz, half, mach, steps, chi=1.0, lum=True, search=False):
    return dict(name=name, form="run", precision=precision, levels=levels, nx=nx, ny=ny, nz=nz,
                half=half, mach=mach, chi=chi, lum=lum, search=search, quadrant=False, steps=steps)


def _quadrant(name, precision, levels, n, steps):
    """The paper's low-Mach hierarchy: quadrant levels of n/2 x n/2 x n cells under a
    ground of n x n x 2n, half-width 3200 lambda at chi = 0.1, Mach 0.1, no luminosity."""
    return dict(name=name, form="run", precision=precision, levels=levels, nx=n // 2, ny=n // 2,
                nz=n, half=2286.0, mach=0.1, chi=0.1, lum=False, search=False, quadrant=True,
                steps=steps)


def _pool(name, precision, runs, small, large, min_levels, max_levels, shapes, batches, steps):
    return dict(name=name, form="pool", precision=precision, runs=runs, small=small, large=large,
                min_levels=min_levels, max_levels=max_levels, shapes=shapes, batches=batches,
                steps=steps)


def listed():
    return [
        # the smallest hierarchy of the workloads, 20 coarse steps: launch latency
        _run("single_32_fp64", "fp64", 1, 32, 32, 32, 4.0, 0.5, 20, lum=False),
        # a restart's operators on a small hierarchy: single calls, each with its set-up
        dict(name="operators_32_fp64", form="operators", precision="fp64", levels=3, nx=32, ny=32,
             nz=32, half=8.0, mach=0.5, chi=1.0, lum=True, search=False, quadrant=False, steps=0),
        # the benchmarked nested workload in both precisions
        _run("nested_64_fp64", "fp64", 3, 64, 64, 64, 8.0, 0.5, 20),
        _run("nested_64_fp32", "fp32", 3, 64, 64, 64, 8.0, 0.5, 20),
        # unequal sides, none a multiple of a block, and the Eq. 55-56 sub-cycling search
        _run("ragged_search_fp64", "fp64", 4, 44, 60, 36, 8.0, 1.2, 10, chi=0.3, search=True),
        # a hierarchy between the small and the large one
        _run("nested_96_fp32", "fp32", 3, 96, 96, 96, 8.0, 0.8, 10),
        # the largest hierarchy of the workloads (the default bench line), both precisions
        _run("precision_128_fp64", "fp64", 5, 128, 128, 128, 16.0, 1.2, 4),
        _run("precision_128_fp32", "fp32", 5, 128, 128, 128, 16.0, 1.2, 10),
        # the paper's own geometry: thousands of small boxes per coarse step
        _quadrant("quadrant_9_fp64", "fp64", 9, 64, 1),
        _quadrant("quadrant_9_fp32", "fp32", 9, 64, 1),
        # uneven runs in one pool, and a server's pool of small requests read every 8 steps
        _pool("pool_uneven_fp32", "fp32", 24, 32, 96, 2, 4, 1812031910, 1, 4),
        _pool("pool_serving_fp32", "fp32", 16, 24, 32, 2, 3, 1812031911, 4, 8),
    ]


def _log_between(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _four(x):
    return max(4, 4 * round(x / 4))


def draw(rng):
    """One more case of the listed ones' ranges; mesh sides are multiples of 4."""
    kind = rng.choice(("run", "run", "run", "quadrant", "pool", "operators"))
    precision = rng.choice(("fp64", "fp32"))
    if kind == "quadrant":
        c = _quadrant("", precision, rng.randint(6, 9), rng.choice((48, 56, 64)), 1)
    elif kind == "pool":
        small = _four(_log_between(rng, 24, 48))
        c = _pool("", precision, rng.randint(3, 16), small, _four(_log_between(rng, small, 80)), 2,
                  rng.randint(2, 3), rng.randrange(1 << 30), rng.randint(1, 4), rng.randint(1, 4))
    else:
        levels = rng.randint(1, 5) if kind == "run" else rng.randint(2, 4)
        top = 128 if kind == "run" and levels < 5 else 64
        n = [_four(_log_between(rng, 24, top)) for _ in range(3)]
        cells = n[0] * n[1] * n[2] * (2 ** levels - 1)
        steps = max(1, min(20, int(6e7 / cells))) if kind == "run" else 0
        c = _run("", precision, levels, n[0], n[1], n[2], rng.choice((4.0, 8.0, 16.0)),
                 _log_between(rng, 0.1, 3.0), steps, chi=_log_between(rng, 0.3, 3.0),
                 lum=rng.random() < 0.5, search=rng.random() < 0.25)
        c["form"] = kind
    del c["name"]
    return c


# ------------------------------------------------------------------ configurations


def _pool_shapes(case):
    """(levels, n, mach, chi, lum) of each run of a pool, from the case alone."""
    rng = random.Random(case["shapes"])
    out = []
    for _ in range(case["runs"]):
        n = _four(_log_between(rng, case["small"], case["large"]))
        out.append((rng.randint(case["min_levels"], case["max_levels"]), n,
                    _log_between(rng, 0.1, 3.0), _log_between(rng, 0.3, 3.0), rng.random() < 0.5))
    return out


def _config(levels, n, half, mach, chi, lum, search=False, quadrant=False):
    """Geometry and parameters of one hierarchy."""
    if quadrant:
        cfg = inputs.quadrant(n=n[2], n_levels=levels, half=half, mach=mach, quarter=True,
                              GM=1e-3, chi=chi)
        return dict(cfg, levels=levels)
    halves = [half * m / n[0] for m in n]
    eps = 2 * (2 * half / n[0] / 2 ** (levels - 1))
    L = inputs.critical_luminosity(0.01, 1.0, chi, 5.0 / 3.0) if lum else 0.0
    p = inputs.base_params(mach=mach, chi=chi, eps=eps, L=L, lum_sigma=eps if lum else 0.0,
                           xi_mode=int(search))
    return dict(levels=levels, n=tuple(n), n0=tuple(n), lo=tuple(-h for h in halves),
                hi=tuple(halves), G=inputs.DEFAULT_G, params=p)


def _configs(case):
    if case["form"] == "pool":
        return [_config(nl, (n,) * 3, 8.0, mach, chi, lum)
                for nl, n, mach, chi, lum in _pool_shapes(case)]
    return [_config(case["levels"], (case["nx"], case["ny"], case["nz"]), case["half"],
                    case["mach"], case["chi"], case["lum"], case["search"], case["quadrant"])]


def _level(cfg, l):
    """cells, lower corner and cell size of level l"""
    n = cfg["n0"] if l == 0 else cfg["n"]
    sc = [n[d] / cfg["n0"][d] * 2.0 ** -l for d in range(3)]
    lo = [cfg["lo"][d] * sc[d] for d in range(3)]
    return n, lo, [(cfg["hi"][d] - cfg["lo"][d]) * sc[d] / n[d] for d in range(3)]


def _background(p):
    e0 = p["cs"] ** 2 * p["rho0"] / (p["gamma"] * (p["gamma"] - 1.0))
    return [p["rho0"], e0] + [p["mach"] * p["cs"] * x for x in p["flow_dir"]]


def _initial(cfg, seed, device):
    """[level][field]: the wind plus a sum of separable long waves of the box, even
    (odd for the normal velocity) across mirror planes; active cells, (nz, ny, nx)."""
    rng = np.random.default_rng(seed)
    mirror = [cfg["lo"][d] == 0.0 for d in range(3)]
    bg, out = _background(cfg["params"]), []
    waves = [[(rng.uniform(-1, 1), rng.integers(0, 3, 3), rng.uniform(0, 2 * math.pi, 3))
              for _ in range(4)] for _ in FIELDS]
    for l in range(cfg["levels"]):
        n, lo, dx = _level(cfg, l)
        fields = []
        for f in range(5):
            q = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device=device)
            for a, k, ph in waves[f]:
                line = []
                for d in range(3):
                    x = lo[d] + (torch.arange(n[d], dtype=torch.float64, device=device)
                                 + (0.0 if f == 2 + d else 0.5)) * dx[d]
                    x = x * (math.pi * float(k[d]) / cfg["hi"][d])
                    odd = mirror[d] and f == 2 + d
                    line.append(torch.sin(x) if odd else
                                torch.cos(x) if mirror[d] else torch.cos(x + float(ph[d])))
                q += a * AMP / 4 * line[2][:, None, None] * line[1][:, None] * line[0]
            fields.append(bg[f] + q)
        out.append(fields)
    return out


# --------------------------------------------------------------------- the passes


def _doubles(t, at=0):
    return ctypes.cast(t.data_ptr() + 8 * at, ctypes.POINTER(ctypes.c_double))


def _precision(case):
    return binding.DF_FP64 if case["precision"] == "fp64" else binding.DF_FP32_STATE


class State:
    """A program's handle, its pinned buffers and, for the FP32 state, their float32
    copies."""

    def __init__(self, case, cfgs, total):
        self.case, self.cfgs = case, cfgs
        self.pinned = [torch.empty(total, dtype=torch.float64, pin_memory=True) for _ in FIELDS]
        self.single = case["precision"] == "fp32"
        self.out = [torch.empty(total, dtype=torch.float32) for _ in FIELDS] if self.single \
            else self.pinned

    def results(self, **scalars):
        if self.single:
            for a, b in zip(self.out, self.pinned):
                a.copy_(b)
        kind = np.float32 if self.single else np.float64
        return dict(zip(FIELDS, self.out), **{k: np.asarray(v, kind) for k, v in scalars.items()})


def prepare(case, seed):
    cfgs = _configs(case)
    stream = torch.cuda.current_stream().cuda_stream
    if case["form"] == "pool":
        total = sum(c["levels"] * math.prod(c["n"]) for c in cfgs)
        s = State(case, cfgs, total)
        s.pool = binding.Pool(64 << 30, precision=_precision(case), stream=stream)
        s.slots = []
        for r, c in enumerate(cfgs):
            s.slots.append(s.pool.admit(c["levels"], c["n"], c["lo"], c["hi"], c["G"],
                                        c["params"]))
            for l, fields in enumerate(_initial(c, [seed, r], "cuda")):
                for f, q in enumerate(fields):
                    s.pool.set_field(s.slots[r], l, f, q.cpu().numpy())
        return s
    c = cfgs[0]
    pad = 2 * c["G"] if case["form"] == "operators" else 0
    total = sum(math.prod(m + pad for m in _level(c, l)[0]) for l in range(c["levels"]))
    s = State(case, cfgs, total)
    s.sim = binding.Sim(c["levels"], c["n"], c["lo"], c["hi"], c["G"], c["params"],
                        precision=_precision(case), stream=stream, n0=c["n0"])
    for l, fields in enumerate(_initial(c, [seed], "cuda")):
        for f, q in enumerate(fields):
            s.sim.set_field(l, f, q.cpu().numpy())
    if case["form"] == "operators":
        s.checkpoint = torch.empty(s.sim.state_size(), dtype=torch.float64, pin_memory=True)
        s.sim.get_state(s.checkpoint.numpy())
    else:
        for l in range(c["levels"] - 1):
            s.sim.prolong(l)
    return s


def run(s):
    if s.case["form"] == "pool":
        return _run_pool(s)
    if s.case["form"] == "operators":
        return _run_operators(s)
    sim, at = s.sim, 0
    t = sim.step(s.case["steps"], want_t=True)
    force, _ = sim.force()
    for l in range(sim.n_levels):
        for f in range(5):
            binding._check(sim.lib.df_get_field(sim.h, l, f, _doubles(s.pinned[f], at)))
        at += math.prod(sim.level_n(l))
    return s.results(force=force, t=t)


def _run_pool(s):
    pool, at, history = s.pool, 0, []
    for _ in range(s.case["batches"]):
        pool.step(s.case["steps"])
        history += [pool.history(slot, s.case["steps"]) for slot in s.slots]
    for slot, c in zip(s.slots, s.cfgs):
        for l in range(c["levels"]):
            for f in range(5):
                binding._check(pool.lib.df_pool_get_field(pool.h, slot, l, f,
                                                          _doubles(s.pinned[f], at)))
            at += math.prod(c["n"])
    history = np.stack(history)
    return s.results(force=history[:, :, :3], t=history[:, :, 3])


def _run_operators(s):
    sim, at = s.sim, 0
    sim.set_state(s.checkpoint.numpy(), 0.0)
    sim.fill_bc()
    for l in range(sim.n_levels - 1):
        sim.prolong(l)
    for l in reversed(range(sim.n_levels - 1)):
        sim.restrict(l)
    dt, dt_level = sim.compute_dt()
    force = sim.force_now()
    for l in range(sim.n_levels):
        for f in range(5):
            binding._check(sim.lib.df_get_full(sim.h, l, f, _doubles(s.pinned[f], at)))
        at += math.prod(sim.full_shape(l))
    return s.results(force=force, dt=dt, dt_level=dt_level)


def work(case):
    """The five fields of every cell read and written once per level step (once for the
    operators), as stored."""
    size = 8 if case["precision"] == "fp64" else 4
    cells = 0
    for c in _configs(case):
        for l in range(c["levels"]):
            n = math.prod(_level(c, l)[0])
            cells += n if case["form"] == "operators" else n * 2 ** l
    if case["form"] == "operators":
        return {"bytes": 10 * size * cells, "flops": 30 * cells}
    cells *= case["steps"] * case.get("batches", 1)
    return {"bytes": 10 * size * cells, "flops": FLOPS_PER_CELL * cells}


# ------------------------------------------------ the same scheme in torch float64


def _cut(q, d, at, n):
    """q[at : at + n] along axis d (0 = x, the tensors' last dimension)"""
    return q.narrow(2 - d, at, n)


def _half_slope(dl, dr):
    """half the van Leer harmonic slope"""
    pr = dl * dr
    return torch.where(pr > 0, pr / torch.where(pr > 0, dl + dr, torch.ones_like(pr)),
                       torch.zeros_like(pr))


def _upwind(q, d, at, n, u, cour):
    """time-centred value of q at the faces at .. at + n - 1 along d"""
    mm, m, c, p = (_cut(q, d, at + o, n) for o in (-2, -1, 0, 1))
    up = u > 0
    a = torch.where(up, m, c)
    dl = a - torch.where(up, mm, m)
    dr = torch.where(up, c, p) - a
    return a + (torch.where(up, 1.0, -1.0) - cour) * _half_slope(dl, dr)


class _Level:
    pass


class _Hierarchy:
    """One run, every operator over the whole padded arrays."""

    def __init__(self, cfg, init, device):
        self.p, self.G, self.nl = cfg["params"], cfg["G"], cfg["levels"]
        p, G = self.p, self.G
        self.bg = _background(p)
        self.mirror = [cfg["lo"][d] == 0.0 and p["bc"][2 * d] == inputs.BC_REFLECT
                       for d in range(3)]
        self.mult = 2.0 ** sum(self.mirror)
        self.t, self.L = 0.0, []
        for l in range(self.nl):
            v = _Level()
            v.n, v.lo, v.dx = _level(cfg, l)
            v.s = [m + 2 * G for m in v.n]
            v.vol = math.prod(v.dx)
            v.q = []
            for f in range(5):
                q = torch.full(v.s[::-1], self.bg[f], dtype=torch.float64, device=device)
                self.act(v, q).copy_(init[l][f])
                v.q.append(q)
            x = [v.lo[d] + (torch.arange(v.s[d], dtype=torch.float64, device=device) - G + 0.5)
                 * v.dx[d] for d in range(3)]
            r2 = x[2][:, None, None] ** 2 + x[1][:, None] ** 2 + x[0] ** 2
            soft = r2 + p["eps"] ** 2
            v.phi = -p["GM"] / torch.sqrt(soft)
            w = p["GM"] * v.vol / soft ** 1.5
            shape = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]
            v.fw = [self.act(v, w * x[d].view(shape[d])) * (0.0 if self.mirror[d] else self.mult)
                    for d in range(3)]
            v.lum = torch.zeros_like(v.phi)
            if p["L"] != 0.0:  # Gaussian, over the whole domain (no mirror planes)
                g = torch.exp(-r2 / (2 * p["lum_sigma"] ** 2))
                a = self.act(v, g)
                self.act(v, v.lum).copy_(a / (a.sum() * v.vol))
            if l > 0:
                c = self.L[l - 1]
                v.off = [round((v.lo[d] - c.lo[d]) / c.dx[d]) for d in range(3)]
                c.child = v
                v.covered = tuple(slice(v.off[d], v.off[d] + v.n[d] // 2) for d in (2, 1, 0))
                for w in c.fw:
                    w[v.covered] = 0.0
            v.child = None
            self.L.append(v)

    def act(self, v, q):
        return q[tuple(slice(self.G, self.G + v.n[d]) for d in (2, 1, 0))]

    # boundary fill along one axis
    def fill(self, v, d, lo, hi):
        G, n = self.G, v.n[d]
        for f, q in enumerate(v.q):
            normal = f == 2 + d
            for side, kind in ((0, lo), (1, hi)):
                ghost = _cut(q, d, 0, G) if side == 0 else _cut(q, d, G + n, G)
                if kind == inputs.BC_OUTFLOW:
                    if normal and side == 1:
                        _cut(q, d, G + n + 1, G - 1).copy_(
                            _cut(q, d, G + n, 1).expand_as(_cut(q, d, G + n + 1, G - 1)))
                    else:
                        ghost.copy_(_cut(q, d, G if side == 0 else G + n - 1, 1).expand_as(ghost))
                elif kind == inputs.BC_INFLOW:
                    ghost.fill_(self.bg[f])
                    if normal and side == 0:
                        _cut(q, d, G, 1).fill_(self.bg[f])
                elif kind == inputs.BC_REFLECT:
                    if not normal:
                        src = _cut(q, d, G if side == 0 else n, G)
                        ghost.copy_(src.flip(2 - d))
                    elif side == 0:
                        ghost.copy_(-_cut(q, d, G + 1, G).flip(2 - d))
                        _cut(q, d, G, 1).fill_(0.0)
                    else:
                        _cut(q, d, G + n + 1, G - 1).copy_(
                            -_cut(q, d, n + 1, G - 1).flip(2 - d))
                        _cut(q, d, G + n, 1).fill_(0.0)

    def mirror_fill(self, v):
        for d in range(3):
            if self.mirror[d]:
                self.fill(v, d, inputs.BC_REFLECT, None)

    def commup(self, v):
        """every element of the child that is not its own, from the level v"""
        self.mirror_fill(v)
        c, G = v.child, self.G
        for f in range(5):
            q = v.q[f]
            for d in range(3):
                q = _cut(q, d, G + c.off[d] - G // 2 - 1, c.n[d] // 2 + G + 2)
            for d in (2, 1, 0):
                n = q.shape[2 - d] - 2
                m, o, p = (_cut(q, d, k, n) for k in range(3))
                if f == 2 + d:
                    pair = (o, 0.5 * (o + p))
                else:
                    h = 0.5 * _half_slope(o - m, p - o)
                    pair = (o - h, o + h)
                q = torch.stack(pair, dim=3 - d).flatten(2 - d, 3 - d)
            own = tuple(slice(G + (f == 2 + d), G + c.n[d]) for d in (2, 1, 0))
            q[own] = c.q[f][own]
            c.q[f] = q

    def commmean(self, v):
        c, G, band = v.child, self.G, self.p["band"]
        h = [m // 2 for m in c.n]
        device = v.phi.device
        dist = torch.full(h[::-1], 1 << 30, device=device)
        for d in range(3):
            a = torch.arange(h[d], device=device)
            far = h[d] - 1 - a if self.mirror[d] else torch.minimum(a, h[d] - 1 - a)
            dist = torch.minimum(dist, far.view([-1 if k == d else 1 for k in (2, 1, 0)]))
        band = dist < band
        for f in range(5):
            fine = self.act(c, c.q[f])
            coarse = self.act(v, v.q[f])[c.covered]
            use = band
            if f >= 2:
                d = f - 2
                use = band.clone()
                _cut(use, d, 1, h[d] - 1).logical_or_(_cut(band, d, 0, h[d] - 1))
                _cut(use, d, 0, 1).fill_(False)
            for k in range(3):
                even = [slice(None)] * 3
                even[2 - k] = slice(0, None, 2)
                odd = list(even)
                odd[2 - k] = slice(1, None, 2)
                fine = fine[tuple(even)] if f == 2 + k else \
                    0.5 * (fine[tuple(even)] + fine[tuple(odd)])
            coarse.copy_(torch.where(use, fine, coarse))

    # frontier fluxes: a child's through its faces, summed per coarse face, and the
    # parent's substitute for its own
    def record(self, v, d, flux, first):
        """sums of a flux array (first: index of its first face along d)"""
        out = []
        for side in range(2):
            a = _cut(flux, d, self.G + side * v.n[d] - first, 1)
            for k in range(3):
                if k != d:
                    a = _cut(a, k, self.G, v.n[k]) if a.shape[2 - k] == v.s[k] else \
                        _cut(a, k, self.G - 1, v.n[k])
                    at = [slice(None)] * 3
                    at[2 - k] = slice(0, None, 2)
                    even = a[tuple(at)]
                    at[2 - k] = slice(1, None, 2)
                    a = even + a[tuple(at)]
            out.append(a)
        return out

    def substitute(self, v, d, flux, sums, first, trim=0):
        """the child's sums in place of the parent's frontier fluxes"""
        G, c = self.G, v.child
        flux = flux.clone()
        for side in range(2):
            if side == 0 and self.mirror[d]:
                continue
            a, at = sums[side], [None] * 3
            face = G + c.off[d] + side * (c.n[d] // 2) - first
            at[2 - d] = slice(face, face + 1)
            for k in range(3):
                if k == d:
                    continue
                lo, n = G + c.off[k] - trim, c.n[k] // 2
                if self.mirror[k]:  # ghost faces across the plane take their image's sum
                    g = min(lo, n)
                    a = torch.cat((_cut(a, k, 0, g).flip(2 - k), a), dim=2 - k)
                    lo, n = lo - g, n + g
                at[2 - k] = slice(lo, lo + n)
            flux[tuple(at)] = a
        return flux

    def kick(self, v, h):
        """v_d -= h [(p_c - p_m) / (dx rho_face) + (Phi_c - Phi_m) / dx]"""
        for d in range(3):
            n = v.s[d] - 1
            rho, e, phi = ((_cut(q, d, 0, n), _cut(q, d, 1, n)) for q in (v.q[0], v.q[1], v.phi))
            acc = (self.p["gamma"] - 1) * (e[1] - e[0]) / (0.5 * (rho[0] + rho[1]))
            _cut(v.q[2 + d], d, 1, n).sub_(h / v.dx[d] * (acc + phi[1] - phi[0]))

    def level_step(self, l, dt, record):
        """one step of level l; record: this level's frontier sums as a child, [d][q]"""
        v, p = self.L[l], self.p
        rho, e = v.q[0], v.q[1]
        sums = v.sums if v.child is not None else None
        if l == 0:
            for d in range(3):
                self.fill(v, d, p["bc"][2 * d], p["bc"][2 * d + 1])
        else:
            self.mirror_fill(v)
        self.kick(v, 0.5 * dt)
        pi = []
        for d in range(3):
            m = torch.zeros_like(rho)
            n = v.s[d] - 1
            _cut(m, d, 1, n).copy_(0.5 * (_cut(rho, d, 0, n) + _cut(rho, d, 1, n))
                                   * _cut(v.q[2 + d], d, 1, n))
            pi.append(m)
        # compression heating, luminosity
        inner = tuple(slice(0, v.s[d] - 1) for d in (2, 1, 0))
        div = 0.0
        for d in range(3):
            w = v.q[2 + d]
            k = (_cut(w, d, 1, v.s[d] - 1) - _cut(w, d, 0, v.s[d] - 1)) / v.dx[d]
            for o in range(3):
                if o != d:
                    k = _cut(k, o, 0, v.s[o] - 1)
            div = div + k
        a = 0.5 * dt * (p["gamma"] - 1) * div
        e[inner] *= (1 - a) / (1 + a)
        if p["L"] != 0.0:
            e += p["L"] * dt * v.lum
        # thermal diffusion, fluxes between the inner cells' faces
        if p["chi"] > 0.0:
            eps = e / rho
            tot = 0.0
            for d in range(3):
                n = v.s[d] - 1
                k = -p["chi"] * dt * v.vol / v.dx[d] ** 2
                r = 0.5 * (_cut(rho, d, 0, n) + _cut(rho, d, 1, n))
                flux = k * r * (_cut(eps, d, 1, n) - _cut(eps, d, 0, n))  # faces 1 ..
                for o in range(3):
                    if o != d:
                        flux = _cut(flux, o, 1, v.s[o] - 2)
                if l > 0:
                    record[d][2].append(self.record(v, d, flux, 1))
                if sums is not None:
                    flux = self.substitute(v, d, flux, sums[d][2], 1, trim=1)
                tot = tot + _cut(flux, d, 1, v.s[d] - 2) - _cut(flux, d, 0, v.s[d] - 2)
            e[1:-1, 1:-1, 1:-1] -= tot / v.vol
        for d in range(3):
            self.sweep(v, l, d, dt, pi, record, sums)
        for d in range(3):
            n = v.s[d] - 1
            _cut(v.q[2 + d], d, 1, n).copy_(
                _cut(pi[d], d, 1, n) / (0.5 * (_cut(rho, d, 0, n) + _cut(rho, d, 1, n))))
        self.kick(v, 0.5 * dt)

    def sweep(self, v, l, d, dt, pi, record, sums):
        rho, e, u = v.q[0], v.q[1], v.q[2 + d]
        s, k = v.s[d], dt / v.dx[d]
        area = v.vol / v.dx[d]
        eps, w = e / rho, []
        for m in range(3):
            x = torch.zeros_like(rho)
            n = v.s[m] - 1
            _cut(x, m, 1, n).copy_(_cut(pi[m], m, 1, n)
                                   / (0.5 * (_cut(rho, m, 0, n) + _cut(rho, m, 1, n))))
            w.append(x)
        n = s - 3  # faces 2 .. s - 2
        uf = _cut(u, d, 2, n)
        F = _upwind(rho, d, 2, n, uf, uf * k) * uf * (area * dt)
        E = _upwind(eps, d, 2, n, uf, uf * k) * F
        if l > 0:
            record[d][0].append(self.record(v, d, F, 2))
            record[d][1].append(self.record(v, d, E, 2))
        P = []
        for m in range(3):
            if m == d:  # cell-centred, cells 2 .. s - 3
                c = n - 1
                uc = 0.5 * (_cut(u, d, 2, c) + _cut(u, d, 3, c))
                P.append(_upwind(w[m], d, 3, c, uc, uc * k)
                         * 0.5 * (_cut(F, d, 0, c) + _cut(F, d, 1, c)))
            else:       # on the d-m edges, m index 1 ..
                c = v.s[m] - 1
                ue = 0.5 * (_cut(uf, m, 0, c) + _cut(uf, m, 1, c))
                P.append(_upwind(_cut(w[m], m, 1, c), d, 2, n, ue, ue * k)
                         * 0.5 * (_cut(F, m, 0, c) + _cut(F, m, 1, c)))
        if sums is not None:
            F = self.substitute(v, d, F, sums[d][0], 2)
            E = self.substitute(v, d, E, sums[d][1], 2)
        n = s - 4  # cells 2 .. s - 3
        _cut(rho, d, 2, n).sub_((_cut(F, d, 1, n) - _cut(F, d, 0, n)) / v.vol)
        _cut(e, d, 2, n).sub_((_cut(E, d, 1, n) - _cut(E, d, 0, n)) / v.vol)
        for m in range(3):
            if m == d:
                _cut(pi[m], d, 3, n - 1).sub_(
                    (_cut(P[m], d, 1, n - 1) - _cut(P[m], d, 0, n - 1)) / v.vol)
            else:
                _cut(_cut(pi[m], m, 1, v.s[m] - 1), d, 2, n).sub_(
                    (_cut(P[m], d, 1, n) - _cut(P[m], d, 0, n)) / v.vol)

    def time_step(self):
        """(dt, per-level limits, xi)"""
        p, limits = self.p, []
        for v in self.L:
            lim = math.inf
            if p["chi"] > 0.0:
                lim = p["cfl_diff"] / (2 * p["chi"] * sum(1 / x ** 2 for x in v.dx))
            rho, e = self.act(v, v.q[0]), self.act(v, v.q[1])
            cs = torch.sqrt(p["gamma"] * (p["gamma"] - 1) * e / rho)
            for d in range(3):
                a = self.act(v, v.q[2 + d]).abs()
                up = v.q[2 + d].roll(-1, 2 - d)
                top = (cs + torch.maximum(a, self.act(v, up).abs())).max().item()
                lim = min(lim, p["cfl"] * v.dx[d] / top)
            limits.append(lim)
        words = [(2,) * (self.nl - 1)]
        if p["xi_mode"] == 1:
            words = [tuple(2 if b >> m & 1 else 1 for m in range(self.nl - 1))
                     for b in range(1 << (self.nl - 1))]
        best = None
        for xi in words:
            dt, cost, pr = math.inf, 0.0, 1.0
            for l in range(self.nl):
                pr *= xi[l - 1] if l else 1
                dt = min(dt, limits[l] * pr)
                cost += math.prod(self.L[l].n) * pr
            if best is None or dt / cost > best[0]:
                best = (dt / cost, dt, xi)
        return best[1], limits, best[2]

    def advance(self, l, dt, xi, record):
        v = self.L[l]
        if v.child is not None:
            parts = [[[], [], []] for _ in range(3)]
            for _ in range(xi[l]):
                self.advance(l + 1, dt / xi[l], xi, parts)
            v.sums = [[[sum(x[side] for x in q) for side in range(2)] if q else None for q in d]
                      for d in parts]
        self.level_step(l, dt, record)
        if v.child is not None:
            self.commup(v)
            self.commmean(v)

    def step(self):
        dt, _, xi = self.time_step()
        self.advance(0, dt, xi, None)
        self.t += dt

    def force(self):
        return [sum(((self.act(v, v.q[0]) - self.bg[0]) * v.fw[d]).sum().item() for v in self.L)
                for d in range(3)]


def exact(case, seed):
    cfgs = _configs(case)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    steps = sum(2 ** c["levels"] - 1 for c in cfgs) * case["steps"] * case.get("batches", 1)
    if steps > 2500:  # about 6 ms each
        return None
    pool = case["form"] == "pool"
    fields, history = [[] for _ in FIELDS], []
    for r, c in enumerate(cfgs):
        h = _Hierarchy(c, _initial(c, [seed, r] if pool else [seed], device), device)
        if case["form"] == "operators":
            for d in range(3):
                h.fill(h.L[0], d, c["params"]["bc"][2 * d], c["params"]["bc"][2 * d + 1])
            for v in h.L[:-1]:
                h.commup(v)
            for v in reversed(h.L[:-1]):
                h.commmean(v)
            dt, limits, _ = h.time_step()
            for v in h.L:
                for f in range(5):
                    fields[f].append(v.q[f].reshape(-1).cpu())
            return dict(zip(FIELDS, (torch.cat(q) for q in fields)), force=np.array(h.force()),
                        dt=np.array(dt), dt_level=np.array(limits))
        if not pool:
            for v in h.L[:-1]:
                h.commup(v)
        past = []
        for _ in range(case["steps"] * case.get("batches", 1)):
            h.step()
            if pool:
                past.append(h.force() + [h.t])
        for v in h.L:
            for f in range(5):
                fields[f].append(h.act(v, v.q[f]).reshape(-1).cpu())
        history.append(past)
    out = dict(zip(FIELDS, (torch.cat(q) for q in fields)))
    if not pool:
        return dict(out, force=np.array(h.force()), t=np.array(h.t))
    # (run, batch, step) to the passes' order: batches of every run
    past = np.array(history).reshape(len(cfgs), case["batches"], case["steps"], 4)
    past = past.transpose(1, 0, 2, 3).reshape(-1, case["steps"], 4)
    return dict(out, force=past[:, :, :3], t=past[:, :, 3])
