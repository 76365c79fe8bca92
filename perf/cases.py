"""Performance cases: the limited lattice Boltzmann solves a user runs.

Every case goes through the public Python API (``lbm.Lattice``, ``lbm.Batch``,
``serve.Server``).  Four kinds of use:

* ``solve``: initial density and velocity in, a number of steps, the fields
  (and the populations, as a checkpoint) out: one whole solve of a small
  lattice, where latency and launches count;
* ``advance``: a resident lattice goes on by a number of steps and its fields
  or populations are read: how a large lattice is run between two outputs;
* ``reload``: populations in, a few steps, populations out: a restart from a
  state far from equilibrium, on which the limiters act everywhere;
* ``batch`` and ``serve``: many lattices of different sizes together, stepped
  as one batch or served as requests.

``exact`` repeats the same steps in FP64 with plain torch operations written
from the formulas of the paper (arXiv:0704.0043), without this repository's
code.
"""
import math
import random

import numpy as np
import torch

from paper_0704_0043_gb300 import inputs, lbm, serve

POS, EHR, MED, SMOOTH, THRESH, ENTTHR = 1, 2, 4, 8, 16, 32
PRECISION = {"fp64": lbm.FP64, "fp32": lbm.FP32, "bf16": lbm.BF16, "fp16": lbm.FP16}
ELEM = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}
STATS = ("step", "mass", "sum_dS", "dS_lbgk", "dS_lim", "n_pos", "n_med", "n_ehr", "n_cand", "n_bad", "status")
SUMS = ("mass", "sum_dS", "dS_lbgk", "dS_lim")

# the lattice sides of the batch of cavities and of the served requests come
# from these seeds: the shape of the work does not depend on the inputs' seed
BATCH_SEED, SERVE_SEED = 7040043, 7040044


def cavity(name, use, nx, ny, steps, limiters, precision="fp32", boundary=0, re=7500.0, u_lid=0.05, entropic=False,
           out="fields"):
    return {"name": name, "use": use, "lattice": "d2q9", "nx": nx, "ny": ny, "steps": steps, "limiters": limiters,
            "precision": precision, "boundary": boundary, "re": re, "u_lid": u_lid, "entropic": entropic, "out": out}


def tube(name, use, nx, steps, limiters, precision, out="fields"):
    return {"name": name, "use": use, "lattice": "d1q3", "nx": nx, "ny": 1, "steps": steps, "limiters": limiters,
            "precision": precision, "boundary": 0, "re": 0.0, "u_lid": 0.0, "entropic": False, "out": out}


def listed():
    return [
        # the paper's shock tube (Sec. 4.3): 800 sites, 400 steps, at most four Ehrenfests' sites a step
        tube("tube800_fp64", "solve", 800, 400, EHR, "fp64", out="both"),
        # a long shock tube, FP32, bound by memory
        tube("tube_1e7_fp32", "solve", 10_000_000, 60, EHR, "fp32"),
        # the paper's 100 x 100 cavity at Re = 5000 (Sec. 4.4.1): boundary nodes on the walls, median filter
        cavity("cavity100_nodes", "solve", 100, 100, 500, MED, boundary=3, re=5000.0, u_lid=0.1, out="both"),
        # one served-size cavity of odd sides with the three fixed limiters
        cavity("cavity_517x389", "solve", 517, 389, 200, POS | EHR | MED, re=5000.0, u_lid=0.1, out="both"),
        # the headline workload: 4096^2, Re = 7500, median filter and Ehrenfests' steps
        cavity("cavity4096_fp32", "advance", 4096, 4096, 20, EHR | MED),
        # the same with 16-bit storage, read back as a checkpoint
        cavity("cavity4096_bf16", "advance", 4096, 4096, 20, EHR | MED, precision="bf16", out="populations"),
        # a restart from a state with every site out of equilibrium
        cavity("active2048_fp32", "reload", 2048, 2048, 4, EHR | MED, out="populations"),
        # entropic quasiequilibria and the exact entropy
        cavity("entropic2048_fp32", "advance", 2048, 2048, 10, EHR | MED, entropic=True),
        # the threshold filter solved on the whole ensemble (Eq. EntThresh)
        cavity("entthresh2048_fp32", "advance", 2048, 2048, 10, EHR | ENTTHR),
        # the FP64 path that reproduces the formulas bit for bit
        cavity("cavity_600x500_fp64", "advance", 600, 500, 20, POS | EHR | MED, precision="fp64", re=5000.0, u_lid=0.1,
               out="populations"),
        # 256 cavities of sides 64 to 512 in one batch, one fixed limiter each, graph replay
        {"name": "batch256", "use": "batch", "count": 256, "lo": 64, "hi": 512, "steps": 40, "graph": 20,
         "shape_seed": BATCH_SEED},
        # a closed queue of requests of the serving mix (70 % cavities, 30 % tubes) through the server
        {"name": "serve16", "use": "serve", "count": 16, "max_side": 1024, "max_tube": 1_000_000, "min_steps": 100,
         "max_steps": 400, "quantum": 100, "graph": 50, "shape_seed": SERVE_SEED},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "tube", "nodes", "small", "small", "large", "low", "active", "entropic", "ensemble",
                       "fp64", "batch", "serve"])
    fixed = rng.choice([POS, EHR, MED, EHR | MED, POS | EHR | MED])
    if kind == "tube":
        prec = rng.choice(["fp32", "fp64"])
        n = _log(rng, 800, 10_000_000 if prec == "fp32" else 1_000_000)
        return _unnamed(tube("", "solve", n, max(20, min(400, 400_000_000 // n)), fixed, prec,
                             out="both" if n < 100_000 else "fields"))
    if kind == "nodes":
        n = _log(rng, 64, 256)
        return _unnamed(cavity("", "solve", n, n + rng.randrange(-20, 21), rng.randrange(200, 501), MED,
                               boundary=rng.choice([3, 3, 4]), re=5000.0, u_lid=0.1, out="both"))
    if kind == "small":
        return _unnamed(cavity("", "solve", _log(rng, 64, 1024), _log(rng, 64, 1024), rng.randrange(100, 301), fixed,
                               re=rng.uniform(2000.0, 5000.0), u_lid=0.1, out="both"))
    if kind in ("large", "low"):
        prec = "fp32" if kind == "large" else rng.choice(["bf16", "fp16"])
        return _unnamed(cavity("", "advance", _log(rng, 1024, 4096), _log(rng, 1024, 4096), 20, fixed, precision=prec,
                               out=rng.choice(["fields", "populations"])))
    if kind == "active":
        return _unnamed(cavity("", "reload", _log(rng, 1100, 2048), _log(rng, 1100, 2048), rng.randrange(2, 5),
                               EHR | MED, precision=rng.choice(["fp32", "fp32", "bf16"]), out="populations"))
    if kind == "entropic":
        return _unnamed(cavity("", "advance", _log(rng, 256, 2048), _log(rng, 256, 2048), 10, fixed, entropic=True))
    if kind == "ensemble":
        return _unnamed(cavity("", "advance", _log(rng, 512, 2048), _log(rng, 512, 2048), 10,
                               rng.choice([0, EHR]) | rng.choice([SMOOTH, THRESH, ENTTHR])))
    if kind == "fp64":
        return _unnamed(cavity("", "advance", _log(rng, 64, 600), _log(rng, 64, 500), 20, fixed, precision="fp64",
                               re=5000.0, u_lid=0.1, entropic=rng.random() < 0.3, out="populations"))
    if kind == "batch":
        return {"use": "batch", "count": _log(rng, 16, 224), "lo": 64, "hi": rng.randrange(200, 513), "steps": 40,
                "graph": rng.choice([0, 20]), "shape_seed": rng.randrange(1 << 30)}
    return {"use": "serve", "count": rng.randrange(4, 13), "max_side": rng.randrange(200, 1025),
            "max_tube": _log(rng, 2000, 1_000_000), "min_steps": 100, "max_steps": 400, "quantum": 100,
            "graph": rng.choice([0, 50]), "shape_seed": rng.randrange(1 << 30)}


def _unnamed(case):
    del case["name"]
    return case


# -- what the lattices of a case are ------------------------------------------

def _config(case):
    """lbm_config fields of a lone lattice."""
    n = case["nx"] * case["ny"]
    cfg = dict(nx=case["nx"], ny=case["ny"], boundary=case["boundary"], precision=PRECISION[case["precision"]],
               limiters=case["limiters"], delta_median=1e-3, delta_ehrenfest=1e-3,
               equilibrium=lbm.EQ_ENTROPIC if case["entropic"] else lbm.EQ_POLYNOMIAL)
    if case["lattice"] == "d1q3":
        return dict(cfg, lattice=lbm.D1Q3, beta=inputs.beta_from_nu(1e-9), k_max=4)
    side = max(case["nx"], case["ny"])
    return dict(cfg, lattice=lbm.D2Q9, beta=inputs.beta_from_nu(inputs.cavity_nu(side, case["u_lid"], case["re"])),
                u_lid=case["u_lid"], rho_wall=1.0, k_max=max(1, n // 10000))


def _workload_config(w):
    return dict(serve.lattice_config(w), delta_median=w.delta_median)


def _batch_workloads(case):
    return inputs.batched_cavities(case["shape_seed"], case["count"], case["lo"], case["hi"], case["steps"])


def _serve_workloads(case):
    trace = inputs.serving_trace(case["shape_seed"], case["count"], min_steps=case["min_steps"],
                                 max_steps=case["max_steps"], max_cavity=case["max_side"], max_tube=case["max_tube"])
    return [w for _, w in trace]


# -- inputs -------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _tube_moments(n, seed):
    """Two-density shock tube at rest, ratio near 1:2, the front near the middle."""
    r = random.Random(seed * 7919 + n)
    right, split = 1.0 / r.uniform(1.8, 2.2), r.uniform(0.45, 0.55)
    rho, ux = inputs.shock_tube(n, 1.0, right, split)
    return torch.from_numpy(rho).to(_device()), torch.from_numpy(ux).to(_device()), None


def _cavity_moments(nx, ny, seed, amp):
    """A few smooth eddies of speed about `amp` that vanish at the walls, density near 1."""
    r = random.Random(seed * 7919 + nx * 31 + ny)
    x = (torch.arange(nx, dtype=torch.float64, device=_device()) + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device=_device()) + 0.5) / ny
    ux = torch.zeros((ny, nx), dtype=torch.float64, device=_device())
    uy, rho = torch.zeros_like(ux), torch.ones_like(ux)
    for _ in range(4):
        m, n, a = r.randrange(1, 4), r.randrange(1, 4), amp * r.uniform(-0.5, 0.5)
        sx, sy = torch.sin(m * math.pi * x), torch.sin(n * math.pi * y)
        # stream function a sin^2(m pi x) sin^2(n pi y), scaled to speed a
        ux += a * torch.outer(2 * sy * torch.cos(n * math.pi * y), sx * sx)
        uy -= a * m / n * torch.outer(sy * sy, 2 * sx * torch.cos(m * math.pi * x))
        rho += 0.02 * amp * r.uniform(-1, 1) * torch.outer(torch.cos(n * math.pi * y), torch.cos(m * math.pi * x))
    return rho, ux, uy


def _moments(case, seed):
    if case["lattice"] == "d1q3":
        return _tube_moments(case["nx"], seed)
    return _cavity_moments(case["nx"], case["ny"], seed, 0.5 * case["u_lid"])


def _active_populations(case, seed):
    """Every population off its rest value by up to 15 %, and a strong local excess at a few sites."""
    w = torch.tensor(_weights(9), dtype=torch.float64, device=_device()).view(9, 1, 1)
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    shape = (9, case["ny"], case["nx"])
    f = w * (1 + 0.15 * (2 * torch.rand(shape, dtype=torch.float64, device=_device(), generator=gen) - 1))
    r = np.random.default_rng(seed)
    k, y, x = r.integers(1, 9, 1000), r.integers(0, case["ny"], 1000), r.integers(0, case["nx"], 1000)
    f[torch.from_numpy(k), torch.from_numpy(y), torch.from_numpy(x)] *= 8.0
    return f


def _member_moments(w, seed, i):
    """One lattice of a batch or request: the tube, or a cavity with weak eddies."""
    if w.lattice == lbm.D1Q3:
        n = w.nx
        rho, ux = inputs.shock_tube(n, 1.0, w.rho_right, random.Random(seed * 7919 + i).uniform(0.45, 0.55))
        return torch.from_numpy(rho).to(_device()), torch.from_numpy(ux).to(_device()), None
    return _cavity_moments(w.nx, w.ny, seed * 613 + i, 0.3 * w.u_lid)


# -- the cases ----------------------------------------------------------------

class State:
    pass


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device=_device())


def prepare(case, seed):
    s = State()
    s.case = case
    if case["use"] == "batch":
        ws = _batch_workloads(case)
        s.batch = lbm.Batch()
        if case["graph"]:
            s.batch.set_graph(case["graph"])
        s.slots = [s.batch.add(**_workload_config(w)) for w in ws]
        s.out = _empty(sum(9 * w.sites for w in ws))
        s.views, at = [], 0
        for i, (slot, w) in enumerate(zip(s.slots, ws)):
            s.batch.init(slot, *_member_moments(w, seed, i))
            s.views.append(s.out[at:at + 9 * w.sites].view(9, w.ny, w.nx))
            at += 9 * w.sites
        return s
    if case["use"] == "serve":
        ws = _serve_workloads(case)
        s.server = serve.Server(64 << 30, quantum=case["quantum"], graph_steps=case["graph"])
        s.requests = []
        for i, w in enumerate(ws):
            fields = [None if a is None else a.cpu().numpy() for a in _member_moments(w, seed, i)]
            s.requests.append(serve.Request(i, 0.0, w, *fields))
        return s
    s.lattice = lbm.Lattice(**_config(case))
    q = s.lattice.q
    if case["use"] == "reload":
        s.f = _active_populations(case, seed)
    else:
        s.moments = _moments(case, seed)
        if case["use"] == "advance":
            s.lattice.init(*s.moments)
    shape = (case["ny"], case["nx"])
    s.fields = tuple(_empty(*shape) for _ in range(3)) if case["out"] in ("fields", "both") else None
    s.populations = _empty(q, *shape) if case["out"] in ("populations", "both") else None
    return s


def run(s):
    case = s.case
    if case["use"] == "batch":
        s.batch.step(case["steps"])
        for slot, view in zip(s.slots, s.views):
            s.batch.get_populations(slot, view)
        return {"populations": s.out}
    if case["use"] == "serve":
        done = sorted(s.server.run(s.requests, realtime=False), key=lambda r: r.rid)
        ok = [r for r in done if r.status == "ok"]
        return {"rid": np.array([r.rid for r in ok]), "steps": np.array([r.steps for r in ok]),
                "rho": np.concatenate([r.rho.ravel() for r in ok]),
                "ux": np.concatenate([r.ux.ravel() for r in ok]),
                "uy": np.concatenate([r.uy.ravel() for r in ok])}
    lat = s.lattice
    if case["use"] == "solve":
        lat.init(*s.moments)
    elif case["use"] == "reload":
        lat.set_populations(s.f)
    lat.step(case["steps"])
    out = {}
    if s.fields is not None:
        lat.moments(s.fields)
        out["rho"], out["ux"] = s.fields[0], s.fields[1]
        if lat.q == 9:
            out["uy"] = s.fields[2]
    if s.populations is not None:
        out["populations"] = lat.get_populations(s.populations)
    st = lat.stats()
    out["stats"] = {k: st[k] for k in STATS}
    return out


def _site_bytes(q, elem, limiters):
    """Bytes a step reads and writes at a site: every population once each; an ensemble-dependent
    limiter reads the populations once more, and Eq. EntThresh writes and reads one entropy."""
    b = 2 * q * elem
    if limiters & (SMOOTH | THRESH | ENTTHR):
        b += q * elem
    if limiters & ENTTHR:
        b += 2 * max(4, elem)
    return b


def work(case):
    # operations of one site's step: moments, f*, collision, the entropies of two states
    ops = {9: 250, 3: 80}
    if case["use"] == "batch":
        n = sum(w.sites for w in _batch_workloads(case))
        return {"bytes": n * (72 * case["steps"] + 9 * 12), "flops": n * case["steps"] * ops[9]}
    if case["use"] == "serve":
        byte = flop = 0
        for w in _serve_workloads(case):
            q = 3 if w.lattice == lbm.D1Q3 else 9
            byte += w.sites * (8 * q * w.steps + 2 * 24 + 8 * q)
            flop += w.sites * w.steps * ops[q]
        return {"bytes": byte, "flops": flop}
    q, n, e = (3 if case["lattice"] == "d1q3" else 9), case["nx"] * case["ny"], ELEM[case["precision"]]
    b = case["steps"] * _site_bytes(q, e, case["limiters"])
    if case["use"] == "solve":
        b += (16 if q == 3 else 24) + q * e
    if case["use"] == "reload":
        b += q * (8 + e)
    if case["out"] in ("fields", "both"):
        b += q * e + (16 if q == 3 else 24)
    if case["out"] in ("populations", "both"):
        b += q * (e + 8)
    return {"bytes": n * b, "flops": n * case["steps"] * ops[q] * (3 if case["entropic"] else 1)}


# -- the same steps in FP64 with plain torch ----------------------------------

def _weights(q):
    return [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if q == 9 else [2 / 3, 1 / 6, 1 / 6]


CX = {9: [0, 1, 0, -1, 0, 1, -1, -1, 1], 3: [0, -1, 1]}
CY = {9: [0, 0, 1, 0, -1, 1, 1, -1, -1], 3: [0, 0, 0]}
OPP = {9: [0, 3, 4, 1, 2, 7, 8, 5, 6], 3: [0, 2, 1]}


def _feq(rho, ux, uy, q, entropic):
    w = _weights(q)
    if entropic:
        axes = []
        for u in (ux, uy):
            s = torch.sqrt(1 + 3 * u * u)
            a, x = 2 - s, (2 * u + s) / (1 - u)
            axes.append({0: a, 1: a * x, -1: a / x})
        return torch.stack([rho * w[k] * axes[0][CX[q][k]] * axes[1][CY[q][k]] for k in range(q)])
    usq = ux * ux + uy * uy
    out = []
    for k in range(q):
        c = CX[q][k] * ux + CY[q][k] * uy
        out.append(rho * w[k] * (1 + 3 * c + 4.5 * c * c - 1.5 * usq))
    return torch.stack(out)


def _macro(f, q):
    rho = f.sum(0)
    ux = sum(CX[q][k] * f[k] for k in range(q) if CX[q][k]) / rho
    uy = sum(CY[q][k] * f[k] for k in range(q) if CY[q][k]) / rho if q == 9 else torch.zeros_like(ux)
    return rho, ux, uy


def _entropy(f, fs, entropic):
    if not entropic:
        return ((f - fs) ** 2 / fs).sum(0)
    # sum f ln(f / f*): the terms with their linear part taken out, which sums to nothing
    d = f - fs
    t = torch.where(f > 0, f * torch.log1p(d / fs) - d, fs)
    return torch.where((f < 0).any(0), torch.full_like(f[0], math.inf), t.sum(0))


class Exact:
    """One lattice stepped in FP64 (Sec. 2 to 4 of the paper)."""

    def __init__(self, q, cfg):
        self.q, self.c = q, cfg
        self.ent = cfg.get("equilibrium", 0) == 1
        self.a = 2 * cfg["beta"] - 1
        self.sums = {}

    def init(self, rho, ux, uy):
        ny, nx = self.c["ny"], self.c["nx"]
        rho, ux = rho.view(ny, nx), ux.view(ny, nx)
        uy = torch.zeros_like(ux) if uy is None else uy.view(ny, nx)
        self.f = _feq(rho, ux, uy, self.q, self.ent)

    def stream(self):
        q, f, c = self.q, self.f, self.c
        ny, nx = f.shape[1:]
        out = torch.empty_like(f)
        node = c["boundary"] >= 3
        missing = torch.zeros((q, ny, nx), dtype=torch.bool, device=f.device) if node else None
        for k in range(q):
            cx, cy, o = CX[q][k], CY[q][k], OPP[q][k]
            out[k] = torch.roll(f[k], (cy, cx), (0, 1))
            lid = 6 * _weights(q)[k] * c.get("rho_wall", 1.0) * cx * c.get("u_lid", 0.0) if cy == -1 else 0.0
            edges = []
            if cx:
                edges.append((slice(None), 0 if cx > 0 else nx - 1))
            if cy:
                edges.append((0 if cy > 0 else ny - 1, slice(None)))
            for e in edges:
                if node:
                    missing[(k,) + e] = True
                else:  # halfway bounce-back: the site's own opposite population
                    out[(k,) + e] = f[(o,) + e]
            if cy == -1 and not node:
                out[k, ny - 1] += lid
        if node:
            self.wall_nodes(out, missing)
        return out

    def wall_nodes(self, out, missing):
        """Boundary nodes on the walls: the populations without a source come from the wall rule."""
        q, c = 9, self.c
        ny, nx = out.shape[1:]
        uw = torch.zeros((ny, nx), dtype=out.dtype, device=out.device)
        uw[ny - 1, 1:nx - 1] = c["u_lid"]
        corner = torch.zeros((ny, nx), dtype=torch.bool, device=out.device)
        corner[::ny - 1, ::nx - 1] = True
        arrived = out.clone()
        fw = _feq(torch.ones_like(uw), uw, torch.zeros_like(uw), 9, self.ent)
        num = sum(torch.where(missing[k], arrived[OPP[9][k]], 0.0) for k in range(q))
        den = sum(torch.where(missing[k], fw[k], 0.0) for k in range(q))
        gamma = num / torch.where(den > 0, den, 1.0)
        for k in range(q):
            o = OPP[9][k]
            bounce = arrived[o] + 6 * _weights(9)[k] * c["rho_wall"] * CX[9][k] * uw
            bounce = torch.where(missing[o], self.f[k], bounce)  # a corner's tangent links keep their value
            v = torch.where(corner, bounce, gamma * fw[k]) if c["boundary"] == 4 else bounce
            out[k] = torch.where(missing[k], v, out[k])

    def median(self, ds, at):
        """Median of the stencil at the sites `at` (flat indices); -inf where the filter skips the site."""
        ny, nx = ds.shape
        y, x = at // nx, at % nx
        if self.q == 3:
            m = torch.stack([ds[0, (x + d).clamp(0, nx - 1)] for d in (-1, 0, 1)]).median(0).values
            return m, (x > 0) & (x < nx - 1)
        b = 1 if self.c["boundary"] >= 3 else 0  # the ring whose stencils lie along the wall
        near_x, near_y = (x == b) | (x == nx - 1 - b), (y == b) | (y == ny - 1 - b)

        def at_(dx, dy):
            return ds[(y + dy).clamp(0, ny - 1), (x + dx).clamp(0, nx - 1)]

        full = torch.stack([at_(i, j) for j in (-1, 0, 1) for i in (-1, 0, 1)]).median(0).values
        row = torch.stack([at_(-1, 0), at_(0, 0), at_(1, 0)]).median(0).values
        col = torch.stack([at_(0, -1), at_(0, 0), at_(0, 1)]).median(0).values
        ix, iy = torch.where(x == b, 1, -1), torch.where(y == b, 1, -1)
        cor = torch.stack([at_(0, 0), at_(ix, torch.zeros_like(iy)), at_(torch.zeros_like(ix), iy)]).median(0).values
        return torch.where(near_x & near_y, cor, torch.where(near_y, row, torch.where(near_x, col, full))), None

    def step(self):
        q, c, a, lim = self.q, self.c, self.a, self.c["limiters"]
        fin = self.stream()
        ny, nx = fin.shape[1:]
        node = c["boundary"] >= 3
        inside = torch.ones((ny, nx), dtype=torch.bool, device=fin.device)
        if node:
            inside[0] = inside[-1] = inside[:, 0] = inside[:, -1] = False
        rho, ux, uy = _macro(fin, q)
        fs = _feq(rho, ux, uy, q, self.ent)
        fp = fs + a * (fs - fin)
        ds = torch.where(inside, _entropy(fp, fs, self.ent), 0.0)
        phi = torch.ones_like(ds)
        if lim & POS:
            r = torch.where(fp < 0, fs / (fs - fp), 1.0).amin(0)
            phi = torch.minimum(phi, r)
        if lim & MED:
            delta = c["delta_median"]
            at = torch.nonzero((ds > delta).flatten()).flatten()
            if at.numel():
                med, on = self.median(ds, at)
                t = torch.clamp(med, min=delta)
                d = ds.flatten()[at]
                p = torch.where(d > t, torch.sqrt(t / d), torch.ones_like(d))
                if on is not None:
                    p = torch.where(on, p, 1.0)
                flat = phi.flatten()
                flat[at] = torch.minimum(flat[at], p)
                phi = flat.view(ny, nx)
        if lim & (SMOOTH | THRESH | ENTTHR):
            mean = ds.mean()
            if lim & SMOOTH:
                phi = torch.minimum(phi, 1 / (1 + 0.01 / mean ** 0.5 * ds ** 0.5))
            if lim & THRESH:
                phi = torch.minimum(phi, torch.where(ds > 10 * mean, torch.sqrt(10 * mean / ds), 1.0))
            if lim & ENTTHR:
                v = torch.sort(ds.flatten(), descending=True).values
                above = torch.cumsum(v, 0) - v * torch.arange(1, v.numel() + 1, dtype=v.dtype, device=v.device)
                rhs = 0.1 * (1 - a * a) * v.sum()
                m = int((above < rhs).sum())  # the values above dS_0
                t = (v[:m].sum() - rhs) / m if m else torch.full_like(mean, math.inf)
                phi = torch.minimum(phi, torch.where(ds > t, torch.sqrt(t.clamp(min=0.0) / ds), 1.0))
        phi = torch.where(inside, phi, 1.0)
        fo = torch.where(phi < 1, fs + phi * (fp - fs), fp)
        if node:
            fo = torch.where(inside, fo, fin)
        if self.ent:
            s_in = (_entropy(fin, fs, True) - ds).sum()
            lost = torch.where(phi < 1, ds - _entropy(fo, fs, True), 0.0).sum()
        else:
            s_in = (1 - a * a) * torch.where(inside, _entropy(fin, fs, False), 0.0).sum()
            lost = ((1 - phi * phi) * ds).sum()
        if lim & EHR:
            d = ds.flatten()
            at = torch.nonzero(d > c["delta_ehrenfest"]).flatten()
            if at.numel() > c["k_max"]:
                at = at[torch.sort(d[at], descending=True, stable=True).indices[:c["k_max"]]]
            if at.numel():
                y, x = at // nx, at % nx
                chosen = fo[:, y, x]
                star = _feq(*_macro(chosen, q), q, self.ent)
                lost = lost + (_entropy(chosen, star, True).sum() if self.ent else (phi[y, x] ** 2 * d[at]).sum())
                fo[:, y, x] = star
        if node:  # a boundary node counts the populations that stream back onto the lattice
            mass = rho[1:-1, 1:-1].sum()
            for k in range(q):
                ys = slice(max(0, -CY[q][k]), ny - max(0, CY[q][k]))
                xs = slice(max(0, -CX[q][k]), nx - max(0, CX[q][k]))
                ring = torch.where(inside, 0.0, fin[k])
                mass = mass + ring[ys, xs].sum()
        else:
            mass = rho.sum()
        self.sums = {"mass": float(mass), "sum_dS": float(ds.sum()), "dS_lbgk": float(s_in), "dS_lim": float(lost)}
        self.f = fo


def _exact_member(w, seed, i, steps):
    e = Exact(3 if w.lattice == lbm.D1Q3 else 9, _workload_config(w))
    e.init(*_member_moments(w, seed, i))
    for _ in range(steps):
        e.step()
    return e


def exact(case, seed):
    if case["use"] == "batch":
        ws = _batch_workloads(case)
        return {"populations": torch.cat([_exact_member(w, seed, i, w.steps).f.flatten() for i, w in enumerate(ws)])}
    if case["use"] == "serve":
        ws = _serve_workloads(case)
        fields = [_macro(e.f, e.q) for e in (_exact_member(w, seed, i, w.steps) for i, w in enumerate(ws))]
        ok = [m for m in fields if all(bool(torch.isfinite(v).all()) for v in m)]
        rho, ux, uy = (torch.cat([m[j].flatten() for m in ok]).cpu().numpy() for j in range(3))
        return {"rid": None, "steps": None, "rho": rho, "ux": ux, "uy": uy}
    cfg = _config(case)
    e = Exact(3 if case["lattice"] == "d1q3" else 9, cfg)
    if case["use"] == "reload":
        e.f = _active_populations(case, seed)
    else:
        e.init(*_moments(case, seed))
    for _ in range(case["steps"]):
        e.step()
    out = {}
    if case["out"] in ("fields", "both"):
        out["rho"], out["ux"], uy = _macro(e.f, e.q)
        if e.q == 9:
            out["uy"] = uy
    if case["out"] in ("populations", "both"):
        out["populations"] = e.f
    out["stats"] = {k: e.sums[k] if k in SUMS else None for k in STATS}
    return out
