"""What this framework's users run, as cases that can be timed and compared.

Every case goes through the public binding (``paper_2501_06717_gb300.bats``)
and keeps what such a program keeps: a solver handle (its tree, tables and
captured graph) or a trainer handle, the initial state on the device and a
buffer for the result.  One pass of a solver case loads the initial state,
advances it by the case's number of steps and fetches the final state, as a
run from one checkpoint to the next does; one pass of a network case infers or
trains on its rows.

A case's "tree" says which grid it runs on:
  orszag         2x2x2 periodic root blocks, Orszag-Tang vortex (the first
                 program a new user runs)
  blast          [-1,1]^3, roots^3 root blocks refined once inside r < 0.4,
                 outflow, spherical blast
  fast_wave      Table 2 of the paper: 15 * 2^m blocks, periodic
  magnetosphere  five levels, dipole B0, inner body, inflow, Powell terms
  batched        `grids` independent periodic grids of log-uniform size
"""
import math
import random

import numpy as np
import torch

from paper_2501_06717_gb300 import bats as B
from paper_2501_06717_gb300 import workloads as W

LIMITERS = {"minmod": W.LIM_MINMOD, "mc": W.LIM_MC, "none": W.LIM_NONE}
SCHEMES = {"midpoint": W.RK_MIDPOINT, "ssp2": W.RK_SSP2, "euler": W.RK_EULER}
FLUXES = {"rusanov": W.FLUX_RUSANOV, "hll": W.FLUX_HLL, "linde": W.FLUX_LINDE}


def _solver(name, tree, precision, steps, **more):
    case = {"name": name, "kind": "solver", "tree": tree, "size": 0, "grids": 1, "tree_seed": 1, "precision": precision,
            "steps": steps, "limiter": "minmod", "scheme": "midpoint", "flux": "rusanov", "local_dt": False,
            "learned": False, "graph": True, "persistent": False, "blocks_per_cta": 1}
    case.update(more)
    return case


def listed():
    return [
        # one eager step of the smallest grid (8 blocks) with the solver's
        # defaults: an interactive call, where launches and the host path count
        _solver("orszag_fp64_one_step", "orszag", "fp64", 1, graph=False),
        # the block-adaptive blast (120 blocks), a whole 100-step run of the
        # mixed form replayed from a CUDA graph: launch-bound steps
        _solver("blast_mixed_100_steps", "blast", "mixed", 100, size=4, limiter="mc"),
        # the same grid in FP64, where a grid this small leaves part of the GPU idle
        _solver("blast_fp64_10_steps", "blast", "fp64", 10, size=4, limiter="mc"),
        # the paper's one-GPU fast-wave run (Table 2 grid at m = 6, 960 blocks,
        # contact-restoring flux), a tenth of its 500 steps
        _solver("fast_wave_linde_mixed", "fast_wave", "mixed", 50, size=6, flux="linde", persistent=True),
        # the magnetosphere-like run (3,872 blocks): dipole, body, inflow, Powell
        _solver("magnetosphere_mixed", "magnetosphere", "mixed", 10, persistent=True),
        # its steady-state session in FP64: local time steps
        _solver("magnetosphere_fp64_local_dt", "magnetosphere", "fp64", 2, local_dt=True),
        # the batched workload (64 uneven grids, 30 M cells) in the mixed form:
        # the largest call, in the launch form the autotuner picks for it
        _solver("batched_mixed", "batched", "mixed", 4, grids=64, tree_seed=20250112, blocks_per_cta=8),
        # a few of those grids in FP64 (the accuracy reference of a mixed run)
        _solver("batched_fp64", "batched", "fp64", 1, grids=6, tree_seed=20250113, flux="hll"),
        # the learned flux correction on a grid that fills the GPU (6,056 blocks)
        _solver("blast_learned_mixed", "blast", "mixed", 4, size=16, limiter="mc", learned=True),
        # the network alone: inference over the faces of a large grid
        {"name": "network_inference", "kind": "infer", "rows": 2000000},
        # training: one epoch of minibatch steps over pairs on the device
        {"name": "network_training_epoch", "kind": "train", "rows": 120003, "batch": 8192},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solver"] * 6 + ["infer", "train"])
    if kind == "infer":
        return {"kind": "infer", "rows": log_int(120000, 2000000)}
    if kind == "train":
        return {"kind": "train", "rows": log_int(1000, 120000), "batch": rng.choice([200, 1000, 4096, 8192])}
    tree = rng.choice(["blast", "fast_wave", "magnetosphere", "batched", "batched", "orszag"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    more = {"limiter": rng.choice(["minmod", "mc"]), "scheme": rng.choice(["midpoint"] * 4 + ["ssp2"]),
            "flux": rng.choice(["rusanov", "rusanov", "hll", "linde"]), "graph": rng.random() < 0.75,
            "persistent": rng.random() < 0.5, "blocks_per_cta": rng.choice([1, 1, 2, 4, 8])}
    if tree == "blast":
        more["size"] = rng.choice([4, 5, 6, 8, 12])
        if precision == "mixed" and more["size"] <= 8 and rng.random() < 0.3:
            more.update(learned=True, scheme="midpoint", flux="rusanov")
        steps = log_int(1, 60 if precision == "mixed" else 10) if more["size"] < 12 else rng.randint(1, 4)
    elif tree == "fast_wave":
        more["size"] = rng.choice([0, 3, 6, 9])
        steps = log_int(1, 40 if precision == "mixed" else 4) if more["size"] < 9 else 1
    elif tree == "magnetosphere":
        more.update(limiter="minmod", flux="rusanov", scheme=rng.choice(["midpoint", "midpoint", "euler"]))
        if more["scheme"] == "euler":
            more["limiter"] = "none"
        else:
            more["local_dt"] = rng.random() < 0.3
        steps = rng.randint(1, 8 if precision == "mixed" else 2)
    elif tree == "batched":
        more["grids"] = log_int(1, 24 if precision == "mixed" else 3)
        more["tree_seed"] = rng.randrange(1 << 20)
        steps = rng.randint(1, 2)
    else:
        steps = log_int(1, 100)
    return {k: v for k, v in _solver("", tree, precision, steps, **more).items() if k != "name"}


# --------------------------------------------------------------------------
# Trees and initial states


def _random_leaves(target, seed):
    """About `target` leaves on the periodic unit cube: 4^3, 8^3 or 16^3
    roots, refined up to two levels inside seeded spheres, 2:1 balanced."""
    rng = np.random.default_rng(seed)
    r = 4 if target < 512 else (8 if target < 4096 else 16)
    ref = [np.zeros((r << l,) * 3, bool) for l in range(2)]

    def hits(n, c, rad):
        e = np.arange(n) / n
        q = [np.clip(c[a], e, e + 1.0 / n) - c[a] for a in range(3)]
        return q[0][:, None, None] ** 2 + q[1][None, :, None] ** 2 + q[2][None, None, :] ** 2 < rad * rad

    def up(a):
        return a.repeat(2, 0).repeat(2, 1).repeat(2, 2)

    for _ in range(200):
        if r ** 3 + 7 * (ref[0].sum() + ref[1].sum()) >= target:
            break
        c, rad, deep = rng.uniform(0, 1, 3), rng.uniform(0.05, 0.25), rng.integers(0, 2)
        new = [ref[0] | hits(r, c, rad), ref[1]]
        if deep:
            new[1] = ref[1] | (hits(2 * r, c, rad) & up(ref[0]))
        if r ** 3 + 7 * (new[0].sum() + new[1].sum()) <= 1.25 * target:
            ref = new
    wide = ref[1].copy()
    for ax in range(3):
        wide = wide | np.roll(wide, 1, ax) | np.roll(wide, -1, ax)
    ref[0] |= wide.reshape(r, 2, r, 2, r, 2).any(axis=(1, 3, 5))
    parts = []
    for lev, m in enumerate((~ref[0], up(ref[0]) & ~ref[1], up(ref[1]))):
        p = np.argwhere(m)
        parts.append(np.concatenate([np.full((len(p), 1), lev), p], 1))
    lv = np.concatenate(parts)
    z = lv[:, 1:] << (2 - lv[:, :1])  # Z order at the finest level
    code = sum(((z[:, a] >> b) & 1) << (3 * b + a) for a in range(3) for b in range(7))
    return (r,) * 3, lv[np.argsort(code, kind="stable")].astype(np.int32)


_trees = {}


def _problems(case):
    """The grids of a case, without their states (the same for every seed)."""
    key = (case["tree"], case["size"], case["grids"], case["tree_seed"])
    if key not in _trees:
        tree, size = case["tree"], case["size"]
        per, out = (W.BC_PERIODIC,) * 6, (W.BC_OUTFLOW,) * 6
        if tree == "orszag":
            g = [((0.0,) * 3, (1.0,) * 3, (2,) * 3, W.as_leaf_array(W.uniform_leaves((2, 2, 2))), per, {})]
        elif tree == "blast":
            lo, hi, root = (-1.0,) * 3, (1.0,) * 3, (size,) * 3
            near = lambda b0, b1: float(np.linalg.norm(np.clip(0.0, b0, b1))) < 0.4  # noqa: E731
            lv = W.balance(W.refine_where(W.uniform_leaves(root), near, lo, hi, root, 1), root, (False,) * 3)
            g = [(lo, hi, root, W.as_leaf_array(W.morton_sort(lv)), out, {})]
        elif tree == "fast_wave":
            g = [W.fast_wave_leaves(size) + (per, {})]
        elif tree == "magnetosphere":
            bc = (W.BC_OUTFLOW, W.BC_INFLOW) + (W.BC_OUTFLOW,) * 4
            b0 = np.zeros(12)
            b0[2] = -31000.0 / W.B_UNIT_NT
            body = np.array([28.0, 0, 0, 0, 0, 0, 0, 28.0 * 2.5e4 / W.KT_UNIT_K])
            g = [W.magnetosphere_leaves() + (bc, dict(b0=W.B0_DIPOLE, b0_param=b0, powell=1, body_r=2.5, body=body))]
        else:
            t = np.exp(np.random.default_rng(case["tree_seed"]).uniform(math.log(64), math.log(4096), case["grids"]))
            g = [((0.0,) * 3, (1.0,) * 3) + _random_leaves(int(n), case["tree_seed"] * 1000 + i) + (per, {})
                 for i, n in enumerate(t)]
        _trees[key] = [(lo, hi, root, lv, bc, kw) for lo, hi, root, lv, bc, kw in g]
    return [W.Problem(case["tree"], lo, hi, root, lv, bc, limiter=LIMITERS[case["limiter"]], rk=SCHEMES[case["scheme"]],
                      flux=FLUXES[case["flux"]], local_dt=int(case["local_dt"]), learned_last_only=int(case["learned"]),
                      **kw) for lo, hi, root, lv, bc, kw in _trees[key]]


def _axes(p):
    """Cell-centre coordinates along x, y, z, each [nb][8]."""
    lv = torch.from_numpy(p.leaves.astype(np.float64)).cuda()
    n = torch.arange(8, device="cuda", dtype=torch.float64) + 0.5
    dx = [(p.hi[a] - p.lo[a]) / (p.root[a] * 8) / 2 ** lv[:, 0] for a in range(3)]
    return [p.lo[a] + (8 * lv[:, 1 + a, None] + n) * dx[a][:, None] for a in range(3)]


def _modes(rng, xs, count=8):
    """A sum of seeded cosine modes |k| <= 4 and its bound: (value and the
    three derivatives, bounds of the value and of the derivatives)."""
    k = rng.integers(-4, 5, (count, 3))
    k[~k.any(1), 0] = 1
    a, ph = rng.uniform(0.2, 1.0, count), rng.uniform(0, 2 * math.pi, count)
    kt, at, pt = (torch.from_numpy(v.astype(np.float64)).cuda() for v in (k, a, ph))
    e = [torch.polar(torch.ones_like(x[:, :, None] * kt[:, c]), 2 * math.pi * x[:, :, None] * kt[:, c])
         for c, x in enumerate(xs)]
    zy = (e[2] * torch.polar(at, pt))[:, :, None] * e[1][:, None]
    val = lambda w: torch.einsum("nkjm,nim->nkji", zy * w, e[0])  # noqa: E731
    one = torch.ones_like(at)
    grad = lambda c: -2 * math.pi * val(kt[:, c].to(zy.dtype)).imag  # noqa: E731
    return (lambda: val(one.to(zy.dtype)).real), grad, a.sum(), 2 * math.pi * (a * np.abs(k).max(1)).sum()


def _initial(case, p, seed):
    """Initial state [8][nb][8][8][8] of one grid (FP64, on the device)."""
    rng = np.random.default_rng(seed)
    xs = _axes(p)
    x, y, z = xs[0][:, None, None, :], xs[1][:, None, :, None], xs[2][:, :, None, None]
    one = torch.ones(p.nb, 8, 8, 8, dtype=torch.float64, device="cuda")
    tree = case["tree"]
    if tree == "orszag":
        a, ph = rng.uniform(0.8, 1.2), 2 * math.pi * rng.uniform(size=2)
        s4, sy, sx = math.sqrt(4 * math.pi), torch.sin(2 * math.pi * y + ph[0]), torch.sin(2 * math.pi * x + ph[1])
        w = [25 / (36 * math.pi), -a * sy, a * sx, 0.0, -sy / s4, torch.sin(4 * math.pi * x + ph[1]) / s4, 0.0,
             5 / (12 * math.pi)]
    elif tree == "blast":
        c, pin, b = rng.uniform(-0.1, 0.1, 3), rng.uniform(3.0, 30.0), rng.normal(size=3)
        b /= np.linalg.norm(b)
        r2 = (x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2
        w = [1.0, 0.0, 0.0, 0.0, b[0], b[1], b[2], torch.where(r2 < 0.01, pin, 0.1)]
    elif tree == "fast_wave":
        c = rng.uniform(0.5, 1.0) * torch.cos(math.pi / 16 * x + rng.uniform(0, 2 * math.pi))
        w = [W.FAST_WAVE_V0[v] + W.FAST_WAVE_V1[v] * c for v in range(8)]
    elif tree == "magnetosphere":
        n, u, t, bz = rng.uniform(4, 7), rng.uniform(-450, -380), rng.uniform(0.8e5, 1.2e5), rng.uniform(-7, -3)
        wind = np.array([n, u, 0, 0, 0, 0, bz / W.B_UNIT_NT, n * t / W.KT_UNIT_K])
        inside = x * x + y * y + z * z < p.body_r ** 2
        p.inflow = wind
        w = [torch.where(inside, float(p.body[v]), float(wind[v])) for v in range(8)]
    else:
        w = []
        for mid in (1.25, 0.0, 0.0, 0.0, 1.25):
            val, _, bound, _ = _modes(rng, xs)
            w.append(mid + (0.75 if mid else 1.0) * val() / bound)
        A = [_modes(rng, xs) for _ in range(3)]
        g, bn = [m[1] for m in A], sum(m[3] for m in A)
        w[4:4] = [(g[2](1) - g[1](2)) / bn, (g[0](2) - g[2](0)) / bn, (g[1](0) - g[0](1)) / bn]
    w = [torch.as_tensor(v, dtype=torch.float64, device="cuda") * one for v in w]
    return torch.stack(_conservative(w, p.gamma))


def _states(case, seed):
    probs = _problems(case)
    U = torch.cat([_initial(case, p, (seed, g)).reshape(-1) for g, p in enumerate(probs)])
    return probs, U


def _network(seed):
    """Weights as training leaves them: hidden layers of unit gain, a small
    output layer."""
    rng = np.random.default_rng((seed, 77))
    return np.concatenate([rng.normal(size=2560) / math.sqrt(40), 0.1 * rng.normal(size=64),
                           rng.normal(size=4096) / 8, 0.1 * rng.normal(size=64),
                           0.02 * rng.normal(size=512), 0.002 * rng.normal(size=8)]).astype(np.float32)


def _face_rows(rows, seed):
    """Network inputs: five neighbouring cells' scaled primitives per row."""
    g = torch.Generator("cuda").manual_seed(seed)
    mid = torch.tensor([1.0, 0, 0, 0, 0.3, 0, 0, 0.2], device="cuda")
    amp = torch.tensor([0.1, 0.4, 0.4, 0.4, 0.3, 0.3, 0.3, 0.1], device="cuda")
    base = torch.randn(rows, 1, 8, generator=g, device="cuda")
    step = torch.randn(rows, 5, 8, generator=g, device="cuda")
    return (mid + amp * (0.9 * base + 0.2 * step).clamp(-2, 2)).reshape(rows, 40)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "infer":
        x = _face_rows(case["rows"], seed)
        s.Xb = torch.zeros(case["rows"], 48, dtype=torch.bfloat16, device="cuda")
        s.Xb[:, :40] = x
        s.Xb = s.Xb.view(torch.int32)
        s.Y = torch.empty(case["rows"], 8, device="cuda")
        s.net = B.Mlp(params=_network(seed), stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        return s
    if case["kind"] == "train":
        s.X = _face_rows(case["rows"], seed)
        s.T = 0.05 * torch.tanh(s.X[:, 8:16] - s.X[:, 16:24])
        s.perm = torch.randperm(case["rows"], generator=torch.Generator().manual_seed(seed)).cuda()
        s.batch = min(case["batch"], case["rows"])
        s.p0 = _network(seed)
        s.net = B.Mlp(params=s.p0)
        torch.cuda.synchronize()
        return s
    probs, s.U0 = _states(case, seed)
    s.out = torch.empty_like(s.U0)
    s.solver = B.Solver(probs, precision=B.BATS_MIXED if case["precision"] == "mixed" else B.BATS_FP64,
                        persistent=int(case["persistent"]), blocks_per_cta=case["blocks_per_cta"],
                        use_graph=int(case["graph"]))
    if case["learned"]:
        s.solver.set_mlp(_network(seed))
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "infer":
        s.net.forward_bf16(s.Xb, s.Y)
        return s.Y
    if kind == "train":
        s.net.set_params(s.p0)
        loss = s.net.train_epoch(s.X, s.T, s.perm, s.batch, 1e-3)
        return {"loss": loss, "params": s.net.get_params()}
    h = s.solver.h
    B.bats_set_states(h, s.U0)
    t = B.bats_step(h, s.case["steps"], 0.8)
    B.bats_get_states(h, s.out)
    return {"state": s.out, "time": t}


def work(case):
    """Per cell and step the state read and written once (FP64) beside the
    pass's own input and output; flops of the two (one) stages' reconstruction,
    fluxes, sources and update as the formulas state them, divisions and roots
    counted as one."""
    if case["kind"] == "infer":
        return {"bytes": case["rows"] * (80 + 32), "flops": case["rows"] * 14336}
    if case["kind"] == "train":
        batch = min(case["batch"], case["rows"])
        n = case["rows"] // batch * batch
        return {"bytes": n * (192 + 8), "flops": n * 3 * 14336}
    cells = 512 * sum(p.nb for p in _problems(case))
    stages = case["steps"] * (1 if case["scheme"] == "euler" else 2)
    net = 3.375 * 14336 * case["steps"] if case["learned"] else 0
    return {"bytes": cells * 128 * (1 + case["steps"]), "flops": cells * (860 * stages + net)}


# --------------------------------------------------------------------------
# The same in plain 64-bit torch


def _gelu(z):
    return 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))


def _layers(p):
    i = np.cumsum([0, 2560, 64, 4096, 64, 512, 8])
    v = [p[a:b] for a, b in zip(i[:-1], i[1:])]
    return v[0].reshape(64, 40), v[1], v[2].reshape(64, 64), v[3], v[4].reshape(8, 64), v[5]


def _mlp(p, x):
    w1, b1, w2, b2, w3, b3 = _layers(p)
    return _gelu(_gelu(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3


def _conservative(w, gamma):
    r, u, b = w[0], w[1:4], w[4:7]
    e = w[7] / (gamma - 1) + 0.5 * r * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) + 0.5 * (b[0] ** 2 + b[1] ** 2 + b[2] ** 2)
    return [r, r * u[0], r * u[1], r * u[2], b[0], b[1], b[2], e]


def _primitive(U, gamma):
    r, m, b = U[0], U[1:4], U[4:7]
    p = (gamma - 1) * (U[7] - 0.5 * (m[0] ** 2 + m[1] ** 2 + m[2] ** 2) / r - 0.5 * (b[0] ** 2 + b[1] ** 2 + b[2] ** 2))
    return torch.stack([r, m[0] / r, m[1] / r, m[2] / r, b[0], b[1], b[2], p])


def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


def _fast(gamma, w, Bn, B2):
    a2, b2 = gamma * w[7] / w[0], B2 / w[0]
    s = a2 + b2
    return torch.sqrt(0.5 * (s + torch.sqrt((s * s - 4 * a2 * Bn * Bn / w[0]).clamp_min(0))))


class _Plain:
    """The scheme on all grids of a case, block by block in 64 bits."""

    def __init__(self, case, probs, net):
        self.case, self.p, self.net = case, probs[0], net
        dev = "cuda"
        lv = np.concatenate([np.concatenate([np.full((p.nb, 1), g), p.leaves], 1) for g, p in enumerate(probs)])
        self.grid, self.lev, *self.b = torch.from_numpy(lv.astype(np.int64)).to(dev).unbind(1)
        self.nb, self.ng = len(lv), len(probs)
        self.root = torch.tensor([p.root for p in probs], device=dev)
        self.lo = torch.tensor(self.p.lo, dtype=torch.float64, device=dev)
        ext = torch.tensor(self.p.hi, dtype=torch.float64, device=dev) - self.lo
        self.dx = ext / (8 * self.root[self.grid]) / (2.0 ** self.lev)[:, None]
        self.key, self.order = torch.sort(self._key(self.grid, self.lev, self.b))
        one = lambda w: torch.stack(_conservative([torch.tensor(float(v), dtype=torch.float64, device=dev) for v in w],  # noqa: E731
                                                  self.p.gamma))
        self.inflow, self.body = one(self.p.inflow), one(self.p.body)
        if self.p.body_r > 0:
            x = [self._pos(slice(None), a, torch.arange(8, device=dev) + 0.5) for a in range(3)]
            self.inside = (x[0][:, None, None, :] ** 2 + x[1][:, None, :, None] ** 2 + x[2][:, :, None, None] ** 2
                           < self.p.body_r ** 2)
        else:
            self.inside = None

    def _pos(self, blocks, axis, cells):
        return self.lo[axis] + (8 * self.b[axis][blocks, None] + cells) * self.dx[blocks, axis, None]

    def _key(self, grid, lev, b):
        return (((grid * 16 + lev) << 14 | b[2]) << 14 | b[1]) << 14 | b[0]

    def _find(self, grid, lev, g):
        k = self._key(grid, lev, [x >> 3 for x in g])
        i = torch.searchsorted(self.key, k).clamp_max(self.nb - 1)
        return torch.where((self.key[i] == k) & (lev >= 0), self.order[i], -1)

    def _sample(self, U, grid, lev, g):
        """(state [8][N] of the cells g of level lev: copy, mean of the 8
        children, or the inflow state; which of them lie in a coarser leaf)."""
        g, fixed = list(g), torch.zeros_like(grid, dtype=torch.bool)
        for a in range(3):
            n = (self.root[grid, a] << lev) * 8
            for side, out in ((0, g[a] < 0), (1, g[a] >= n)):
                bc = self.p.bc[2 * a + side]
                if bc == W.BC_PERIODIC:
                    g[a] = torch.where(out, g[a] + (n if side == 0 else -n), g[a])
                else:
                    if bc == W.BC_INFLOW:
                        fixed = fixed | out
                    g[a] = torch.where(out, n - 1 if side else 0, g[a])
        at = lambda leaf, c: U[:, leaf.clamp_min(0), c[2] & 7, c[1] & 7, c[0] & 7]  # noqa: E731
        same = self._find(grid, lev, g)
        v = at(same, g)
        fine = torch.nonzero(self._find(grid, lev + 1, [2 * x for x in g]) >= 0).squeeze(1)
        if len(fine):
            f = [2 * x[fine] for x in g]
            leaf = self._find(grid[fine], lev[fine] + 1, f)
            v[:, fine] = sum(at(leaf, [f[0] + (o & 1), f[1] + (o >> 1 & 1), f[2] + (o >> 2)]) for o in range(8)) / 8
            same[fine] = leaf
        v[:, fixed] = self.inflow[:, None]
        return v, (same < 0) & ~fixed, g

    def _ghosts(self, U, grid, lev, g):
        v, coarse, g = self._sample(U, grid, lev, g)
        c = torch.nonzero(coarse).squeeze(1)
        if len(c):
            gr, lv, f = grid[c], lev[c] - 1, [x[c] for x in g]
            q = [x >> 1 for x in f]
            mid = self._sample(U, gr, lv, q)[0]
            acc = mid.clone()
            for a in range(3):
                lo, hi = (self._sample(U, gr, lv, [x + d if b == a else x for b, x in enumerate(q)])[0] for d in (-1, 1))
                acc += torch.where((f[a] & 1).bool(), 0.25, -0.25) * _minmod(mid - lo, hi - mid)
            v[:, c] = acc
        return v

    def _tile(self, U, n):
        """Padded tiles [8][n][12][12][12] of the blocks n (face slabs only)."""
        T = torch.ones(8, len(n), 12, 12, 12, dtype=torch.float64, device=U.device)
        T[:, :, 2:10, 2:10, 2:10] = U[:, n]
        r = torch.arange(8, device=U.device)
        for s in range(6):
            d, side = s >> 1, s & 1
            ax = [r, r, r]
            ax[d] = torch.tensor([8, 9] if side else [-2, -1], device=U.device)
            z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
            g = [(8 * self.b[a][n])[:, None] + c.reshape(-1) for a, c in enumerate((x, y, z))]
            m = g[0].shape[1]
            gr, lv = self.grid[n].repeat_interleave(m), self.lev[n].repeat_interleave(m)
            v = self._ghosts(U, gr, lv, [c.reshape(-1) for c in g])
            sl = [slice(2, 10)] * 3
            sl[2 - d] = slice(10, 12) if side else slice(0, 2)
            T[(slice(None), slice(None), *sl)] = v.reshape(8, len(n), *x.shape)
        return T

    def _b0(self, x):
        m = [float(v) for v in self.p.b0_param[:3]]
        r2 = x[0] ** 2 + x[1] ** 2 + x[2] ** 2
        mr = m[0] * x[0] + m[1] * x[1] + m[2] * x[2]
        return [(3 * mr * x[c] - m[c] * r2) / r2 ** 2.5 for c in range(3)]

    def _b0_at(self, n, d):
        """B0 on the faces normal to axis d (cell centres for d = None)."""
        if self.p.b0 != W.B0_DIPOLE:
            return None
        at = [self._pos(n, a, torch.arange(9 if a == d else 8, device="cuda") + (0.0 if a == d else 0.5)) for a in range(3)]
        x = torch.broadcast_tensors(at[0][:, None, None, :], at[1][:, None, :, None], at[2][:, :, None, None])
        return torch.stack(self._b0(x))

    def _flux(self, w, B0):
        """Physical flux, state and fast speed of face-frame primitives."""
        g = self.p.gamma
        u, b = w[1:4], w[4:7]
        Bt = b if B0 is None else b + B0
        b2 = (b * b).sum(0)
        pt = w[7] + 0.5 * b2
        U = torch.stack(_conservative(list(w), g))
        ub = (u * b).sum(0)
        F = [U[1]] + [U[1 + c] * u[0] - b[c] * Bt[0] for c in range(3)] + [u[0] * Bt[c] - Bt[0] * u[c] for c in range(3)]
        if B0 is not None:
            pt = pt + (B0 * b).sum(0)
            for c in range(3):
                F[1 + c] = F[1 + c] - B0[c] * b[0]
        F[1] = F[1] + pt
        F.append(u[0] * (U[7] + pt) - ub * Bt[0])
        return torch.stack(F), U, _fast(g, w, Bt[0], (Bt * Bt).sum(0))

    def _face(self, L, R, B0):
        (FL, UL, cl), (FR, UR, cr) = self._flux(L, B0), self._flux(R, B0)
        if self.p.flux == W.FLUX_RUSANOV:
            c = torch.maximum(L[1].abs() + cl, R[1].abs() + cr)
            return 0.5 * (FL + FR) - 0.5 * c * (UR - UL), c, (0.5 * c * (UR - UL)).abs()
        sl = torch.minimum(L[1] - cl, R[1] - cr).clamp_max(0)
        sr = torch.maximum(L[1] + cl, R[1] + cr).clamp_min(0)
        F = FL - sl / (sr - sl) * ((FR - FL) - sr * (UR - UL))
        if self.p.flux == W.FLUX_LINDE:
            m = 0.5 * (L + R)
            c2 = self.p.gamma * m[7] / m[0]
            dr = R[0] - L[0]
            q = c2.sqrt() / (c2.sqrt() + m[1].abs()) * _minmod(dr - (R[7] - L[7]) / c2, dr) * sl * sr / (sr - sl)
            F = F - q * torch.stack([torch.ones_like(q), m[1], m[2], m[3], 0 * q, 0 * q, 0 * q,
                                     0.5 * (m[1] ** 2 + m[2] ** 2 + m[3] ** 2)])
        return F, None, None

    def residual(self, U, learned):
        R = torch.empty_like(U)
        for n in torch.arange(self.nb, device=U.device).split(2048):
            w = _primitive(self._tile(U, n), self.p.gamma)
            c = w[:, :, 2:10, 2:10, 2:10]
            acc, divb, cb0 = torch.zeros_like(c), 0, []
            for d in range(3):
                ax = 4 - d
                rot = [0, 1 + d, 1 + (d + 1) % 3, 1 + (d + 2) % 3, 4 + d, 4 + (d + 1) % 3, 4 + (d + 2) % 3, 7]
                sl = [slice(2, 10)] * 3
                sl[2 - d] = slice(None)
                v = w[(slice(None), slice(None), *sl)][rot]
                df = v.diff(dim=ax)
                a, b = df.narrow(ax, 0, 10), df.narrow(ax, 1, 10)
                s = _minmod(a, b)
                if self.p.limiter == W.LIM_MC:
                    s = _minmod(2 * s, 0.5 * (a + b))
                elif self.p.limiter == W.LIM_NONE:
                    s = 0 * s
                L = v.narrow(ax, 1, 9) + 0.5 * s.narrow(ax, 0, 9)
                Rt = v.narrow(ax, 2, 9) - 0.5 * s.narrow(ax, 1, 9)
                b0 = self._b0_at(n, d)
                F, cmax, lim = self._face(L, Rt, None if b0 is None else b0[[d, (d + 1) % 3, (d + 2) % 3]])
                if learned:
                    st = [v.narrow(ax, k, 9) for k in range(4)] + [0.5 * (L + Rt)]
                    rho = 0.25 * (st[0][0] + st[1][0] + st[2][0] + st[3][0])
                    u = [rho] + [cmax] * 3 + [rho.sqrt() * cmax] * 3 + [rho * cmax ** 2]
                    u[0] = rho
                    x = torch.stack([q[k] / u[k] for q in st for k in range(8)], -1)
                    y = _mlp(self.net, x.reshape(-1, 40)).reshape(*x.shape[:-1], 8).movedim(-1, 0)
                    sc = [rho * cmax] + [rho * cmax ** 2] * 3 + [rho.sqrt() * cmax ** 2] * 3 + [rho * cmax ** 3]
                    F = F + torch.maximum(torch.minimum(y * torch.stack(sc), lim), -lim)
                h = self.dx[n, d][:, None, None, None]
                back = [rot.index(k) for k in range(8)]
                acc -= F.diff(dim=ax)[back] / h
                divb = divb + (0.5 * (L[4] + Rt[4])).diff(dim=ax - 1) / h
                if b0 is not None:
                    cb0.append(b0.diff(dim=ax) / h)
            if self.p.powell:
                b0 = self._b0_at(n, None)
                Bt = c[4:7] if b0 is None else c[4:7] + b0
                acc[1:4] -= divb * Bt
                acc[4:7] -= divb * c[1:4]
                acc[7] -= divb * (c[1:4] * c[4:7]).sum(0)
            if cb0:
                gx, gy, gz = cb0
                div = gx[0] + gy[1] + gz[2]
                cu = torch.stack([gy[2] - gz[1], gz[0] - gx[2], gx[1] - gy[0]])
                acc[1:4] += -c[4:7] * div + torch.linalg.cross(c[4:7], cu, dim=0)
            R[:, n] = acc
        return R

    def speed(self, U):
        s = torch.zeros(self.nb, 8, 8, 8, dtype=torch.float64, device=U.device)
        for n in torch.arange(self.nb, device=U.device).split(8192):
            w = _primitive(U[:, n], self.p.gamma)
            b0 = self._b0_at(n, None)
            Bt = w[4:7] if b0 is None else w[4:7] + b0
            B2 = (Bt * Bt).sum(0)
            s[n] = sum((w[1 + a].abs() + _fast(self.p.gamma, w, Bt[a], B2)) / self.dx[n, a][:, None, None, None]
                       for a in range(3))
        if self.inside is not None:
            s[self.inside] = 0
        return s

    def advance(self, U, steps, cfl):
        t = 0.0
        for _ in range(steps):
            s = self.speed(U)
            top = torch.zeros(self.ng, dtype=torch.float64, device=U.device)
            top.scatter_reduce_(0, self.grid, s.amax((1, 2, 3)), "amax")
            t += float(cfl / top[0])
            dt = (cfl / top)[self.grid][:, None, None, None]
            if self.case["local_dt"]:
                dt = torch.where(s > 0, cfl / s, 0.0)
            if self.p.rk == W.RK_MIDPOINT:
                V = self._hold(U + 0.5 * dt * self.residual(U, False))
                U = U + dt * self.residual(V, self.net is not None)
            else:
                V = self._hold(U + dt * self.residual(U, False))
                U = V if self.p.rk == W.RK_EULER else 0.5 * U + 0.5 * (V + dt * self.residual(V, False))
            U = self._hold(U)
        return U, t

    def _hold(self, U):
        if self.inside is not None:
            U[:, self.inside] = self.body[:, None]
        return U


def exact(case, seed):
    if case["kind"] == "infer":
        x = _face_rows(case["rows"], seed).to(torch.bfloat16).double()
        p = torch.from_numpy(_network(seed)).cuda().double()
        return torch.cat([_mlp(p, r) for r in x.split(1 << 18)])
    if case["kind"] == "train":
        x = _face_rows(case["rows"], seed).double()
        tgt = (0.05 * torch.tanh(x[:, 8:16] - x[:, 16:24]))
        perm = torch.randperm(case["rows"], generator=torch.Generator().manual_seed(seed)).cuda()
        batch = min(case["batch"], case["rows"])
        p = torch.from_numpy(_network(seed)).cuda().double().requires_grad_()
        opt = torch.optim.Adam([p], lr=1e-3)
        losses = []
        for s in range(case["rows"] // batch):
            i = perm[s * batch:(s + 1) * batch]
            opt.zero_grad()
            loss = ((_mlp(p, x[i]) - tgt[i]) ** 2).mean()
            loss.backward()
            opt.step()
            losses.append(loss.item())
        return {"loss": sum(losses) / len(losses), "params": p.detach()}
    probs, flat = _states(case, seed)
    net = torch.from_numpy(_network(seed)).cuda().double() if case["learned"] else None
    sizes = [8 * p.nb * 512 for p in probs]
    U = torch.cat([v.reshape(8, -1, 8, 8, 8) for v in flat.split(sizes)], 1)
    U, t = _Plain(case, probs, net).advance(U, case["steps"], 0.8)
    return {"state": torch.cat([v.reshape(-1) for v in U.split([p.nb for p in probs], 1)]), "time": t}


if __name__ == "__main__":
    for c in listed() + [draw(random.Random(k)) for k in range(6)]:
        print(c, work(c))
