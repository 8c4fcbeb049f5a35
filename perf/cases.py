"""The work a user of the framework has it do, as measurable cases.

Every case is one call sequence through the public entry points of
``paper_2508_02626_gb300.binding``, of one of these kinds:

  eval   ``Tree.eval`` on a resident tree (charges and positions fixed, evaluated again and again)
  step   one time step of a particle code on the GPU: build the tree of new positions, evaluate,
         free (a pooled context, device arrays)
  host   the same from page-locked host arrays, with the results back in page-locked host arrays
  batch  many uneven independent problems at once: build the forest, evaluate, free (device arrays)
  graph  the captured evaluation of a resident forest, replayed
  serve  a burst of requests through the serving loop, until every one is answered

The FP64 and float-float modes return their float64 results as they are.  The FP32 and MIXED
modes carry FP32 accuracy (about 1e-6) in float64 arrays, so a program that chooses them keeps
its results as float32 tensors, and so do the cases: the conversion is part of the pass.

A program keeps one context (or server) for all its solves; the contexts here are made once per
process in the same way.
"""
import math

import numpy as np
import torch

from paper_2508_02626_gb300 import binding as B

UNIT_CUBE = np.array([0.0, 0.0, 0.0, 1.0])
POOL_BYTES = 16 << 30
# pairs that the direct sum of `exact` handles in well under 20 seconds
EXACT_PAIRS = 9e10


def listed():
    return [
        # one small FP64 solve of 10,000 particles, order 6, 512 leaves: the plain configuration
        # checked against the direct sum; launches and latency count
        {"name": "eval-uniform-1e4-p6-fp64", "kind": "eval", "dist": "uniform", "n": 10_000, "depth": 3, "leaf": 0,
         "order": 6, "precision": "fp64"},
        # the smallest useful call: a time step of a few thousand particles at low order
        {"name": "step-uniform-3001-p4-fp32", "kind": "step", "dist": "uniform", "n": 3001, "depth": 2, "leaf": 0,
         "order": 4, "precision": "fp32"},
        # the headline configuration: a million uniform particles, depth 5, order 8
        {"name": "eval-uniform-1e6-p8-fp32", "kind": "eval", "dist": "uniform", "n": 1_000_000, "depth": 5, "leaf": 0,
         "order": 8, "precision": "fp32"},
        # the same in the mode that keeps its shifts in FP64
        {"name": "eval-uniform-1e6-p8-mixed", "kind": "eval", "dist": "uniform", "n": 1_000_000, "depth": 5,
         "leaf": 0, "order": 8, "precision": "mixed"},
        # full double precision at an odd medium size (uneven leaves), order 8
        {"name": "eval-uniform-200003-p8-fp64", "kind": "eval", "dist": "uniform", "n": 200_003, "depth": 4,
         "leaf": 0, "order": 8, "precision": "fp64"},
        # FP64-level accuracy on the FP32 pipe (float-float)
        {"name": "eval-uniform-200003-p8-ff", "kind": "eval", "dist": "uniform", "n": 200_003, "depth": 4, "leaf": 0,
         "order": 8, "precision": "ff"},
        # the clustered configuration: 4 million particles in 32 Gaussian clusters, at most 64 per
        # leaf, order 10, mixed precision; the largest solve
        {"name": "eval-clustered-4e6-p10-mixed", "kind": "eval", "dist": "clustered", "n": 4_000_000, "depth": -1,
         "leaf": 64, "order": 10, "precision": "mixed"},
        # a time step on the paper's own shape (a Gaussian blob, order 4, at most 128 per leaf):
        # the adaptive build and the evaluation together
        {"name": "step-gaussian-1e6-p4-fp32", "kind": "step", "dist": "gaussian", "n": 1_000_000, "depth": -1,
         "leaf": 128, "order": 4, "precision": "fp32"},
        # the paper's accuracy study at high order: an adaptive tree in double precision
        {"name": "eval-gaussian-100003-p8-fp64", "kind": "eval", "dist": "gaussian", "n": 100_003, "depth": -1,
         "leaf": 256, "order": 8, "precision": "fp64"},
        # end to end from a host program: copies in, tree build, evaluation, results out
        {"name": "host-uniform-1e6-p8-fp32", "kind": "host", "dist": "uniform", "n": 1_000_000, "depth": 5, "leaf": 0,
         "order": 8, "precision": "fp32"},
        # the batched configuration: uneven solves of 1e3 to 1e5 particles, order 6, one captured graph
        {"name": "graph-64-problems-p6-fp32", "kind": "graph", "dist": "mix", "n": 64, "lo": 1000, "hi": 100_000,
         "leaf": 128, "order": 6, "precision": "fp32"},
        # the serving configuration: requests of 1e3 to 1e6 particles, orders 4, 6 and 8
        {"name": "serve-48-requests-fp32", "kind": "serve", "dist": "mix", "n": 48, "lo": 1000, "hi": 1_000_000,
         "leaf": 64, "order": 0, "precision": "fp32"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "step", "step", "host", "batch", "graph", "serve"])
    if kind in ("batch", "graph"):
        return {"kind": kind, "dist": "mix", "n": _log_uniform(rng, 4, 128), "lo": _log_uniform(rng, 500, 4000),
                "hi": _log_uniform(rng, 8000, 100_000), "leaf": rng.choice([32, 64, 100, 128, 256]),
                "order": rng.choice([4, 5, 6, 8]), "precision": rng.choice(["fp32", "fp32", "mixed"])}
    if kind == "serve":
        return {"kind": kind, "dist": "mix", "n": _log_uniform(rng, 8, 48), "lo": _log_uniform(rng, 500, 4000),
                "hi": _log_uniform(rng, 50_000, 1_000_000), "leaf": rng.choice([48, 64, 128]), "order": 0,
                "precision": "fp32"}
    precision = rng.choice(["fp32", "fp32", "fp32", "mixed", "fp64", "ff"])
    if kind == "host":
        precision = rng.choice(["fp32", "mixed"])
    order = rng.choice([2, 3, 4, 5, 6, 7, 8, 8, 9, 10])
    top = 3_000_000 if precision in ("fp32", "mixed") else 200_000
    n = _log_uniform(rng, 2000, top)
    dist = "uniform" if precision == "ff" else rng.choice(["uniform", "uniform", "clustered", "gaussian"])
    if dist == "uniform":
        # about 20 to 160 particles per leaf
        depth = max(2, int(round(math.log(n / rng.uniform(30.0, 60.0)) / math.log(8.0))))
        leaf = 0
    else:
        depth = -1
        leaf = rng.choice([32, 64, 100, 128]) if order <= 4 else rng.choice([64, 128, 200, 256])
    return {"kind": kind, "dist": dist, "n": n, "depth": depth, "leaf": leaf, "order": order, "precision": precision}


# ---- inputs -----------------------------------------------------------------------------------
def _members(case):
    """(n, dist, order) of each problem of a batch or burst: sizes at the quantiles of a
    log-uniform law, shapes in turn, in a fixed shuffled order."""
    k = case["n"]
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    perm = np.random.default_rng(97).permutation(k)
    out = []
    for i in perm:
        n = int(round(math.exp(lo + (i + 0.5) / k * (hi - lo))))
        out.append((n, "uniform" if i % 2 == 0 else "clustered", case["order"] or (4, 6, 8)[i % 3]))
    return out


def _points(dist, n, gen):
    dev = gen.device
    if dist == "uniform":
        x = torch.rand(n, 3, dtype=torch.float64, device=dev, generator=gen)
    elif dist == "gaussian":
        x = torch.randn(n, 3, dtype=torch.float64, device=dev, generator=gen)
    else:  # 32 isotropic Gaussian clusters, sigma in [0.02, 0.1], centres in the unit cube
        c = torch.rand(32, 3, dtype=torch.float64, device=dev, generator=gen)
        s = 0.02 + 0.08 * torch.rand(32, dtype=torch.float64, device=dev, generator=gen)
        k = torch.randint(0, 32, (n,), device=dev, generator=gen)
        x = c[k] + s[k, None] * torch.randn(n, 3, dtype=torch.float64, device=dev, generator=gen)
    return x


def _inputs(case, seed):
    """(xyz, q, offsets) on the GPU; the problems of a batch end to end."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["dist"] == "mix":
        mem = _members(case)
        xyz = torch.cat([_points(d, n, gen) for n, d, _ in mem])
        offs = np.cumsum([0] + [n for n, _, _ in mem])
        q = 2.0 * torch.rand(len(xyz), dtype=torch.float64, device="cuda", generator=gen) - 1.0
        return xyz, q, offs
    n = case["n"]
    xyz = _points(case["dist"], n, gen)
    if case["dist"] == "uniform":
        q = 2.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    else:
        q = torch.ones(n, dtype=torch.float64, device="cuda")
    return xyz, q, np.array([0, n])


# ---- what a program keeps ---------------------------------------------------------------------
_kept = {}


def _context(pooled):
    key = "pool" if pooled else "plain"
    if key not in _kept:
        B.load()
        _kept[key] = B.Context(0, pool_bytes=POOL_BYTES) if pooled else B.Context(0)
    return _kept[key]


def _server():
    if "server" not in _kept:
        B.load()
        _kept["server"] = B.Server(0, pool_bytes=POOL_BYTES, slots=4, max_batch=32, max_job_particles=1 << 21)
    return _kept["server"]


class State:
    """One case's inputs, output buffers and handles; a resident tree is freed with it."""

    def __init__(self, case, seed):
        self.case = case
        self.kind = case["kind"]
        self.order = case["order"]
        self.precision = case["precision"]
        self.narrow = self.precision in ("fp32", "mixed")
        self.tree = self.graph = None
        self.xyz, self.q, self.offsets = _inputs(case, seed)
        n = len(self.q)
        self.phi = torch.empty(n, dtype=torch.float64, device="cuda")
        self.field = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        self.domain = UNIT_CUBE if case["dist"] == "uniform" else None
        torch.cuda.synchronize()  # the inputs are complete before another stream or context reads them
        if self.kind == "eval":
            self.ctx = _context(False)
            self.tree = self.ctx.build_tree(self.xyz, self.q, domain=self.domain, uniform_depth=case["depth"],
                                            max_leaf=case["leaf"])
        elif self.kind == "graph":
            self.ctx = _context(False)
            self.tree = self.ctx.build_forest(self.xyz, self.q, self.offsets, max_leaf=case["leaf"])
            self.graph = self.tree.graph(self.order, self.phi, self.field, precision=self.precision)
        elif self.kind == "serve":
            self.server = _server()
            self.xyz, self.q = self.xyz.cpu().pin_memory(), self.q.cpu().pin_memory()
        else:
            self.ctx = _context(True)
            if self.kind == "host":
                self.xyz, self.q = self.xyz.cpu().pin_memory(), self.q.cpu().pin_memory()
                self.host_phi = torch.empty(n, dtype=torch.float32).pin_memory()
                self.host_field = torch.empty((n, 3), dtype=torch.float32).pin_memory()

    def results(self):
        if self.narrow:
            return {"phi": self.phi.float(), "field": self.field.float()}
        return {"phi": self.phi, "field": self.field}

    def __del__(self):
        if self.graph is not None:
            torch.cuda.synchronize()
            self.graph.free()
        if self.tree is not None:
            self.tree.free()


def prepare(case, seed):
    return State(case, seed)


def _solve(s):
    """Build, evaluate, wait (dafmm_sync reports what the kernels recorded), free."""
    case = s.case
    if s.kind == "batch":
        tree = s.ctx.build_forest(s.xyz, s.q, s.offsets, max_leaf=case["leaf"])
    else:
        tree = s.ctx.build_tree(s.xyz, s.q, domain=s.domain, uniform_depth=case["depth"], max_leaf=case["leaf"])
    tree.eval(s.order, s.phi, s.field, precision=s.precision)
    if s.kind == "host":
        s.host_phi.copy_(s.phi, non_blocking=True)
        s.host_field.copy_(s.field, non_blocking=True)
        out = {"phi": s.host_phi, "field": s.host_field}
    else:
        out = s.results()
    B.dafmm_sync(s.ctx.h)
    tree.free()
    return out


def run(s):
    if s.kind == "eval":
        s.tree.eval(s.order, s.phi, s.field, precision=s.precision)
        return s.results()
    if s.kind == "graph":
        s.graph.launch()
        return s.results()
    if s.kind == "serve":
        # requests arrive in page-locked host arrays; the results are wanted on the GPU
        prec = B.PRECISIONS[s.precision]
        ids = []
        for (n, _, order), o in zip(_members(s.case), s.offsets):
            e = o + n
            ids.append(B.dafmm_server_submit(s.server.h, s.xyz[o:e], s.q[o:e], order, prec, s.case["leaf"],
                                             s.phi[o:e], s.field[o:e]))
        for i in ids:
            status, _ = B.dafmm_server_wait(s.server.h, i)
            if status != B.DAFMM_OK:
                raise B.DafmmError(status, B.dafmm_server_last_error(s.server.h))
        return s.results()
    return _solve(s)


# ---- what a pass cannot do without --------------------------------------------------------------
def _problem_work(n, dist, order, depth, leaf):
    """FLOPs of one FMM solve: the near field (about 18 per pair), the far field's pairwise
    translations in the (p + 1)^2 harmonic coefficients, and the particle operators."""
    nh = (order + 1) ** 2
    if dist == "uniform" and depth >= 0:
        boxes = 8.0 ** depth
        side = 2.0 ** depth
        near = n * (n / boxes) * (3.0 - 2.0 / side) ** 3
        pairs = sum(8.0 ** l * min(189.0, 8.0 ** l) for l in range(2, depth + 1))
    else:
        occ = leaf / 2.0
        near = min(27.0 * n * occ, float(n) * n)
        pairs = 189.0 * (n / occ) * 8.0 / 7.0 if n > 64 * leaf else 0.0
        pairs *= 0.5  # clustered and Gaussian boxes lack part of their neighbours
    return 18.0 * near + 2.0 * nh * nh * pairs + 8.0 * nh * n


def work(case):
    if case["dist"] == "mix":
        mem = _members(case)
        total = sum(n for n, _, _ in mem)
        flops = sum(_problem_work(n, "adaptive", p, -1, case["leaf"]) for n, _, p in mem)
    else:
        total = case["n"]
        flops = _problem_work(total, case["dist"], case["order"], case["depth"], case["leaf"])
    out = 16 if case["precision"] in ("fp32", "mixed") else 32
    return {"bytes": float(total) * (32 + out), "flops": flops}


# ---- the same in 64 bits --------------------------------------------------------------------------
def _direct(xyz, q):
    """phi_i = sum_j q_j / r_ij and E_i = sum_j q_j (x_i - x_j) / r_ij^3 in float64, j != i."""
    n = len(q)
    phi = torch.empty(n, dtype=torch.float64, device="cuda")
    field = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    xs = [xyz[:, d].contiguous() for d in range(3)]
    block = max(1, (1 << 26) // n)
    for i in range(0, n, block):
        j = min(n, i + block)
        d = [x[i:j, None] - x[None, :] for x in xs]
        w = (d[0] * d[0]).addcmul_(d[1], d[1]).addcmul_(d[2], d[2]).rsqrt_()
        w.masked_fill_(torch.isinf(w), 0.0)  # the particle itself, and coincident ones
        phi[i:j] = w @ q
        w.mul_(w * w).mul_(q)
        for k in range(3):
            field[i:j, k] = d[k].mul_(w).sum(1)
    return phi, field


def exact(case, seed):
    if case["dist"] == "mix":
        sizes = [n for n, _, _ in _members(case)]
    else:
        sizes = [case["n"]]
    if sum(float(n) * n for n in sizes) > EXACT_PAIRS:
        return None
    xyz, q, offs = _inputs(case, seed)
    parts = [_direct(xyz[a:b], q[a:b]) for a, b in zip(offs[:-1], offs[1:])]
    return {"phi": torch.cat([p for p, _ in parts]), "field": torch.cat([f for _, f in parts])}
