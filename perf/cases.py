"""What the speed of this framework is measured on: factorizations and solves as
a user's program has them done, through the package's Python entry points.

Matrices are the grid problems of this repository's configurations: 2D 5-point
and 3D 7-point Laplacians with a small reaction term, and 2D 5-point / 3D
27-point diffusion with log-normal conductivity (contrast 1e2 and 1e4), ordered
by geometric nested dissection.  Right-hand sides come from a manufactured
solution, uniform in (-1, 1): coefficients are multiples of 2^-24 and the
solution's entries of 2^-15, so that b = A x holds without rounding and the
exact solution is known.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from gridgen import geometric_nd
from paper_1608_00044_gb300 import FP32, FP64, FP64_TC, TF32, TF32X3, SparseCholesky, hostplan, spchol

PRECISIONS = {"fp64": FP64, "fp32": FP32, "tf32": TF32, "tf32x3": TF32X3, "fp64_tc": FP64_TC}
# (max_width, relax_zeros, tile_rows): the library's defaults, and the plan its
# autotuner picks for batches of small grids in either precision
DEFAULT_PLAN = "64,4,0"
BATCH_PLAN = "32,16,32"


def _single(name, kind, dims, precision, nrhs, **more):
    case = {"name": name, "what": "factor_solve", "kind": kind, "dims": "x".join(map(str, dims)),
            "precision": precision, "nrhs": nrhs, "deterministic": 0, "host": False}
    case.update(more)
    return case


def _batch(name, precision, count, lo, hi, nrhs=1):
    return {"name": name, "what": "batch", "kind": "diff2d", "precision": precision, "nrhs": nrhs, "count": count,
            "lo": lo, "hi": hi}


def listed():
    return [
        # one small 2D system, the configuration that is all latency
        _single("lap2d_64", "lap2d", (64, 64), "fp64", 1),
        # a request of the serving stream: a ragged 2D system in host memory, the
        # result back in host memory
        _single("diff2d_181x203_host", "diff2d", (181, 203), "fp64", 5, host=True),
        # a request of the serving stream: a middling, ragged 3D system
        _single("lap3d_31x34x29", "lap3d", (31, 34, 29), "fp64", 4),
        # the headline configuration: the 64^3 Laplacian with 8 right-hand sides
        _single("lap3d_64", "lap3d", (64, 64, 64), "fp64", 8),
        # the same on the BF16 tensor cores
        _single("lap3d_64_fp64_tc", "lap3d", (64, 64, 64), "fp64_tc", 8),
        # new right-hand sides for a factor that is resident: a time step or a
        # serving repeat; large with 8, and middling and ragged with 16
        _single("lap3d_64_resolve", "lap3d", (64, 64, 64), "fp64", 8, what="resolve"),
        _single("lap3d_33x41x37_resolve", "lap3d", (33, 41, 37), "fp64", 16, what="resolve"),
        # the mixed-precision configuration (FP32 factor, refined to 1e-12), and a
        # smaller ragged one with split-TF32 updates
        _single("diff3d_48_fp32", "diff3d", (48, 48, 48), "fp32", 1),
        _single("diff3d_35x31x38_tf32x3", "diff3d", (35, 31, 38), "tf32x3", 3),
        # bitwise reproducible by fan-in aggregation
        _single("lap3d_27_fanin", "lap3d", (27, 27, 27), "fp64", 2, deterministic=2),
        # the batch configuration, in both precisions: 512 grids of sides 16..128
        _batch("batch_512_fp64", "fp64", 512, 16, 128),
        _batch("batch_512_fp32", "fp32", 512, 16, 128),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, int(lo * math.exp(rng.random() * math.log((hi + 1) / lo))))

    def box(ndim, side, most):
        return tuple(max(4, min(most, round(side * rng.uniform(0.8, 1.25)))) for _ in range(ndim))

    roll = rng.random()
    if roll < 0.2:  # batches of small grids
        lo = log_int(8, 64)
        return {"what": "batch", "kind": rng.choice(["diff2d", "lap2d"]), "precision": rng.choice(["fp64", "fp32"]),
                "nrhs": rng.choice([1, 1, 2, 5]), "count": log_int(16, 500), "lo": lo, "hi": rng.randint(lo, 128)}
    deterministic = 2 if roll < 0.3 else 0
    kind = rng.choice(["lap2d", "diff2d", "lap3d", "lap3d", "diff3d", "diff3d"])
    precision = "fp64" if deterministic else rng.choice(["fp64", "fp64", "fp64", "fp32", "tf32x3", "tf32", "fp64_tc"])
    if precision == "tf32" and kind in ("lap2d", "diff2d"):
        precision = "fp32"  # a TF32 factor is too coarse to refine a large 2D grid with
    if kind in ("lap2d", "diff2d"):
        dims = box(2, log_int(16, 256), 256)
    else:
        most = 28 if deterministic else 62 if kind == "lap3d" else 47
        dims = box(3, log_int(8, most), most)
    what = rng.choice(["factor_solve", "factor_solve", "resolve"])
    host = what == "factor_solve" and rng.random() < 0.25
    case = _single("", kind, dims, precision, rng.choice([1, 1, 2, 3, 4, 7, 8, 11, 16]), what=what, host=host,
                   deterministic=deterministic)
    del case["name"]
    return case


class _Grid:
    """The pattern of one grid operator (lower triangle, CSC, C order of the points) and its ordering."""

    def __init__(self, kind, dims):
        self.kind, self.dims, self.n = kind, dims, math.prod(dims)
        ids = np.arange(self.n, dtype=np.int64).reshape(dims)
        box = kind == "diff3d"  # 27 points: every neighbour of the box around a point; else its faces
        self.edges = []  # (weight, lower ids, higher ids) of each stencil direction
        self.ghost = np.zeros(self.n)  # weight of the couplings that leave the grid (Dirichlet)
        for off in itertools.product((-1, 0, 1), repeat=len(dims)):
            faces = sum(map(abs, off))
            if faces == 0 or (faces > 1 and not box):
                continue
            weight = 0.5 ** (faces - 1)
            at = ids[tuple(slice(max(0, -d), m - max(0, d)) for d, m in zip(off, dims))].ravel()
            to = ids[tuple(slice(max(0, d), m - max(0, -d)) for d, m in zip(off, dims))].ravel()
            outside = np.ones(self.n, bool)
            outside[at] = False
            self.ghost[outside] += weight
            if next(d for d in off if d) > 0:
                self.edges.append((weight, at, to))
        cols = np.concatenate([ids.ravel()] + [u for _, u, _ in self.edges])
        rows = np.concatenate([ids.ravel()] + [v for _, _, v in self.edges])
        self.order = np.lexsort((rows, cols))
        self.colptr = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=self.n))]).astype(np.int64)
        self.rowind = rows[self.order].astype(np.int32)
        self.perm = geometric_nd(dims)

    def numbers(self, nrhs, rng):
        """(values, x, b): one matrix of this pattern, nrhs solutions (a row each) and their right-hand sides."""
        n, unit = self.n, 2.0 ** -24
        if self.kind in ("lap2d", "lap3d"):
            off = [np.full(u.size, -1.0) for _, u, _ in self.edges]
            diag = 2.0 * len(self.dims) + rng.integers(0, 16, n) / 1024.0
        else:
            sigma = 2.0 if self.kind == "diff3d" else 1.0
            k = np.exp(sigma * np.clip(rng.standard_normal(n), -2.303, 2.303))
            off, diag = [], np.ceil(self.ghost * k / unit) * unit
            for weight, u, v in self.edges:
                w = np.ceil(weight * 2.0 * k[u] * k[v] / (k[u] + k[v]) / unit) * unit
                off.append(-w)
                diag = diag + np.bincount(u, w, n) + np.bincount(v, w, n)
        x = rng.integers(-(2 ** 15) + 1, 2 ** 15, (nrhs, n)) / 2.0 ** 15
        b = diag * x
        for (_, u, v), a in zip(self.edges, off):
            for r in range(nrhs):
                b[r] += np.bincount(v, a * x[r][u], n) + np.bincount(u, a * x[r][v], n)
        return np.concatenate([diag] + off)[self.order], x, b


@functools.lru_cache(maxsize=256)
def _grid(kind, dims):
    return _Grid(kind, dims)


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _sides(case):
    """The grid sides of a batch, uniform in [lo, hi]: the same for every seed, as a plan is kept for."""
    return np.random.default_rng(1234).integers(case["lo"], case["hi"] + 1, case["count"])


def _numbers(case, seed):
    rng = np.random.default_rng(seed)
    if case["what"] == "batch":
        return [_grid(case["kind"], (int(s), int(s))).numbers(case["nrhs"], rng) for s in _sides(case)]
    return _grid(case["kind"], _dims(case)).numbers(case["nrhs"], rng)


def _options(case, plan):
    width, relax, tile = (int(v) for v in plan.split(","))
    return {"precision": PRECISIONS[case["precision"]], "max_width": width, "relax_zeros": relax, "tile_rows": tile,
            "deterministic": case.get("deterministic", 0)}


class _Batch:
    """A batch handle that is given back with its owner."""

    def __init__(self, grids, options):
        self.h = None
        self.h = spchol.batch_analyze([g.n for g in grids], [g.colptr for g in grids], [g.rowind for g in grids],
                                      [g.perm for g in grids], spchol.default_options(**options))

    def __del__(self):
        if self.h is not None:
            spchol.destroy(self.h)


def prepare(case, seed):
    numbers = _numbers(case, seed)
    if case["what"] == "batch":
        grids = [_grid(case["kind"], (int(s), int(s))) for s in _sides(case)]
        # every matrix's values, right-hand sides and solutions lie one after another in one buffer each
        values = torch.from_numpy(np.concatenate([v for v, _, _ in numbers])).cuda()
        b = torch.from_numpy(np.concatenate([b.ravel() for _, _, b in numbers])).cuda()
        x = torch.empty_like(b)
        ns = [g.n for g in grids]
        return {"case": case, "plan": _Batch(grids, _options(case, BATCH_PLAN)), "ns": ns, "b": b, "x": x,
                "values": values.split([len(v) for v, _, _ in numbers]), "xs": x.split([n * case["nrhs"] for n in ns])}
    grid = _grid(case["kind"], _dims(case))
    values, _, b = numbers
    plan = SparseCholesky(grid.n, grid.colptr, grid.rowind, grid.perm, **_options(case, DEFAULT_PLAN))
    state = {"case": case, "plan": plan}
    if case["host"]:
        state["values"], state["b"] = values, np.asfortranarray(b.T)
    else:
        state["values"], state["b"] = torch.from_numpy(values).cuda(), torch.from_numpy(b).cuda()
    if case["what"] == "resolve":
        _positive(plan.factorize(state["values"]))
    return state


def _positive(column):
    if column != 0:
        raise RuntimeError(f"the matrix is not positive definite at column {column}")


def run(state):
    case, plan = state["case"], state["plan"]
    if case["what"] == "batch":
        _positive(spchol.batch_factorize(plan.h, state["values"]))
        state["x"].copy_(state["b"])
        spchol.batch_solve(plan.h, state["xs"], state["ns"], [case["nrhs"]] * case["count"])
        return state["x"]
    if case["what"] == "factor_solve":
        _positive(plan.factorize(state["values"]))
    x = state["b"].copy(order="F") if case["host"] else state["b"].clone()
    return plan.solve(x)


@functools.lru_cache(maxsize=256)
def _counts(kind, dims):
    """(entries of A's lower triangle, entries of L, sum over L's columns of entries^2)."""
    grid = _grid(kind, dims)
    plan = hostplan.HostPlan(grid.n, grid.colptr, grid.rowind, grid.perm)
    try:
        return int(grid.colptr[-1]), int(plan.scalars()["nnz_l"]), plan.flops
    finally:
        plan.close()


def work(case):
    """The factorization reads A and writes L (4 bytes an entry in the FP32-panel
    modes), a solve reads L (here once, though it has two directions), and reads
    b and writes x; 2 flops per entry of L, direction and right-hand side."""
    if case["what"] == "batch":
        grids = [(case["kind"], (int(s), int(s))) for s in _sides(case)]
    else:
        grids = [(case["kind"], _dims(case))]
    entry = 8 if case["precision"] in ("fp64", "fp64_tc") else 4
    total_bytes, flops = 0.0, 0.0
    for kind, dims in grids:
        nnz_a, nnz_l, factor_flops = _counts(kind, dims)
        n = math.prod(dims)
        total_bytes += entry * nnz_l + 16 * n * case["nrhs"]
        flops += 4.0 * nnz_l * case["nrhs"]
        if case["what"] != "resolve":
            total_bytes += 8 * nnz_a
            flops += factor_flops
    return {"bytes": total_bytes, "flops": flops}


def exact(case, seed):
    numbers = _numbers(case, seed)
    if case["what"] == "batch":
        return torch.from_numpy(np.concatenate([x.ravel() for _, x, _ in numbers]))
    _, x, _ = numbers
    return np.asfortranarray(x.T) if case["host"] else torch.from_numpy(x)
