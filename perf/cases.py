"""Work that users of this library have it do, as measurable cases.

Every case goes through a public entry point of ``paper_2403_03571_gb300.capi``
and stands for one use of it, from a single evaluation of a small 2D diagram
to a weight solve of 10^4 seeds on 512^3 voxels.  Inputs follow the laws of the
repository's workloads (``synth.py``): seeds uniform in the unit box without
close pairs, lognormal or alpha-law anisotropy, equal or lognormal volumes; they
are drawn on the GPU, since they are made many times.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2403_03571_gb300 import capi, synth, warmstart

F64 = torch.float64
PRECISION = {"fp32": capi.APD_FP32, "tc_tf32": capi.APD_TC_TF32, "tc_bf16": capi.APD_TC_BF16}
MOMENTS = {2: 6, 3: 10}   # moment words per cell
FEATURES = {2: 6, 3: 10}  # features of the expanded quadratic


def _res(text):
    return tuple(int(r) for r in text.split("x"))


def _text(res):
    return "x".join(str(int(r)) for r in res)


def _eq210(dim, n):
    """Pixels per axis that eq. (2.10) asks for n equal volumes at 1 %."""
    return synth.required_resolution(dim, 1.0 / n)


def listed():
    return [
        # one label map of a small 2D diagram with default settings: the smallest call, all latency
        {"name": "assign_2d_n25", "kind": "assign", "dim": 2, "n": 25, "res": "100x100", "alpha": 0.0,
         "precision": "fp32", "prune": False, "weighted": False},
        # the paper's runtime test (a) at its largest 2D point: labels, W = 0, odd resolution
        {"name": "assign_2d_n5000", "kind": "assign", "dim": 2, "n": 5000, "res": "1415x1415", "alpha": 0.3,
         "precision": "tc_tf32", "prune": True, "weighted": False},
        # runtime test (a) at its largest 3D point with strongly anisotropic grains
        {"name": "assign_3d_n10000_a07", "kind": "assign", "dim": 3, "n": 10000, "res": "200x200x200", "alpha": 0.7,
         "precision": "fp32", "prune": True, "weighted": False},
        # one evaluation of the dual and its gradient, for a caller's own optimiser, on the benchmark's grid
        {"name": "dual_3d_n1000", "kind": "dual", "dim": 3, "n": 1000, "res": "256x256x256", "alpha": -1.0,
         "precision": "tc_tf32", "prune": True},
        # cell volumes and centroids with default settings (the dense sweep of Algorithm 1) on a ragged box
        {"name": "moments_3d_n700_dense", "kind": "moments", "dim": 3, "n": 700, "res": "203x190x161", "alpha": -1.0,
         "precision": "fp32", "prune": False},
        # the smallest weight solve: 20 equal grains
        {"name": "solve_2d_n20", "kind": "solve", "dim": 2, "n": 20, "res": "256x256", "alpha": -1.0, "equal": True,
         "precision": "tc_tf32", "prune": True, "multires": True},
        # the largest: 10^4 grains on 512^3 voxels, coarse to fine
        {"name": "solve_3d_n10000", "kind": "solve", "dim": 3, "n": 10000, "res": "512x512x512", "alpha": -1.0,
         "equal": False, "precision": "tc_tf32", "prune": True, "multires": True},
        # the benchmark: Algorithm 3 with five Lloyd steps, coarse-to-fine solves, learned first start
        {"name": "lloyd_3d_n1000", "kind": "lloyd", "dim": 3, "n": 1000, "res": "256x256x256", "rounds": 5,
         "precision": "tc_tf32", "prune": True},
        # many small diagrams at once (parameter studies): a batch with learned starts
        {"name": "batch_2d_48", "kind": "batch", "dim": 2, "count": 48, "n_lo": 50, "n_hi": 2000},
        # a non-uniform discretisation: labels and moments of scattered sample points with measures
        {"name": "points_3d_n1000", "kind": "points", "dim": 3, "n": 1000, "points": 4000003, "dual": False},
        # the dual on a two-level grid whose boundary voxels are refined
        {"name": "masked_3d_n1000", "kind": "masked", "dim": 3, "n": 1000, "res": "128x128x128", "refine": 2},
        # one training step (forward, backward, Adam) of the warm-start network on whole instances
        {"name": "train_3d_6000", "kind": "train", "dim": 3, "n": 1000, "instances": 6},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ragged(rng, dim, lo, hi):
    """A resolution per axis: around one size, each axis its own."""
    m = _log(rng, lo, hi)
    return _text(max(8, int(round(m * rng.uniform(0.8, 1.0)))) for _ in range(dim))


def draw(rng):
    kind = rng.choice(["assign", "assign", "dual", "moments", "solve", "solve", "lloyd", "batch", "points", "masked",
                       "train"])
    dim = rng.choice([2, 3])
    prune = rng.random() < 0.75
    precision = rng.choice(["fp32", "tc_tf32"]) if prune else "fp32"
    if kind == "assign":  # the grid of runs (a) of the paper
        n = _log(rng, 25, 5000) if dim == 2 else _log(rng, 50, 10000)
        return {"kind": kind, "dim": dim, "n": n, "res": _text([_eq210(dim, n)] * dim),
                "alpha": rng.choice([0.0, 0.3, 0.7]), "precision": precision, "prune": prune,
                "weighted": rng.random() < 0.5}
    if kind in ("dual", "moments"):
        n = _log(rng, 20, 5000)
        res = _ragged(rng, 2, 100, 3000) if dim == 2 else _ragged(rng, 3, 32, 320)
        return {"kind": kind, "dim": dim, "n": n, "res": res, "alpha": rng.choice([-1.0, 0.3]),
                "precision": precision, "prune": prune}
    if kind == "solve":
        n = _log(rng, 20, 1500) if dim == 2 else _log(rng, 50, 3000)
        m = _eq210(dim, n)
        m = int(m * rng.uniform(1.0, 1.6)) + 1
        return {"kind": kind, "dim": dim, "n": n, "res": _text([m] * dim), "alpha": -1.0,
                "equal": rng.random() < 0.5, "precision": precision if prune else "tc_tf32", "prune": True,
                "multires": rng.random() < 0.6}
    if kind == "lloyd":
        n = _log(rng, 50, 1000)
        m = int(_eq210(dim, n) * rng.uniform(1.3, 1.7)) + 1
        return {"kind": kind, "dim": dim, "n": n, "res": _text([m] * dim), "rounds": rng.randint(1, 5),
                "precision": "tc_tf32", "prune": True}
    if kind == "batch":
        if dim == 2:
            return {"kind": kind, "dim": 2, "count": rng.randint(8, 40), "n_lo": 50, "n_hi": rng.choice([300, 800])}
        return {"kind": kind, "dim": 3, "count": rng.randint(4, 12), "n_lo": 50, "n_hi": rng.choice([200, 500])}
    if kind == "points":
        return {"kind": kind, "dim": dim, "n": _log(rng, 20, 3000), "points": _log(rng, 5000, 6000000),
                "dual": rng.random() < 0.5}
    if kind == "masked":
        r = rng.choice([2, 3, 4])
        res = _ragged(rng, 2, 64, 1024) if dim == 2 else _ragged(rng, 3, 32, 300 // r)
        return {"kind": kind, "dim": dim, "n": _log(rng, 20, 1500), "res": res, "refine": r}
    return {"kind": "train", "dim": dim, "n": _log(rng, 100, 2000), "instances": rng.randint(2, 10)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 11)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, dtype=F64, device="cuda")


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=F64, device="cuda")


def _seeds(g, n, dim):
    """Uniform seeds in the unit box, none within 0.2 n^(-1/dim) of an earlier one."""
    m = n + n // 2 + 32
    p = _rand(g, m, dim)
    r2 = (0.2 * n ** (-1.0 / dim)) ** 2
    keep = torch.empty(m, dtype=torch.bool, device="cuda")
    for a in range(0, m, 2048):
        b = min(m, a + 2048)
        d2 = ((p[a:b, None, :] - p[None, :b, :]) ** 2).sum(-1)
        near = (d2 < r2) & (torch.arange(b, device="cuda")[None, :] < torch.arange(a, b, device="cuda")[:, None])
        keep[a:b] = ~near.any(1)
    return p[keep][:n].contiguous()


def _rot2(theta, d0, d1):
    c, s = torch.cos(theta), torch.sin(theta)
    off = c * s * (d0 - d1)
    return torch.stack([c * c * d0 + s * s * d1, off, off, s * s * d0 + c * c * d1], -1).reshape(-1, 2, 2)


def _anisotropy(g, n, dim, alpha):
    """alpha < 0: the lognormal law (sigma 0.3); else the alpha law of the paper's runtime tests."""
    if dim == 2:
        theta = math.pi * _rand(g, n)
        if alpha < 0:
            a = torch.exp(0.3 * _randn(g, n))
            return _rot2(theta, a, 1.0 / a).contiguous()
        a = 1.0 - alpha * _rand(g, n)
        return _rot2(theta, a ** 2, a ** -2).contiguous()
    q = _randn(g, n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    x, y, z, w = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).reshape(n, 3, 3)
    if alpha < 0:
        s = torch.exp(0.3 * _randn(g, n, 3))
        s = s / s.prod(1, keepdim=True) ** (1.0 / 3.0)
    else:
        a = 1.0 - alpha * _rand(g, n)
        b = (1.0 - alpha) + (1.0 / (1.0 - alpha) - (1.0 - alpha)) * _rand(g, n)
        s = torch.stack([a, b, 1.0 / (a * b)], 1) ** -2
    A = torch.einsum("nij,nj,nkj->nik", R, s, R)
    return (0.5 * (A + A.transpose(1, 2))).contiguous()


def _volumes(g, n, equal, measure=1.0):
    if equal:
        return torch.full((n,), measure / n, dtype=F64, device="cuda")
    v = torch.exp(0.5 * _randn(g, n))
    return (v * (measure / v.sum())).contiguous()


def _weights(g, n, dim):
    """Weights of the size that a solve ends with."""
    return (0.3 * _randn(g, n) * n ** (-2.0 / dim)).contiguous()


class _Inst:
    """What warmstart.predict reads of an instance."""

    def __init__(self, n, grid):
        self.n, self.grid = n, grid


def _batch_sizes(case):
    """Seed counts of a batch, log-uniform: the same for every draw of its inputs."""
    r = np.random.Generator(np.random.PCG64(77 + case["count"]))
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    return [int(k) for k in np.exp(r.uniform(lo, hi, case["count"])).round()]


def prepare(case, seed):
    g = _generator(seed)
    dim, kind = case["dim"], case["kind"]
    s = {"case": case}
    if kind == "batch":
        return _prepare_batch(case, g, s)
    n = case["n"]
    if kind == "train":
        return _prepare_train(case, g, s)
    s["x"] = _seeds(g, n, dim)
    s["A"] = _anisotropy(g, n, dim, case.get("alpha", -1.0))
    s["v"] = _volumes(g, n, case.get("equal", False))
    zeros = torch.zeros(n, dtype=F64, device="cuda")
    if kind == "points":
        s["w"] = _weights(g, n, dim)
        s["y"] = _rand(g, case["points"], dim)
        mass = 0.5 + _rand(g, case["points"])
        s["mass"] = (mass / mass.sum()).contiguous()
        s["ws"] = capi.Workspace(dim, n, 64)
        s["labels"] = torch.empty(case["points"], dtype=torch.int32, device="cuda")
        s["moments"] = torch.empty((n, MOMENTS[dim]), dtype=F64, device="cuda")
    else:
        grid = synth.Grid(dim, _res(case["res"]))
        s["grid"] = grid
        if kind == "masked":
            s["w"] = _weights(g, n, dim)
            s["labels"] = torch.empty(grid.num_pixels, dtype=torch.int32, device="cuda")
            s["ws"] = capi.Workspace(dim, n, grid.num_pixels)
            s["ws"].set_pruning(True)
        else:
            weighted = kind in ("dual", "moments") or case.get("weighted", False)
            s["w"] = _weights(g, n, dim) if weighted else zeros
            s["ws"] = capi.Workspace(dim, n, grid.num_pixels)
            s["ws"].set_pruning(case["prune"])
            s["precision"] = PRECISION[case["precision"]]
    if kind == "assign":
        s["labels"] = torch.empty(s["grid"].num_pixels, dtype=torch.int32, device="cuda")
    if kind == "moments":
        s["moments"] = torch.empty((n, MOMENTS[dim]), dtype=torch.int64, device="cuda")
    if kind in ("dual", "points", "masked"):
        s["g"] = torch.empty(1, dtype=F64, device="cuda")
        s["err"] = torch.empty(1, dtype=F64, device="cuda")
        s["grad"] = torch.empty(n, dtype=F64, device="cuda")
    if kind in ("solve", "lloyd"):
        s["w_out"] = torch.empty(n, dtype=F64, device="cuda")
        s["x_out"] = torch.empty((n, dim), dtype=F64, device="cuda")
        s["opts"] = capi.solve_opts(eps=0.01, max_evals=400, precision=s["precision"])
        s["mopts"] = capi.multires_opts(factor=2, coarse_eps=0.015, coarse_max_evals=200, carry_history=True)
        s["net"] = warmstart.load(dim) if kind == "lloyd" else None
    return s


def _prepare_batch(case, g, s):
    dim = case["dim"]
    counts = _batch_sizes(case)
    x, A, v, insts = [], [], [], []
    for n in counts:
        x.append(_seeds(g, n, dim))
        A.append(_anisotropy(g, n, dim, -1.0))
        v.append(_volumes(g, n, False))
    for n, vmin in zip(counts, torch.stack([t.min() for t in v]).tolist()):
        need = synth.required_resolution(dim, vmin)
        if dim == 2:
            m = next((r for r in synth.BATCH_2D_RES if r >= need), synth.BATCH_2D_RES[-1])
        else:
            m = min(need, 128)
        insts.append(_Inst(n, synth.Grid.cube(dim, m)))
    s["x"], s["A"], s["v"] = torch.cat(x), torch.cat(A), torch.cat(v)
    s["insts"] = insts
    s["w_out"] = torch.empty(sum(counts), dtype=F64, device="cuda")
    s["net"] = warmstart.load(dim)
    s["batch"] = capi.Batch(dim, [i.grid for i in insts], counts)
    s["batch"].set_pruning(True)
    s["opts"] = capi.solve_opts(eps=0.01, max_evals=400)
    s["mopts"] = capi.multires_opts(factor=2, coarse_eps=0.015, coarse_max_evals=200)
    return s


def _prepare_train(case, g, s):
    dim, n, k = case["dim"], case["n"], case["instances"]
    x = torch.cat([_seeds(g, n, dim) for _ in range(k)])
    A = _anisotropy(g, n * k, dim, -1.0)
    v = torch.cat([_volumes(g, n, False) for _ in range(k)])
    n_features, _ = capi.warmstart_sizes(dim)
    s["features"] = torch.empty((n * k, n_features), dtype=torch.float32, device="cuda")
    s["knn"] = torch.empty((n * k, 8), dtype=torch.int32, device="cuda")
    s["net"] = capi.WarmStart(dim, warmstart.init_params(dim, 3))
    s["net"].features([n] * k, [synth.Grid.cube(dim, 64)] * k, x, A, v, s["features"], knn=s["knn"])
    s["net"].fit_norm(s["features"])
    s["targets"] = (0.3 * _randn(g, n * k) + 0.5 * (v * n - 1.0)).float().contiguous()
    s["idx"] = torch.randperm(n * k, generator=g, device="cuda").to(torch.int32)
    s["y_buf"] = torch.zeros(n * k, dtype=torch.float32, device="cuda")
    s["dy_buf"] = torch.zeros(n * k, dtype=torch.float32, device="cuda")
    s["grad"] = torch.empty(s["net"].n_params, dtype=torch.float32, device="cuda")
    s["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "assign":
        capi.apd_assign(s["grid"], s["x"], s["A"], s["w"], s["labels"], s["ws"], precision=s["precision"])
        return {"labels": s["labels"]}
    if kind == "moments":
        capi.apd_cell_moments(s["grid"], s["x"], s["A"], s["w"], s["moments"], s["ws"], precision=s["precision"])
        return {"moments": s["moments"]}
    if kind == "dual":
        capi.apd_dual_value_grad(s["grid"], s["x"], s["A"], s["w"], s["v"], s["g"], s["grad"], s["err"], s["ws"],
                                 precision=s["precision"])
        return {"g": s["g"], "grad": s["grad"], "err": s["err"]}
    if kind == "points" and not case["dual"]:
        capi.apd_points_moments(s["y"], s["mass"], s["x"], s["A"], s["w"], s["moments"], s["ws"], labels=s["labels"])
        return {"moments": s["moments"], "labels": s["labels"]}
    if kind == "points":
        capi.apd_points_dual_value_grad(s["y"], s["mass"], s["x"], s["A"], s["w"], s["v"], s["g"], s["grad"], s["err"],
                                        s["ws"])
        return {"g": s["g"], "grad": s["grad"], "err": s["err"]}
    if kind == "masked":
        capi.apd_masked_dual_value_grad(s["grid"], case["refine"], s["x"], s["A"], s["w"], s["v"], s["g"], s["grad"],
                                        s["err"], s["labels"], s["ws"])
        return {"g": s["g"], "grad": s["grad"], "err": s["err"], "labels": s["labels"]}
    if kind == "solve":
        if case["multires"]:
            _, info, _ = capi.apd_solve_weights_multires(s["grid"], s["x"], s["A"], s["w"], s["v"], s["w_out"],
                                                         s["ws"], s["opts"], s["mopts"])
        else:
            _, info = capi.apd_solve_weights(s["grid"], s["x"], s["A"], s["w"], s["v"], s["w_out"], s["ws"],
                                             s["opts"])
        return {"w": s["w_out"], "g": info.g, "err": info.max_rel_err}
    if kind == "lloyd":
        _, info, _ = capi.apd_lloyd_multires(s["grid"], s["x"], s["A"], s["w"], s["v"], case["rounds"], s["x_out"],
                                             s["w_out"], s["ws"], s["opts"], s["mopts"], s["net"])
        return {"x": s["x_out"], "w": s["w_out"], "g": info.g, "err": info.max_rel_err}
    if kind == "batch":
        start = warmstart.predict(s["net"], s["insts"], s["x"], s["A"], s["v"])
        _, infos, _ = capi.apd_batch_solve_weights_multires(s["batch"], s["x"], s["A"], start, s["v"], s["w_out"],
                                                            s["opts"], s["mopts"], judge=True)
        return {"w": s["w_out"], "g": np.array([i.g for i in infos]),
                "err": np.array([i.max_rel_err for i in infos])}
    s["net"].train_step_pairs(s["idx"], s["features"], s["targets"], s["knn"], s["y_buf"], s["dy_buf"], 2e-3, mu=0.02,
                              grad_out=s["grad"], loss_out=s["loss"])
    return {"grad": s["grad"], "loss": s["loss"]}


def work(case):
    """Least bytes and operations: inputs read and outputs written once; one cost
    of eq. (2.1) per pixel, voxel or sample point (a label is at least that),
    except the dense sweep, which is asked to score every seed; a solve is at
    least one evaluation per grid and round."""
    dim, kind = case["dim"], case["kind"]
    cost = 2.0 * FEATURES[dim]
    if kind == "batch":
        n = case["count"] * math.sqrt(case["n_lo"] * case["n_hi"])
        pixels = case["count"] * (512.0 ** 2 if dim == 2 else 96.0 ** 3)
        return {"bytes": n * (dim + dim * dim + 3) * 8, "flops": cost * pixels}
    n = case["n"]
    if kind == "train":
        n_features, n_params = capi.warmstart_sizes(dim)
        rows = n * case["instances"]
        return {"bytes": rows * (n_features * 4 + 8 * 4 + 8) + n_params * 4 * 6, "flops": 6.0 * n_params * rows}
    seeds = n * (dim + dim * dim + 1) * 8.0
    if kind == "points":
        out = n * 16.0 if case["dual"] else n * MOMENTS[dim] * 8.0 + case["points"] * 4.0
        return {"bytes": case["points"] * (dim + 1) * 8.0 + seeds + out, "flops": cost * case["points"]}
    pixels = float(np.prod(_res(case["res"])))
    if kind == "assign":
        pairs = pixels if case["prune"] else pixels * n
        return {"bytes": seeds + pixels * 4, "flops": cost * pairs}
    if kind == "moments":
        pairs = pixels if case["prune"] else pixels * n
        return {"bytes": seeds + n * MOMENTS[dim] * 8.0, "flops": cost * pairs}
    if kind == "dual":
        pairs = pixels if case["prune"] else pixels * n
        return {"bytes": seeds + n * 16.0 + 16, "flops": cost * pairs}
    if kind == "masked":
        return {"bytes": seeds + n * 16.0 + pixels * 4, "flops": cost * pixels * 2}
    solves = case["rounds"] + 1 if kind == "lloyd" else 1
    return {"bytes": seeds + n * 24.0, "flops": cost * pixels * solves}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _phi(x, A, w):
    """Coefficients of the costs in the features [y_a y_b (a <= b), y_a, 1], a column per seed."""
    dim = x.shape[1]
    S = 0.5 * (A + A.transpose(1, 2))
    Ax = torch.einsum("nab,nb->na", S, x)
    rows = [S[:, a, b] * (1.0 if a == b else 2.0) for a in range(dim) for b in range(a, dim)]
    rows += [-2.0 * Ax[:, a] for a in range(dim)]
    rows.append((x * Ax).sum(1) - w)
    return torch.stack(rows)


def _least(y, phi):
    """Smallest cost and its seed at the points y, in 64 bits (y about the box centre)."""
    dim = y.shape[1]
    f = [y[:, a] * y[:, b] for a in range(dim) for b in range(a, dim)] + [y[:, a] for a in range(dim)]
    f = torch.stack(f + [torch.ones_like(y[:, 0])], 1)
    return (f @ phi).min(1)


def _centres(grid, a, b):
    """Centres of the pixels a .. b - 1, first axis fastest."""
    j = torch.arange(a, b, device="cuda")
    cols = []
    for d in range(grid.dim):
        h = (grid.hi[d] - grid.lo[d]) / grid.res[d]
        cols.append(grid.lo[d] + ((j % grid.res[d]).to(F64) + 0.5) * h)
        j = torch.div(j, grid.res[d], rounding_mode="floor")
    return torch.stack(cols, 1)


def _dual_sums(n, chunks):
    """Sum of measures per cell, and of measure times smallest cost."""
    vol = torch.zeros(n, dtype=F64, device="cuda")
    total = torch.zeros((), dtype=F64, device="cuda")
    for cost, label, mass in chunks:
        vol.index_add_(0, label, mass)
        total = total + (mass * cost).sum()
    return vol, total


def _dual_values(s, vol, total):
    grad = s["v"] - vol
    g = (s["v"] * s["w"]).sum() + total
    return {"g": g.reshape(1), "grad": grad, "err": (grad.abs() / s["v"]).max().reshape(1)}


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("dual", "points", "masked", "train"):
        return None  # labels and moments are whole numbers; a solve's iterates have no closed value
    s = prepare(case, seed)
    if kind == "train":
        return _exact_train(s)
    n, dim = case["n"], case["dim"]
    mid = torch.full((dim,), 0.5, dtype=F64, device="cuda")
    phi = _phi(s["x"] - mid, s["A"], s["w"])
    step = max(4096, (1 << 28) // n)
    if kind == "points" and not case["dual"]:
        mom = torch.zeros((n, MOMENTS[dim]), dtype=F64, device="cuda")
        for a in range(0, case["points"], step):
            y, mass = s["y"][a:a + step], s["mass"][a:a + step]
            label = _least(y - mid, phi)[1]
            cols = [mass] + [mass * y[:, i] for i in range(dim)]
            cols += [mass * y[:, i] * y[:, k] for i in range(dim) for k in range(i, dim)]
            mom.index_add_(0, label, torch.stack(cols, 1))
        return {"moments": mom, "labels": None}
    if kind == "points":
        def chunks():
            for a in range(0, case["points"], step):
                cost, label = _least(s["y"][a:a + step] - mid, phi)
                yield cost, label, s["mass"][a:a + step]
        return _dual_values(s, *_dual_sums(n, chunks()))
    grid = s["grid"]
    if kind == "dual":
        cell = grid.measure / grid.num_pixels

        def chunks():
            for a in range(0, grid.num_pixels, step):
                cost, label = _least(_centres(grid, a, min(grid.num_pixels, a + step)) - mid, phi)
                yield cost, label, torch.full_like(cost, cell)
        return _dual_values(s, *_dual_sums(n, chunks()))
    # masked: fine pixels of interior coarse pixels keep the coarse label, the others are labelled
    r = case["refine"]
    coarse = torch.cat([_least(_centres(grid, a, min(grid.num_pixels, a + step)) - mid, phi)[1]
                        for a in range(0, grid.num_pixels, step)])
    lab = coarse.reshape(tuple(reversed(grid.res)))
    boundary = torch.zeros_like(lab, dtype=torch.bool)
    near = [(i,) for i in (-1, 0, 1)]
    for _ in range(dim - 1):
        near = [t + (i,) for t in near for i in (-1, 0, 1)]
    for off in near:
        here = tuple(slice(max(0, -o), lab.shape[d] - max(0, o)) for d, o in enumerate(off))
        there = tuple(slice(max(0, o), lab.shape[d] - max(0, -o)) for d, o in enumerate(off))
        boundary[here] |= lab[here] != lab[there]
    boundary = boundary.reshape(-1)
    fine = synth.Grid(dim, tuple(m * r for m in grid.res))
    cell = fine.measure / fine.num_pixels

    def chunks():
        for a in range(0, fine.num_pixels, step):
            b = min(fine.num_pixels, a + step)
            y = _centres(fine, a, b)
            j = torch.arange(a, b, device="cuda")
            at, stride = torch.zeros_like(j), 1
            for d in range(dim):
                at += torch.div(j % fine.res[d], r, rounding_mode="floor") * stride
                j = torch.div(j, fine.res[d], rounding_mode="floor")
                stride *= grid.res[d]
            cost, label = _least(y - mid, phi)
            label = torch.where(boundary[at], label, coarse[at])
            dy = y - s["x"][label]
            cost = torch.einsum("pa,pab,pb->p", dy, s["A"][label], dy) - s["w"][label]
            yield cost, label, torch.full_like(cost, cell)
    out = _dual_values(s, *_dual_sums(n, chunks()))
    out["labels"] = None
    return out


def _exact_train(s):
    params, norm = s["net"].get()
    F = s["net"].n_features
    p = torch.from_numpy(params).cuda().to(F64).requires_grad_(True)
    mean, istd = torch.from_numpy(norm).cuda().to(F64).split(F)
    h, at = (s["features"].to(F64) - mean) * istd, 0
    for fan_in, fan_out in ((F, 64), (64, 64), (64, 64), (64, 1)):
        W = p[at:at + fan_in * fan_out].reshape(fan_out, fan_in)
        b = p[at + fan_in * fan_out:at + fan_in * fan_out + fan_out]
        at += fan_in * fan_out + fan_out
        h = h @ W.T + b
        h = torch.relu(h) if fan_out > 1 else h
    d = h[:, 0] - s["targets"].to(F64)
    knn = s["knn"].long()
    pair = torch.where(knn >= 0, d[:, None] - d[knn.clamp(min=0)], torch.zeros((), dtype=F64, device="cuda"))
    loss = (pair ** 2).sum() / (8 * d.numel()) + 0.02 * (d ** 2).mean()
    grad, = torch.autograd.grad(loss, p)
    return {"grad": grad, "loss": loss.detach().reshape(1)}
