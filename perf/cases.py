"""Workloads that stand for what a program does with this library: chains plus combination on dense and sparse rows
(device buffers), rounds of periodic averaging, a solve from host buffers, and the evaluation of a model.

A case names sizes and hyper-parameters only; `prepare` makes the inputs on the GPU from a seed, `run` is one pass through
the public entry points. Step counts follow linear node speeds with ratio `ratio` between the fastest and the slowest node
(the shape of the benchmark configurations and of the paper's unbalanced clusters), dealt to the nodes in a fixed mixed order.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1708_04801_b200 as P

LOSS = {"hinge": P.LOSS_HINGE, "logistic": P.LOSS_LOGISTIC, "squared": P.LOSS_SQUARED}
SCHEDULE = {"const": P.LR_CONST, "inv_sqrt": P.LR_INV_SQRT}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _dense(name, k, d, rows, steps, ratio, dtype, loss, schedule, eta, lam, path="dense", **more):
    return dict({"name": name} if name else {}, **{"path": path, "k": k, "d": d, "rows": rows, "steps": steps, "ratio": ratio, "dtype": dtype,
                 "loss": loss, "schedule": schedule, "eta": eta, "lam": lam}, **more)


def listed():
    return [
        # the smallest call: four short chains of narrow rows; a program that solves many small problems in turn, where the
        # latency of the call and of its launches counts
        _dense("tiny_f32_hinge", 4, 64, 4096, 1000, 4.0, "f32", "hinge", "const", 0.01, 1e-3),
        # few nodes with ordinary dense rows: a small cluster (the benchmark's logistic configuration)
        _dense("few_f32_logistic", 16, 1024, 8192, 20000, 4.0, "f32", "logistic", "const", 0.05, 1e-4),
        # the largest: a hundred nodes with wide half-precision rows (the benchmark's headline configuration with fewer
        # rows per node)
        _dense("wide_bf16_squared", 128, 4096, 8192, 50000, 10.0, "bf16", "squared", "const", 0.01, 1e-4),
        # many nodes with narrow rows: the heterogeneity study
        _dense("many_f32_logistic", 1024, 256, 2048, 26214, 4.0, "f32", "logistic", "const", 0.02, 1e-3),
        # wide single-precision rows, decaying step size: raw feature vectors of a few nodes
        _dense("wide_f32_logistic", 24, 4096, 2048, 5000, 4.0, "f32", "logistic", "inv_sqrt", 0.5, 1e-4),
        # rows as they come from a file: an odd number of columns, no row but the first aligned, unequal shards
        _dense("odd_f32_squared", 12, 999, 4096, 5000, 5.0, "f32", "squared", "const", 0.01, 1e-4),
        # a medium cluster with half-precision rows of an ordinary width, decaying step size
        _dense("mid_bf16_hinge", 64, 1000, 4096, 12000, 4.0, "bf16", "hinge", "inv_sqrt", 0.3, 1e-3),
        # the paper's kind of data at the benchmark's size: some 40 Zipf-distributed features per row, a million columns
        {"name": "csr_zipf_hinge", "path": "csr", "k": 64, "d": 1 << 20, "rows": 8192, "nnz": 40, "zipf": True, "steps": 65536,
         "ratio": 10.0, "loss": "hinge", "schedule": "inv_sqrt", "eta": 0.1, "lam": 1e-5, "segments": 1, "test_rows": 0},
        # the paper's analog experiment: ten nodes, 5 to 10 features per row, the chains cut into segments, after each the
        # combined model and its objective on a test set
        {"name": "csr_analog_logistic", "path": "csr", "k": 10, "d": 100000, "rows": 46000, "nnz": 7, "zipf": False, "steps": 20000,
         "ratio": 5.0, "loss": "logistic", "schedule": "const", "eta": 0.05, "lam": 1e-4, "segments": 2, "test_rows": 40000},
        # averaging every span of steps: combination, broadcast and continued chains, many short launches in a row
        _dense("rounds_f32_logistic", 32, 512, 2048, 4000, 4.0, "f32", "logistic", "const", 0.05, 1e-4, path="rounds", rounds=16),
        # one solve whose rows start in (page-locked) host memory
        _dense("host_f32_logistic", 16, 1024, 4096, 8000, 4.0, "f32", "logistic", "const", 0.05, 1e-4, path="host"),
        # objective and error rate of a model over a test set
        _dense("evaluate_f32_logistic", 1, 1024, 262144, 0, 1.0, "f32", "logistic", "const", 0.05, 1e-4, path="evaluate"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["dense"] * 6 + ["csr"] * 2 + ["rounds", "host", "evaluate"])
    loss = rng.choice(["hinge", "logistic", "squared"])
    schedule = rng.choice(["const", "inv_sqrt"])
    ratio = round(rng.uniform(1.0, 16.0), 2)
    eta = {"hinge": 0.02, "logistic": 0.05, "squared": 0.01}[loss] * (10.0 if schedule == "inv_sqrt" and loss != "squared" else 1.0)
    lam = rng.choice([1e-3, 1e-4, 1e-5])
    if path == "csr":
        zipf = rng.random() < 0.6
        nnz = rng.randint(5, 60)
        return {"path": "csr", "k": _log_uniform(rng, 2, 148), "d": _log_uniform(rng, 10000, 1 << 20), "rows": _log_uniform(rng, 500, 8192),
                "nnz": nnz, "zipf": zipf, "steps": _log_uniform(rng, 500, 40000), "ratio": ratio, "loss": loss, "schedule": schedule,
                "eta": eta, "lam": lam, "segments": rng.choice([1, 1, 2, 3]), "test_rows": rng.choice([0, _log_uniform(rng, 1000, 40000)])}
    dtype = rng.choice(["f32", "f32", "bf16"])
    # row widths: odd ones, and ones that are a multiple of 4 or of 8 and no power of two
    d = _log_uniform(rng, 8, 8192)
    step = rng.choice([1, 4, 8, 8, 8])
    d = max(8, d // step * step)
    if path == "evaluate":
        rows = _log_uniform(rng, 1000, max(2000, min(500000, int(1.5e9 / (4 * d)))))
        return _dense("", 1, d, rows, 0, 1.0, dtype, loss, schedule, eta, lam, path=path)
    if path == "rounds":
        d = min(d, 2048)
        return _dense("", _log_uniform(rng, 2, 128), d, 1024, _log_uniform(rng, 200, 4000), ratio, dtype, loss, schedule, eta, lam,
                      path=path, rounds=rng.randint(2, 16))
    k = _log_uniform(rng, 1, 1024)
    rows = _log_uniform(rng, 64, 8192)
    most = 2.0e8 if path == "host" else 4.0e9  # bytes of all rows
    rows = max(16, min(rows, int(most / (k * d * 4.0))))
    # steps of the longest chain: bounded so that no drawn case is longer than the largest listed one
    cap = min(50000.0, 1.2e4 / (0.25 + d / 2048.0) / max(1.0, k / 148.0), 2.0e10 / (k * d * 4.0))
    steps = _log_uniform(rng, min(200, int(cap)), max(201, int(cap)))
    return _dense("", k, d, rows, steps, ratio, dtype, loss, schedule, eta, lam, path=path)


def _steps(case):
    """Steps of every node: linear speeds from 1 down to 1 / ratio, in a mixed order."""
    k = case["k"]
    speed = 1.0 - (1.0 - 1.0 / case["ratio"]) * (np.arange(k) / max(k - 1, 1))
    return np.maximum(1, np.floor(case["steps"] * speed[np.random.default_rng(k).permutation(k)])).astype(np.int64)


def _shards(case, n_steps):
    """Row offsets: a slower node also holds fewer rows (the paper's unbalanced data), at least half of a fast one's."""
    share = 0.5 + 0.5 * n_steps / n_steps.max()
    rows = np.maximum(1, np.floor(case["rows"] * share)).astype(np.int64)
    return np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)


def _rows(case, seed, n):
    """n dense rows and their labels."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 17)
    d, dt = case["d"], DTYPE[case["dtype"]]
    w_star = torch.randn(d, generator=g, device="cuda")
    X = torch.empty((n, d), dtype=dt, device="cuda")
    z = torch.empty(n, device="cuda")
    chunk = max(1, (1 << 26) // d)
    for r0 in range(0, n, chunk):
        blk = torch.randn((min(chunk, n - r0), d), generator=g, device="cuda").mul_(1.0 / math.sqrt(d))
        X[r0:r0 + chunk] = blk
        z[r0:r0 + chunk] = X[r0:r0 + chunk].float() @ w_star
    return X, _labels(case, z, g)


def _labels(case, z, g):
    u = torch.rand(z.shape[0], generator=g, device="cuda")
    if case["loss"] == "squared":
        return (z + 0.1 * torch.randn(z.shape[0], generator=g, device="cuda")).contiguous()
    if case["loss"] == "logistic":
        return torch.where(u < torch.sigmoid(z), 1.0, -1.0).contiguous()
    y = torch.where(z >= 0, 1.0, -1.0)
    return torch.where(u < 0.05, -y, y).contiguous()


def _sparse_rows(case, seed, n):
    """n unit-length CSR rows with distinct ascending columns, and their labels."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 29)
    d, mean = case["d"], case["nnz"]
    if case["zipf"]:
        cdf = torch.cumsum(torch.arange(1, d + 1, dtype=torch.float64, device="cuda").pow(-1.1), 0)
        cdf /= cdf[-1].clone()
        most = min(d, 2 * mean + 30)
        # 1.28 draws for every distinct column at 40 columns a row
        nnz = torch.poisson(torch.full((n,), 1.28 * mean, device="cuda"), generator=g).long().clamp_(1, most)
    else:
        most = mean + 3
        nnz = torch.randint(max(1, mean - 2), most + 1, (n,), generator=g, device="cuda")
    scatter = torch.randperm(d, generator=g, device="cuda")
    w_star = torch.randn(d, generator=g, device="cuda") * (torch.rand(d, generator=g, device="cuda") < (0.05 if case["zipf"] else 1.0))
    lane = torch.arange(most, device="cuda")
    cols_all, vals_all, count_all, z_all = [], [], [], []
    for r0 in range(0, n, 1 << 18):
        c = nnz[r0:r0 + (1 << 18)]
        u = torch.rand((c.shape[0], most), generator=g, device="cuda", dtype=torch.float64)
        rank = torch.searchsorted(cdf, u).clamp_(max=d - 1) if case["zipf"] else (u * d).long().clamp_(max=d - 1)
        cols = torch.where(lane[None, :] < c[:, None], scatter[rank], d)
        cols = torch.sort(cols, dim=1).values
        keep = cols < d
        keep[:, 1:] &= cols[:, 1:] != cols[:, :-1]  # a column drawn twice in a row counts once
        cnt = keep.sum(1)
        if case["zipf"]:  # binary features scaled to unit length
            val = keep.float() * cnt.float().rsqrt()[:, None]
        else:
            val = keep.float() * (0.05 + torch.rand(cols.shape, generator=g, device="cuda"))
            val = val / val.pow(2).sum(1, keepdim=True).sqrt()
        z_all.append((w_star[cols.clamp(max=d - 1)] * val).sum(1))
        cols_all.append(cols[keep].to(torch.int32))
        vals_all.append(val[keep])
        count_all.append(cnt)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.cat(count_all), 0)
    return row_ptr, torch.cat(cols_all), torch.cat(vals_all), _labels(case, torch.cat(z_all), g)


def prepare(case, seed):
    torch.cuda.set_device(0)
    s = {"case": case, "seed": int(seed) & 0xFFFF, "loss": LOSS[case["loss"]], "schedule": SCHEDULE[case["schedule"]]}
    d = case["d"]
    if case["path"] == "evaluate":
        s["X"], s["y"] = _rows(case, seed, case["rows"])
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 5)
        s["w"] = torch.randn(d, generator=g, device="cuda")
        s["ctx"] = P.Context(1, d)
        return s
    k = case["k"]
    n = s["n"] = _steps(case)
    off = s["off"] = _shards(case, n)
    N = int(off[-1])
    s["ctx"] = P.Context(k, d)
    s["v"] = torch.empty(d, device="cuda")
    s["models"] = torch.empty((k, d), device="cuda")
    if case["path"] == "csr":
        s["rows"] = _sparse_rows(case, seed, N)
        s["parts"] = _parts(n, case["segments"])
        if case["test_rows"]:
            s["test"] = _sparse_rows(case, int(seed) + 500, case["test_rows"])
        return s
    s["X"], s["y"] = _rows(case, seed, N)
    if case["path"] == "rounds":
        s["parts"] = _parts(n, case["rounds"])
    if case["path"] == "host":
        s["X"], s["y"] = s["X"].cpu().pin_memory(), s["y"].cpu().pin_memory()
        s["v"] = torch.empty(d).pin_memory()
        del s["models"]
    return s


def _parts(n, count):
    """The steps of every node cut into `count` segments."""
    cuts = [n * i // count for i in range(count + 1)]
    return [cuts[i + 1] - cuts[i] for i in range(count)]


def run(s):
    case, ctx = s["case"], s["ctx"]
    path, hyper = case["path"], (case["eta"], s["schedule"], case["lam"], s["loss"], s["seed"])
    if path == "evaluate":
        return ctx.objective(s["X"], s["y"], s["w"], case["lam"], s["loss"])
    if path == "host":
        return ctx.solve_host(s["X"], s["y"], s["off"], s["n"], *hyper, out=s["v"])
    if path == "csr":
        row_ptr, col, val, y = s["rows"]
        out = {}
        for i, part in enumerate(s["parts"]):
            if i == 0:
                ctx.run_csr(row_ptr, col, val, y, s["off"], part, *hyper)
            else:
                ctx.continue_csr(row_ptr, col, val, y, s["off"], part)
            v = ctx.combine(out=s["v"])
            if case["test_rows"]:
                out["objective%d" % i] = ctx.objective_csr(*s["test"], v, case["lam"], s["loss"])
        return dict(out, v=v, models=ctx.get_models(out=s["models"]))
    if path == "rounds":
        for i, part in enumerate(s["parts"]):
            if i == 0:
                ctx.run(s["X"], s["y"], s["off"], part, *hyper)
            else:
                ctx.set_models(v)
                ctx.continue_(s["X"], s["y"], s["off"], part)
            v = ctx.combine(out=s["v"])
        return {"v": v, "models": ctx.get_models(out=s["models"])}
    ctx.run(s["X"], s["y"], s["off"], s["n"], *hyper)
    return {"v": ctx.combine(out=s["v"]), "models": ctx.get_models(out=s["models"])}


def work(case):
    """Bytes: every sample visit brings its row, its label and its index (for the host path: the copy of all rows as
    well); the models and the combined model are written once. Operations: margin and update of a sample."""
    d = case["d"]
    es = 4.0 if case.get("dtype", "f32") == "f32" else 2.0
    if case["path"] == "evaluate":
        return {"bytes": case["rows"] * (d * es + 4.0) + 4.0 * d, "flops": 2.0 * case["rows"] * d}
    n = _steps(case)
    total, out = float(n.sum()), 4.0 * d * (case["k"] + 1)
    if case["path"] == "csr":
        mean = float(case["nnz"])
        test = case["segments"] * case["test_rows"] * (mean * 8.0 + 12.0)
        return {"bytes": total * (mean * 16.0 + 16.0) + test + out, "flops": 4.0 * total * mean}
    rows = float(_shards(case, n)[-1]) if case["path"] == "host" else 0.0
    return {"bytes": total * (d * es + 8.0) + out + rows * (d * es + 4.0), "flops": 4.0 * total * d}


def tolerance(case):
    """Relative error of models and combined model: about four times what chains of the same precision with their sums in
    another order, or in 64 bits, differ by. Rounding collects along a chain (5e-5 after 50000 steps, 8e-6 after 5000)."""
    if case["path"] == "evaluate":
        return {"rel": 1e-6}
    if case["loss"] == "hinge":  # a margin within rounding of 1 may flip one subgradient, and the flip stays in the model
        return {"rel": 1e-3}
    return {"rel": 1e-5 if case["path"] == "csr" else max(3e-5, 4e-9 * case["steps"])}
