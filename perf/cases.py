"""Workloads of the pseudo-projection solver, each one pass of a user's program through the public
binding: a call with its inputs at hand, the iterations it asks for, and the iterate it reads back.

Inputs are the dense random system of ``workloads.dense_system`` (a_ij ~ N(0, 1), an interior point
z ~ U(-1, 1)^n, b0 = A z + U(0.1, 1), a unit translation direction, x0 ~ N(0, 25 I)), its sparse form,
and the model system (a box with a cut corner), drawn on the GPU.  Matrices stored in bf16 and FP8 are
drawn on that storage's grid, so that the stored system is the drawn one.  The right-hand side is moved
away from the few rows that x0 lies almost on: whether such a row is violated would be decided by
rounding, and a flipped row changes the step by 1 / h.  A pass starts from x0 (given with the call, as a
program with a new starting point gives it), so every pass does the same work.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2003_09956_gb300 import nsli

RHO = 1e-4        # translation per iteration, the benchmark's
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "fp8": 1}
CHUNK = 1 << 27   # entries of A drawn or widened to binary64 at a time


def listed():
    return [
        # a control loop: every tick brings a new b and the measured point; one iteration, x read back
        {"name": "tick_f32_2000x500", "kind": "tick", "m": 2000, "n": 500, "storage": "f32"},
        # the paper's model system held dense in binary64: latency and launches, 256 iterations a call
        {"name": "model_f64_256", "kind": "model", "n": 256, "iters": 256},
        # a small dense system, one short run from a new starting point
        {"name": "dense_f32_8192x2048", "kind": "dense", "m": 8192, "n": 2048, "storage": "f32",
         "rule": "relaxed", "iters": 24},
        # odd sizes (ragged rows), bf16 storage, the ModAP rule
        {"name": "dense_bf16_20011x4099_modap", "kind": "dense", "m": 20011, "n": 4099, "storage": "bf16",
         "rule": "modap", "iters": 32},
        # the benchmark system, binary32
        {"name": "dense_f32_131072x16384", "kind": "dense", "m": 131072, "n": 16384, "storage": "f32",
         "rule": "relaxed", "iters": 8},
        # the benchmark system in FP8
        {"name": "dense_fp8_131072x16384", "kind": "dense", "m": 131072, "n": 16384, "storage": "fp8",
         "rule": "relaxed", "iters": 8},
        # rows of the paper's largest dimension (n = 54000), bf16: the cluster kernel
        {"name": "long_bf16_27000x54000", "kind": "dense", "m": 27000, "n": 54000, "storage": "bf16",
         "rule": "relaxed", "iters": 4},
        # a large sparse system, 32 entries per row at random columns
        {"name": "sparse_f32_1048576x262144x32", "kind": "sparse", "m": 1048576, "n": 262144, "k": 32,
         "storage": "f32", "rule": "relaxed", "iters": 8},
        # the model system in compressed rows, solved to the paper's step rule (one CTA)
        {"name": "model_solve_256", "kind": "model_solve", "n": 256},
        # 64 problems sharing one matrix, on the tensor cores
        {"name": "batch_64x65536x8192", "kind": "batch", "nprob": 64, "m": 65536, "n": 8192, "iters": 8},
        # serving: twelve resident problems of mixed sizes, one persistent launch
        {"name": "serve_bf16_mix12", "kind": "serve", "mix": 7, "count": 12, "rounds": 8},
        # a matrix that changes with time: all rows rewritten, then one iteration
        {"name": "rewrite_bf16_32768x16384", "kind": "rewrite", "m": 32768, "n": 16384, "storage": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _iters(n, most):
    """Iterations of a run from x0: fewer for short rows, whose iterate moves by 1 / n each time."""
    return max(1, min(most, int((n / 400.0) ** 2)))


def draw(rng):
    kind = rng.choice(["tick", "model", "dense", "dense", "dense", "long", "sparse", "model_solve", "batch",
                       "serve", "rewrite"])
    storage = rng.choice(["f32", "bf16", "fp8"])
    rule = rng.choice(["relaxed", "relaxed", "modap"])
    if kind == "tick":
        n = _log(rng, 100, 3000)
        return {"kind": kind, "m": int(n * rng.uniform(2, 8)) + 1, "n": n, "storage": storage}
    if kind == "model":
        return {"kind": kind, "n": _log(rng, 40, 500), "iters": rng.randint(50, 400)}
    if kind == "model_solve":
        return {"kind": kind, "n": _log(rng, 24, 256)}
    if kind == "dense":
        n = _log(rng, 300, 16384)
        m = min(131072, int(n * rng.uniform(2, 8)) + 1)
        return {"kind": kind, "m": m, "n": n, "storage": storage, "rule": rule, "iters": _iters(n, rng.randint(4, 32) if n < 9000 else 8)}
    if kind == "long":
        n = _log(rng, 16400, 60000)
        return {"kind": "dense", "m": min(27000, int(n * rng.uniform(0.25, 1.5))), "n": n, "storage": storage,
                "rule": rule, "iters": rng.randint(1, 4)}
    if kind == "sparse":
        k = rng.randint(3, 32)
        n = _log(rng, 20000, 262144)
        m = min(1048576, int(n * rng.uniform(1.5, 5)))
        return {"kind": kind, "m": m, "n": n, "k": k, "storage": rng.choice(["f32", "f32", "f64"]), "rule": rule,
                "iters": rng.randint(2, 8)}
    if kind == "batch":
        n = _log(rng, 2000, 8192)
        return {"kind": kind, "nprob": rng.randint(2, 64), "m": int(n * rng.uniform(1, 8)), "n": n,
                "iters": 8 if n >= 4096 else 2}
    if kind == "serve":
        return {"kind": kind, "mix": rng.randint(100, 10 ** 6), "count": rng.randint(2, 12), "rounds": 8}
    n = _log(rng, 600, 16384)
    return {"kind": "rewrite", "m": min(32768, int(n * rng.uniform(2, 8))), "n": n, "storage": storage}


# ---------------------------------------------------------------- inputs ----

def _rows_at_a_time(n):
    return max(1, CHUNK // n)


def _on_grid(a, storage):
    """Rows rounded in place onto the storage's grid (FP8: a power-of-two scale per row)."""
    if storage == "bf16":
        a.copy_(a.to(torch.bfloat16))
    elif storage == "fp8":
        f, e2 = torch.frexp(a.abs().amax(1, keepdim=True))
        s = torch.ldexp(torch.ones_like(f), torch.where(f <= 0.875, e2 - 9, e2 - 8))
        a.copy_((a / s).to(torch.float8_e4m3fn).float() * s)
    return a


def _wide(a, *vs):
    """a @ v in binary64 for every v."""
    step = _rows_at_a_time(a.shape[1])
    out = [[] for _ in vs]
    for r in range(0, a.shape[0], step):
        w = a[r:r + step].double()
        for o, v in zip(out, vs):
            o.append(w @ v)
    return [torch.cat(o) for o in out]


def _matrix(g, m, n, storage):
    a = torch.empty((m, n), device="cuda")
    step = _rows_at_a_time(n)
    for r in range(0, m, step):
        _on_grid(a[r:r + step].normal_(generator=g), storage)
    return a


def _off_faces(b0, r, margin):
    """b0 raised where |r| (rows of every problem, at its x0) is below the margin: r moves with -b0."""
    for _ in range(12):
        near = (r.abs() < margin).any(1)
        if not bool(near.any()):
            break
        push = near.double() * (2.5 * margin)
        b0 += push
        r -= push[:, None]
    return b0


def _moved(iters, n):
    """How far (in residuals' standard deviations) a row can move over the run, with room to spare."""
    return 0.01 + 4.0 * iters / n


def _dense(seed, m, n, storage, iters, nprob=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = _matrix(g, m, n, storage)
    z = torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * 2 - 1
    slack = torch.rand(m, device="cuda", dtype=torch.float64, generator=g) * 0.9 + 0.1
    v = torch.randn(n, device="cuda", dtype=torch.float64, generator=g)
    v /= v.norm()
    x0 = (torch.randn((nprob, n), device="cuda", dtype=torch.float32, generator=g) * 5).double()
    az, av, *ax = _wide(a, z, v, *x0)
    b0 = az + slack
    r = torch.stack(ax, 1) - b0[:, None]
    b0 = _off_faces(b0, r, (_moved(iters, n) - (0.009 if nprob > 1 else 0.0)) * 5 * math.sqrt(n))
    return {"A": a, "b0": b0, "Av": av, "x0": x0 if nprob > 1 else x0[0]}


def _model(seed, n):
    """0 <= x_j <= 200, sum x_j <= 200 (n - 1) + 100, x0 ~ U[300, 400]^n, in compressed rows."""
    idx = np.arange(n, dtype=np.int64)
    b0 = np.zeros(2 * n + 1)
    b0[n:2 * n] = 200.0
    b0[2 * n] = 200.0 * (n - 1) + 100.0
    return {"rp": np.concatenate([np.arange(0, 2 * n + 1, dtype=np.int64), [3 * n]]),
            "ci": np.concatenate([idx, idx, idx]).astype(np.int32),
            "val": np.concatenate([-np.ones(n), np.ones(n), np.ones(n)]), "b0": b0,
            "x0": np.random.Generator(np.random.PCG64(seed)).uniform(300.0, 400.0, n), "m": 2 * n + 1, "n": n}


def _model_dense(p):
    n = p["n"]
    a = np.zeros((2 * n + 1, n))
    a[np.arange(n), np.arange(n)] = -1.0
    a[n + np.arange(n), np.arange(n)] = 1.0
    a[2 * n] = 1.0
    return a


def _sparse(seed, m, n, k, iters):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ci = torch.randint(0, n - k + 1, (m, k), device="cuda", generator=g).sort(1)[0] + torch.arange(k, device="cuda")
    val = torch.randn((m, k), device="cuda", generator=g).double()
    z = torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * 2 - 1
    slack = torch.rand(m, device="cuda", dtype=torch.float64, generator=g) * 0.9 + 0.1
    v = torch.randn(n, device="cuda", dtype=torch.float64, generator=g)
    v /= v.norm()
    x0 = (torch.randn(n, device="cuda", dtype=torch.float32, generator=g) * 5).double()
    b0 = (val * z[ci]).sum(1) + slack
    r = (val * x0[ci]).sum(1) - b0
    b0 = _off_faces(b0, r[:, None], _moved(iters, n) * 5 * math.sqrt(k))
    return {"ci": ci, "val": val, "b0": b0, "Av": (val * v[ci]).sum(1), "x0": x0}


def _mix(case):
    """Shapes of a serving mix: n over the request classes, m = 2, 4 or 8 n (4 n for the longest rows)."""
    g = np.random.Generator(np.random.PCG64(case["mix"]))
    ns = [1024, 1448, 2048, 2896, 4096, 5793, 8192]
    got = []
    for _ in range(case["count"]):
        n = int(ns[g.integers(len(ns))])
        got.append((n * int(g.choice([2, 4, 8] if n < 8192 else [2, 4])), n))
    return got


def _lam(case):
    """Step length: 1 for the relaxed rule; for ModAP about the relaxed rule's step at x0."""
    return 5.0 / math.sqrt(case["n"]) if case.get("rule") == "modap" else 1.0


# ------------------------------------------------------------------ cases ----

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("tick", "dense", "rewrite"):
        p = _dense(seed, case["m"], case["n"], case["storage"], case.get("iters", 1))
        a = p.pop("A")
        s = {"case": case, "solver": nsli.Solver(a, p["b0"], p["x0"], Av=p["Av"], storage=case["storage"]),
             "x0": p["x0"], "b0": p["b0"], "out": torch.empty_like(p["x0"])}
        if kind == "rewrite":
            q = _dense(seed + 7919, case["m"], case["n"], case["storage"], 1)
            s.update(A=q["A"], b0=q["b0"], x0=q["x0"])
        if kind == "tick":
            s["b0"] = p["b0"] + 0.125   # the tick's new right-hand side
        return s
    if kind == "model":
        p = _model(seed, case["n"])
        return {"case": case, "solver": nsli.Solver(_model_dense(p), p["b0"], p["x0"], storage="f64"),
                "x0": torch.from_numpy(p["x0"]).cuda(), "out": torch.empty(case["n"], dtype=torch.float64, device="cuda")}
    if kind == "model_solve":
        p = _model(seed, case["n"])
        return {"case": case, "solver": nsli.SparseSolver(p["m"], p["n"], p["rp"], p["ci"], p["val"], p["b0"], p["x0"], storage="f64"),
                "x0": torch.from_numpy(p["x0"]).cuda(), "out": torch.empty(case["n"], dtype=torch.float64, device="cuda")}
    if kind == "sparse":
        m, n, k = case["m"], case["n"], case["k"]
        p = _sparse(seed, m, n, k, case["iters"])
        rp = np.arange(0, m * k + 1, k, dtype=np.int64)
        solver = nsli.SparseSolver(m, n, rp, p["ci"].reshape(-1).to(torch.int32).cpu().numpy(),
                                   p["val"].reshape(-1).cpu().numpy(), p["b0"], p["x0"], Av=p["Av"],
                                   storage=case["storage"])
        return {"case": case, "solver": solver, "x0": p["x0"], "out": torch.empty_like(p["x0"])}
    if kind == "batch":
        p = _dense(seed, case["m"], case["n"], "bf16", case["iters"], nprob=case["nprob"])
        return {"case": case, "solver": nsli.BatchSolver(p["A"], p["b0"], p["x0"], Av=p["Av"])}
    pool = nsli.Pool(storage="bf16")
    slots = []
    for q, (m, n) in enumerate(_mix(case)):
        p = _dense(seed + 104729 * q, m, n, "bf16", case["rounds"])
        slots.append((pool.add(p["A"], p["b0"], p["x0"], Av=p["Av"], lam=1.0, stop="none", max_iter=1 << 40, rho=RHO), n))
    return {"case": case, "pool": pool, "slots": slots}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        pool = state["pool"]
        pool.launch(max_rounds=case["rounds"], max_seconds=5.0)
        pool.wait()
        return [pool.get_x(slot, n) for slot, n in state["slots"]]
    s = state["solver"]
    if kind == "batch":
        s.iterate(case["iters"], rho=RHO)
        return s.get_x()
    if kind == "model_solve":
        s.set_x(state["x0"])
        r = s.solve(lam=1.0, stop="step", eps=1e-8, max_iter=100000)
        return {"x": s.get_x(state["out"]), "iters": r["iters"]}
    if kind == "rewrite":
        s.update_rows(0, state["A"], b0=state["b0"])
        s.set_x(state["x0"])
        s.update_b(tick=0)
        s.iterate(1, rho=RHO)
        return s.get_x(state["out"])
    s.set_x(state["x0"])
    if kind == "tick":
        s.update_b(state["b0"], tick=3)
        s.iterate(1, rho=RHO)
    elif kind == "model":
        s.iterate(case["iters"])
    else:
        s.update_b(tick=0)
        s.iterate(case["iters"], lam=_lam(case), rule=case["rule"], rho=RHO)
    return s.get_x(state["out"])


def work(case):
    """Per iteration: A read once, its records (b0, Av, 1 / ||a||^2) and x; 2 operations for a row's dot
    and 2 for its slice per entry (half of the rows are violated far from the polytope)."""
    kind = case["kind"]

    def dense(m, n, eb, iters):
        return {"bytes": iters * (m * n * eb + 12.0 * m + 16.0 * n), "flops": iters * 3.0 * m * n}

    if kind == "dense":
        return dense(case["m"], case["n"], BYTES[case["storage"]], case["iters"])
    if kind == "tick":
        w = dense(case["m"], case["n"], BYTES[case["storage"]], 1)
        return {"bytes": w["bytes"] + 8.0 * case["m"], "flops": w["flops"]}
    if kind == "rewrite":
        w = dense(case["m"], case["n"], BYTES[case["storage"]], 1)
        stored = case["m"] * case["n"] * float(4 + BYTES[case["storage"]])   # the source read, the rows written
        return {"bytes": w["bytes"] + stored, "flops": w["flops"] + 2.0 * case["m"] * case["n"]}
    if kind == "model":
        return dense(2 * case["n"] + 1, case["n"], 8, case["iters"])
    if kind == "model_solve":
        # about 12.3 n iterations over 3 n entries (value and column)
        return {"bytes": 12.3 * case["n"] * 3 * case["n"] * 12.0, "flops": 12.3 * case["n"] * 9.0 * case["n"]}
    if kind == "sparse":
        nnz, eb = case["m"] * case["k"], BYTES[case["storage"]]
        return {"bytes": case["iters"] * (nnz * (4.0 + eb) + 20.0 * case["m"] + 20.0 * case["n"]),
                "flops": case["iters"] * 3.0 * nnz}
    if kind == "batch":
        m, n, p = case["m"], case["n"], case["nprob"]
        return {"bytes": case["iters"] * (2.0 * m * n + 12.0 * m + 16.0 * n * p), "flops": case["iters"] * 4.0 * m * n * p}
    parts = [dense(m, n, 2, case["rounds"]) for m, n in _mix(case)]
    return {"bytes": sum(w["bytes"] for w in parts), "flops": sum(w["flops"] for w in parts)}


# ----------------------------------------------------------- in 64 bits ----

def _exact_dense(a, b0, av, x, iters, lam=1.0, rule="relaxed", tick=0):
    for k in range(iters):
        b = b0 if av is None else b0 + (tick + k) * RHO * av
        y, h = torch.zeros_like(x), 0
        step = _rows_at_a_time(a.shape[1])
        for q in range(0, a.shape[0], step):
            w = a[q:q + step].double()
            r = (w @ x - b[q:q + step]).clamp_min(0)
            h += int((r > 0).sum())
            y += (r / (w * w).sum(1)) @ w
        if h:
            x = x - (lam / float(y.norm()) if rule == "modap" else lam / h) * y
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dense", "tick", "rewrite"):
        p = _dense(seed + (7919 if kind == "rewrite" else 0), case["m"], case["n"], case["storage"], case.get("iters", 1))
        b0 = p["b0"] + 0.125 if kind == "tick" else p["b0"]
        return _exact_dense(p["A"], b0, None if kind == "rewrite" else p["Av"], p["x0"], case.get("iters", 1), _lam(case), case.get("rule", "relaxed"),
                            tick=3 if kind == "tick" else 0)
    if kind == "model":
        p = _model(seed, case["n"])
        a = torch.from_numpy(_model_dense(p))
        return _exact_dense(a, torch.from_numpy(p["b0"]), None, torch.from_numpy(p["x0"]), case["iters"])
    if kind == "model_solve":
        p = _model(seed, case["n"])
        a, b, x = _model_dense(p), p["b0"], p["x0"].copy()
        n2 = (a * a).sum(1)
        for it in range(1, 100001):
            r = np.maximum(a @ x - b, 0)
            h = int((r > 0).sum())
            if h == 0:
                return {"x": x, "iters": it - 1}
            d = ((r / n2) @ a) / h
            x -= d
            if np.linalg.norm(d) < 1e-8:
                break
        return {"x": x, "iters": it}
    if kind == "sparse":
        p = _sparse(seed, case["m"], case["n"], case["k"], case["iters"])
        ci, val, x, n2 = p["ci"], p["val"], p["x0"], (p["val"] ** 2).sum(1)
        for k in range(case["iters"]):
            r = ((val * x[ci]).sum(1) - (p["b0"] + k * RHO * p["Av"])).clamp_min(0)
            y = torch.zeros_like(x).index_add_(0, ci.reshape(-1), ((r / n2)[:, None] * val).reshape(-1))
            x = x - (_lam(case) / float(y.norm()) if case["rule"] == "modap" else _lam(case) / int((r > 0).sum())) * y
        return x
    if kind == "batch":
        p = _dense(seed, case["m"], case["n"], "bf16", case["iters"], nprob=case["nprob"])
        a, x = p["A"].double(), p["x0"]
        n2 = (a * a).sum(1)
        for k in range(case["iters"]):
            r = (x @ a.T - (p["b0"] + k * RHO * p["Av"])).clamp_min(0)
            x = x - ((r / n2) @ a) / (r > 0).sum(1, keepdim=True)
        return x
    return [_exact_dense(p["A"], p["b0"], p["Av"], p["x0"], case["rounds"])
            for p in (_dense(seed + 104729 * q, m, n, "bf16", case["rounds"]) for q, (m, n) in enumerate(_mix(case)))]
