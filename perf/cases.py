"""Performance cases: the work that a user of this library has it do.

Every case goes through the public package: handles (``cg_create``,
``cg_solve``, ``cg_spmv``), the vector calls (``cg_axpy``, ``cg_ewmul``,
``cg_dot``) and the batched and served solves (``Batch``).  Sizes come from
the library's configurations, tests and benchmark: the 16^3 7-point Laplacian,
the 27-point finite-element systems of 64^3 and 160^3, the batch of uneven
systems with edges in [8, 48], the request stream with edges in [16, 96], and
the vector lengths of its BLAS-1 tests.  Matrices are assembled on the GPU
with torch, as a finite-element program would.

Matrices:
  lap7  7-point Laplacian on an N^3 grid (diagonal 6, neighbours -1)
  q1    trilinear hexahedral (27-point) stiffness on an N^3 grid of interior
        nodes, one lognormal density per element, nodes numbered along the grid
  mesh  the same operator on an irregular mesh: a fifth of the couplings
        absent (the diagonal keeps the row sums), nodes numbered in a locally
        shuffled order, so that rows differ in length and in pattern

A solve returns its solution and whether it converged.  The step count and
the reported residual move with the last rounding of any sum (a residual may
cross the tolerance one step earlier or later), so they are not outputs.
"""
import math

import numpy as np
import torch

import paper_2112_10823_gb300 as cg

# One digit below the 1e-10 that the configurations state: at 1e-10 two solves
# whose sums round differently end up to 1e-9 apart in x (the systems' condition
# numbers reach 1e6); at 1e-11 the solutions agree to about 1e-10.
TOL = 1e-11


def listed():
    return [
        # one small system: 4,096 rows, 7 entries each; launch and synchronisation latency of a whole solve
        {"name": "solve_lap7_16", "op": "solve", "matrix": "lap7", "grid": 16, "mixed": False, "jacobi": False},
        # one ordinary finite-element system (262,144 rows, 6.9 M entries), FP64
        {"name": "solve_q1_64", "op": "solve", "matrix": "q1", "grid": 64, "mixed": False, "jacobi": False},
        # the largest single system of the configurations (4.1 M rows, 109 M entries), FP64
        {"name": "solve_q1_160", "op": "solve", "matrix": "q1", "grid": 160, "mixed": False, "jacobi": False},
        # the same size with the FP32 product and FP64 residual replacement
        {"name": "solve_q1_160_mixed", "op": "solve", "matrix": "q1", "grid": 160, "mixed": True, "jacobi": False},
        # an irregular mesh of 300,763 nodes, preconditioned, FP64
        {"name": "solve_mesh_67_jacobi", "op": "solve", "matrix": "mesh", "grid": 67, "mixed": False, "jacobi": True},
        # the product alone on a small system (13,824 rows): a caller's own Krylov loop, one call after another
        {"name": "spmv_q1_24", "op": "spmv", "matrix": "q1", "grid": 24},
        # the product alone on a large irregular mesh (1,331,000 rows)
        {"name": "spmv_mesh_110", "op": "spmv", "matrix": "mesh", "grid": 110},
        # the vector operations on short vectors: launch latency
        {"name": "vectors_10007", "op": "vectors", "n": 10007},
        # the vector operations on long vectors of odd length
        {"name": "vectors_5000001", "op": "vectors", "n": 5000001},
        # a matrix that is solved once: handle from host arrays, solve, release
        {"name": "once_q1_40", "op": "once", "matrix": "q1", "grid": 40, "mixed": False},
        # many uneven systems solved together (edges 8..48), mixed precision, the requests checked by the library
        {"name": "batch_256_mixed", "op": "batch", "count": 256, "lo": 8, "hi": 48, "mixed": True, "chunk": 0,
         "target_ms": 50, "validate": True},
        # a burst of a served stream (edges 16..96), FP64, continuous batching in rounds of 50 steps
        {"name": "served_40", "op": "batch", "count": 40, "lo": 16, "hi": 96, "mixed": False, "chunk": 50,
         "target_ms": 5, "validate": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "spmv", "vectors", "once", "batch"])
    if op == "vectors":
        return {"op": op, "n": _log(rng, 1000, 64_000_000)}
    if op == "batch":
        served = rng.random() < 0.5
        return {"op": op, "count": _log(rng, 4, 40 if served else 256), "lo": 16 if served else 8,
                "hi": 96 if served else 48, "mixed": rng.random() < 0.5, "chunk": rng.choice([20, 50]) if served else 0,
                "target_ms": rng.choice([5, 50]), "validate": rng.random() < 0.5}
    matrix = rng.choice(["q1", "q1", "lap7", "mesh"])
    case = {"op": op, "matrix": matrix, "grid": _log(rng, 8, {"solve": 150, "spmv": 160, "once": 80}[op])}
    if op != "spmv":
        case["mixed"] = rng.random() < 0.4
    if op == "solve":
        case["jacobi"] = rng.random() < 0.3
    return case


# ------------------------------------------------------------------ matrices

def _grid_rows(N, offsets, values, dev):
    """CSR of an N^3 grid operator: values[..., u] couples a node to the one at offsets[u] (ascending columns)."""
    keep = torch.ones(N, N, N, len(offsets), dtype=torch.bool, device=dev)
    for u, off in enumerate(offsets):
        for axis, d in enumerate(off):
            if d:
                keep[..., u].select(axis, N - 1 if d > 0 else 0).fill_(False)
    n = N ** 3
    keep = keep.reshape(n, -1)
    shift = torch.tensor([(dz * N + dy) * N + dx for dz, dy, dx in offsets], dtype=torch.int32, device=dev)
    cols = torch.arange(n, dtype=torch.int32, device=dev)[:, None] + shift[None, :]
    rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(keep.sum(1), 0)
    return rp.to(torch.int32), cols[keep], values.reshape(n, -1)[keep]


def _lap7(N, dev):
    offsets = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)]
    values = torch.full((N, N, N, 7), -1.0, dtype=torch.float64, device=dev)
    values[..., 3] = 6.0
    return _grid_rows(N, offsets, values, dev)


def _q1(N, gen, dev):
    rho = torch.exp(torch.randn(N + 1, N + 1, N + 1, dtype=torch.float64, device=dev, generator=gen))
    h = 1.0 / (N + 1)
    offsets = [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    values = torch.empty(N, N, N, 27, dtype=torch.float64, device=dev)
    for u, off in enumerate(offsets):
        s = rho
        for axis, d in enumerate(off):  # the elements that hold both nodes
            a, b = s.narrow(axis, 0, N), s.narrow(axis, 1, N)
            s = a + b if d == 0 else (b if d > 0 else a)
        values[..., u] = (h / 3.0, 0.0, -h / 12.0, -h / 12.0)[sum(d != 0 for d in off)] * s
    return _grid_rows(N, offsets, values, dev)


def _mesh(N, gen, dev):
    rp, ci, va = _q1(N, gen, dev)
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=dev), (rp[1:] - rp[:-1]).long())
    cols = ci.long()
    # a coupling (i, j) is there or not for both of its rows
    drop_of = torch.rand(1 << 20, device=dev, generator=gen) < 0.2
    a, b = torch.minimum(rows, cols), torch.maximum(rows, cols)
    drop = drop_of[(a * 40503 + b * 69069 + (a ^ b)) & ((1 << 20) - 1)] & (rows != cols)
    gone = _row_sums(rp, torch.where(drop, va, torch.zeros_like(va)))
    va = torch.where(rows == cols, va + gone[rows], va)
    rows, cols, va = rows[~drop], cols[~drop], va[~drop]
    number = torch.argsort(torch.argsort(torch.arange(n, dtype=torch.float64, device=dev)
                                         + 2048.0 * torch.rand(n, dtype=torch.float64, device=dev, generator=gen)))
    rows, cols = number[rows], number[cols]
    order = torch.argsort(rows * n + cols)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rp.to(torch.int32), cols[order].to(torch.int32), va[order]


def _row_sums(rp, terms):
    return torch.segment_reduce(terms, "sum", offsets=rp.long(), axis=0, unsafe=True)


def _matrix(kind, N, gen, dev):
    if kind == "lap7":
        return _lap7(N, dev)
    return (_q1 if kind == "q1" else _mesh)(N, gen, dev)


def _uniform(n, gen, dev):
    return 2.0 * torch.rand(n, dtype=torch.float64, device=dev, generator=gen) - 1.0


def _generator(seed, dev):
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return gen


def _system(kind, N, seed, dev):
    """Matrix, manufactured solution x* ~ U(-1, 1) and b = A x*."""
    gen = _generator(seed, dev)
    rp, ci, va = _matrix(kind, N, gen, dev)
    xs = _uniform(rp.numel() - 1, gen, dev)
    b = _row_sums(rp, va * xs[ci.long()])
    return rp, ci, va, xs, b


def _edges(case):
    """Grid edges of a batch: uniform on [lo, hi], or for a served stream lognormal around their geometric mean.
    They belong to the case; the seed makes the densities and the right-hand sides."""
    rng = np.random.default_rng([4, case["count"], case["lo"], case["hi"]])
    lo, hi = case["lo"], case["hi"]
    if case["chunk"] == 0:
        return [int(v) for v in rng.integers(lo, hi + 1, size=case["count"])]
    z = rng.standard_normal(case["count"])
    e = np.clip(np.rint(np.exp(0.5 * (math.log(lo) + math.log(hi)) + 0.448 * z)), lo, hi)
    return [int(v) for v in e]


# --------------------------------------------------------------------- cases

def prepare(case, seed):
    dev = torch.device("cuda")
    op = case["op"]
    if op == "vectors":
        gen = _generator(seed, dev)
        x, y, w = (_uniform(case["n"], gen, dev) for _ in range(3))
        return {"op": op, "x": x, "y": y, "w": w, "z": torch.empty_like(x), "d": torch.empty(1, dtype=torch.float64, device=dev)}
    if op == "batch":
        systems = []
        edges = _edges(case)
        xall = torch.zeros(sum(N ** 3 for N in edges), dtype=torch.float64, device=dev)
        at = 0
        for i, N in enumerate(edges):
            rp, ci, va, _, b = _system("q1", N, 1000 * int(seed) + i, dev)
            systems.append(cg.Request(rp, ci, va, b, xall[at:at + N ** 3], tol=TOL, maxit=10 * N ** 3, tag=i))
            at += N ** 3
        bt = cg.Batch(precision=cg.CG_PREC_MIXED if case["mixed"] else cg.CG_PREC_FP64, budget_bytes=12 << 30,
                      chunk_iters=case["chunk"], group_target_ms=case["target_ms"], validate=case["validate"])
        return {"op": op, "batch": bt, "requests": systems, "x": xall}
    rp, ci, va, xs, b = _system(case["matrix"], case["grid"], seed, dev)
    precision = cg.CG_PREC_MIXED if case.get("mixed") else cg.CG_PREC_FP64
    if op == "once":
        host = [t.cpu().numpy() for t in (rp, ci, va, b)]
        return {"op": op, "host": host, "precision": precision}
    h = cg.cg_create(rp, ci, va, precision=precision,
                     preconditioner=cg.CG_PRECOND_JACOBI if case.get("jacobi") else cg.CG_PRECOND_NONE)
    if op == "spmv":
        return {"op": op, "h": h, "x": xs, "y": torch.empty_like(xs)}
    return {"op": op, "h": h, "b": b}


def run(state):
    op = state["op"]
    if op == "vectors":
        cg.cg_axpy(-0.731, state["x"], state["w"])
        cg.cg_ewmul(state["x"], state["y"], state["z"])
        cg.cg_dot(state["x"], state["y"], state["d"])
        return {"axpy": state["w"], "ewmul": state["z"], "dot": state["d"]}
    if op == "spmv":
        cg.cg_spmv(state["h"], state["x"], state["y"])
        return {"y": state["y"]}
    if op == "solve":
        x = torch.zeros_like(state["b"])
        res = cg.cg_solve(state["h"], state["b"], x, tol=TOL)
        return {"x": x, "converged": res.ok}
    if op == "once":
        rp, ci, va, b = state["host"]
        x = np.zeros_like(b)
        with cg.cg_create(rp, ci, va, precision=state["precision"]) as h:
            res = cg.cg_solve(h, b, x, tol=TOL)
        return {"x": x, "converged": res.ok}
    bt = state["batch"]
    res = bt.wait_all(bt.submit(state["requests"]))
    return {"x": state["x"], "converged": all(r.done and r.status == cg.CG_OK for r in res)}


def exact(case, seed):
    dev = torch.device("cuda")
    op = case["op"]
    if op == "vectors":
        gen = _generator(seed, dev)
        x, y, w = (_uniform(case["n"], gen, dev) for _ in range(3))
        return {"axpy": -0.731 * x + w, "ewmul": x * y, "dot": torch.sum(x * y).reshape(1)}
    if op == "batch":
        xs = [_system("q1", N, 1000 * int(seed) + i, dev)[3] for i, N in enumerate(_edges(case))]
        return {"x": torch.cat(xs), "converged": None}
    rp, ci, va, xs, b = _system(case["matrix"], case["grid"], seed, dev)
    if op == "spmv":
        return {"y": b}
    return {"x": xs if op == "solve" else xs.cpu().numpy(), "converged": None}


def _entries(kind, N):
    if kind == "lap7":
        return 7 * N ** 3 - 6 * N ** 2
    full = (3 * N - 2) ** 3
    return full if kind == "q1" else int(0.8 * (full - N ** 3)) + N ** 3


def _solve_work(kind, N, mixed, jacobi):
    """A solve of the usual number of steps (it grows with the grid edge), each reading the matrix once."""
    n, nnz = N ** 3, _entries(kind, N)
    steps = (4.8 if kind == "lap7" else 2.9 if jacobi else 7.0) * N
    return {"bytes": steps * ((8 if mixed else 12) * nnz + 4 * n + 48 * n), "flops": steps * (2 * nnz + 10 * n)}


def work(case):
    op = case["op"]
    if op == "vectors":
        return {"bytes": 64 * case["n"] + 8, "flops": 5 * case["n"]}
    if op == "batch":
        parts = [_solve_work("q1", N, case["mixed"], False) for N in _edges(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, nnz = case["grid"] ** 3, _entries(case["matrix"], case["grid"])
    if op == "spmv":
        return {"bytes": 12 * nnz + 4 * (n + 1) + 16 * n, "flops": 2 * nnz}
    return _solve_work(case["matrix"], case["grid"], case.get("mixed", False), case.get("jacobi", False))
