"""What a user of this solver has it do, as cases that can be timed and checked.

Five kinds of use, all through the package's public calls (paper_2202_13995_gb300.lu):

  solve    one dense FP64 system, factored and solved (gesv): `Context.factor` + `Factor.solve_`,
           with the plain FP64 update or the split one (`ozaki`), as the caller asks
  refine   one system by a low-precision factor and FP64 refinement: `Context.factor` + `Factor.refine`,
           with FP32, BF16 or FP16 factors, with pivoting or (the paper's variant) without
  again    new right-hand sides for a factor that the program has kept: `Factor.solve_` or `Factor.refine`
  batch    many small systems planned once: `Batch.run`
  serve    a burst of requests to a solve server, some of them for factors that it holds: `Server.submit` / `wait`

Matrices are those of the LINPACK workloads: i.i.d. uniform[-0.5, 0.5) ("shift" 0: pivoting moves a row in
nearly every column) or the same plus shift * n on the diagonal (the diagonally dominant form of HPL-AI, which
low-precision factors are used for), in some cases with its rows in random order ("shuffle": every column's
pivot is far from the diagonal, the matrix well conditioned).  Right-hand sides are uniform[-0.5, 0.5).
"""
import math
import os

# what the server's documentation asks a serving process to set before its CUDA context exists
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import torch

from paper_2202_13995_gb300 import lu

GB = 1 << 30


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one small FP64 system, where launches and the latency of a column decide
        {"name": "f64_n150", "kind": "solve", "prec": "f64", "ozaki": False, "n": 150, "nrhs": 1, "shift": 0.0},
        # an ordinary FP64 system of an odd size with a few right-hand sides
        {"name": "f64_n1023_r4", "kind": "solve", "prec": "f64", "ozaki": False, "n": 1023, "nrhs": 4, "shift": 0.0},
        # a large FP64 system with the plain update (the LINPACK run itself)
        {"name": "f64_n8192", "kind": "solve", "prec": "f64", "ozaki": False, "n": 8192, "nrhs": 1, "shift": 0.0},
        # FP64 with the split update on the tensor cores, a ragged size
        {"name": "f64_split_n7001_r8", "kind": "solve", "prec": "f64", "ozaki": True, "n": 7001, "nrhs": 8, "shift": 0.0},
        # an ordinary mixed-precision solve: BF16 update, a size between two table entries
        {"name": "bf16_n1500_r2", "kind": "refine", "prec": "bf16", "nopiv": False, "n": 1500, "nrhs": 2, "shift": 0.25},
        # the paper's no-pivot variant at a middle size, FP16 operands
        {"name": "fp16_nopiv_n6000_r8", "kind": "refine", "prec": "fp16", "nopiv": True, "n": 6000, "nrhs": 8, "shift": 0.25},
        # the largest: the HPL-AI run (mixed precision, one right-hand side)
        {"name": "bf16_n32768", "kind": "refine", "prec": "bf16", "nopiv": False, "n": 32768, "nrhs": 1, "shift": 0.25},
        # a large mixed solve with a block of right-hand sides
        {"name": "bf16_n12288_r32", "kind": "refine", "prec": "bf16", "nopiv": False, "n": 12288, "nrhs": 32, "shift": 0.25},
        # FP32 factors of a general matrix: every panel pivots
        {"name": "f32_general_n2500", "kind": "refine", "prec": "f32", "nopiv": False, "n": 2500, "nrhs": 1, "shift": 0.0},
        # new right-hand sides for kept FP64 factors (a time-stepping or Newton loop)
        {"name": "again_f64_n5000_r3", "kind": "again", "prec": "f64", "n": 5000, "nrhs": 3, "shift": 0.0},
        # many small systems planned once (n 32..512, 1..8 right-hand sides)
        {"name": "batch_1000", "kind": "batch", "count": 1000, "nmin": 32, "nmax": 512, "kmax": 8, "shift": 1.0},
        # a burst of requests to a server, as in the served workload (log-uniform sizes)
        {"name": "serve_48", "kind": "serve", "prec": "fp16", "count": 48, "nmin": 64, "nmax": 4096, "kmax": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "split", "refine", "refine", "general", "again", "batch", "serve"])
    if kind == "solve":
        return {"kind": "solve", "prec": "f64", "ozaki": False, "n": _log(rng, 24, 7000), "nrhs": rng.choice([1, 1, 2, 3, 7, 16]),
                "shift": rng.choice([0.0, 0.0, 0.25])}
    if kind == "split":
        return {"kind": "solve", "prec": "f64", "ozaki": True, "n": _log(rng, 500, 12000), "nrhs": rng.choice([1, 1, 4, 16]),
                "shift": 0.0}
    if kind == "refine":
        return {"kind": "refine", "prec": rng.choice(["bf16", "fp16", "f32"]), "nopiv": rng.random() < 0.3,
                "n": _log(rng, 200, 14000), "nrhs": rng.choice([1, 1, 2, 5, 16, 20, 32]), "shift": 0.25}
    if kind == "general":
        if rng.random() < 0.5:
            return {"kind": "refine", "prec": "f32", "nopiv": False, "n": _log(rng, 200, 3000), "nrhs": rng.choice([1, 2, 6]),
                    "shift": 0.0}
        return {"kind": "refine", "prec": rng.choice(["f32", "bf16", "fp16"]), "nopiv": False, "n": _log(rng, 200, 6000),
                "nrhs": rng.choice([1, 2, 6]), "shift": 0.25, "shuffle": True}
    if kind == "again":
        prec = rng.choice(["f64", "f64", "bf16", "f32"])
        return {"kind": "again", "prec": prec, "n": _log(rng, 100, 9000), "nrhs": rng.choice([1, 1, 3, 8, 24, 32]),
                "shift": 0.0 if prec == "f64" else 0.25}
    if kind == "batch":
        lo = rng.choice([8, 32, 64])
        return {"kind": "batch", "count": _log(rng, 12, 1500), "nmin": lo, "nmax": _log(rng, 2 * lo, 512),
                "kmax": rng.choice([1, 3, 8]), "shift": rng.choice([0.5, 1.0])}
    return {"kind": "serve", "prec": rng.choice(["fp16", "bf16"]), "count": rng.randrange(12, 60), "nmin": 64,
            "nmax": _log(rng, 700, 4096), "kmax": rng.choice([1, 8, 16])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _matrix(case, g):
    """A column-major (n, n) FP64 tensor: uniform[-0.5, 0.5) plus shift * n on the diagonal, its rows shuffled if asked."""
    n = case["n"]
    a = torch.empty((n, n), dtype=torch.float64, device="cuda").uniform_(-0.5, 0.5, generator=g)  # a[j] is column j
    if case["shift"]:
        a.diagonal().add_(case["shift"] * n)
    if case.get("shuffle"):
        a = a[:, torch.randperm(n, generator=g, device="cuda")].contiguous()
    return a.t()


def _rhs(n, k, g):
    return torch.empty((k, n), dtype=torch.float64, device="cuda").uniform_(-0.5, 0.5, generator=g).t()


def _sizes(case):
    """(n, nrhs) of the systems of a batch or a burst: fixed by the case, so that its work is."""
    g = torch.Generator().manual_seed(case["count"] * 1000003 + case["nmax"])
    u = torch.rand(case["count"], generator=g, dtype=torch.float64).tolist()
    k = torch.randint(1, case["kmax"] + 1, (case["count"],), generator=g).tolist()
    lo, hi = case["nmin"], case["nmax"]
    if case["kind"] == "batch":
        ns = [min(hi, lo + int(x * (hi - lo + 1))) for x in u]
    else:
        ns = [int(round(lo * (hi / lo) ** x)) for x in u]
    return list(zip(ns, k))


def _systems(case, seed):
    """The systems of a batch or a burst: views into one buffer of matrices, one of right-hand sides."""
    sizes, g = _sizes(case), _gen(seed)
    shift = case.get("shift", 0.25)
    # each matrix and right-hand side starts 16-byte aligned, as separate allocations would
    up = lambda v: (v + 1) // 2 * 2  # noqa: E731
    abuf = torch.empty(sum(up(n * n) for n, _ in sizes), dtype=torch.float64, device="cuda")
    bbuf = torch.empty(sum(up(n * k) for n, k in sizes), dtype=torch.float64, device="cuda")
    abuf.uniform_(-0.5, 0.5, generator=g)
    bbuf.uniform_(-0.5, 0.5, generator=g)
    xbuf = torch.zeros_like(bbuf)
    A, B, X = [], [], []
    oa = ob = 0
    for n, k in sizes:
        a = abuf[oa:oa + n * n].view(n, n)
        a.diagonal().add_(shift * n)
        A.append(a.t())
        B.append(bbuf[ob:ob + n * k].view(k, n).t())
        X.append(xbuf[ob:ob + n * k].view(k, n).t())
        oa, ob = oa + up(n * n), ob + up(n * k)
    return A, B, X, xbuf


def _held(case):
    """How many of a burst's requests are for factors that the server holds already (3 in 10)."""
    return case["count"] * 3 // 10


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "refine", "again"):
        g = _gen(seed)
        n, k = case["n"], case["nrhs"]
        s = {"case": case, "A": _matrix(case, g), "B": _rhs(n, k, g), "ctx": lu.Context()}
        s["X"] = lu.colmajor_empty(n, k)
        if kind == "again":
            s["factor"] = s["ctx"].factor(s["A"], case["prec"], 0)
        return s
    A, B, X, xbuf = _systems(case, seed)
    if kind == "batch":
        ctx = lu.Context()
        info = torch.full((case["count"],), -9, dtype=torch.int32, device="cuda")
        return {"case": case, "ctx": ctx, "plan": lu.Batch(ctx, A, B, X), "xbuf": xbuf, "info": info}
    server = lu.Server(60 * GB, case["prec"], max_slots=24)
    torch.cuda.synchronize()  # the server's slots have streams of their own
    held = _held(case)
    t = [server.submit(A[i], B[i], X[i], factor_key=i + 1, keep_factor=True) for i in range(held)]
    for x in t:
        if server.wait(x).status:
            raise RuntimeError("a request that leaves its factor failed")
    return {"case": case, "server": server, "reqs": list(zip(A, B, X)), "xbuf": xbuf, "held": held}


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        f = s["ctx"].factor(s["A"], case["prec"], 0, ozaki=case["ozaki"])
        s["X"].copy_(s["B"])
        f.solve_(s["X"])
        ipiv = f.ipiv()
        f.free()
        return {"x": s["X"], "ipiv": ipiv}
    if kind == "refine":
        f = s["ctx"].factor(s["A"], case["prec"], 0, nopiv=case["nopiv"])
        f.refine(s["A"], s["B"], s["X"], 16.0, 50)
        f.free()
        return {"x": s["X"]}
    if kind == "again":
        if case["prec"] == "f64":
            s["X"].copy_(s["B"])
            s["factor"].solve_(s["X"])
        else:
            s["factor"].refine(s["A"], s["B"], s["X"], 16.0, 50)
        return {"x": s["X"]}
    if kind == "batch":
        s["plan"].run(s["info"])
        return {"x": s["xbuf"], "info": s["info"]}
    srv = s["server"]
    tickets = [srv.submit(a, b, x, factor_key=i + 1 if i < s["held"] else 0, use_resident=i < s["held"])
               for i, (a, b, x) in enumerate(s["reqs"])]
    status = [srv.wait(t).status for t in tickets]
    return {"x": s["xbuf"], "status": torch.tensor(status, dtype=torch.int32)}


# ------------------------------------------------------------------ what a pass cannot do without
def _one(n, k, factor, wbytes=0):
    """One system: A and B read, X written; the factorization's and the solve's operations."""
    return 8.0 * n * n + 16.0 * n * k + wbytes, (2.0 * n ** 3 / 3.0 if factor else 0.0) + 2.0 * n * n * k


def work(case):
    kind = case["kind"]
    if kind in ("solve", "refine"):
        b, f = _one(case["n"], case["nrhs"], True)
    elif kind == "again":
        n, k = case["n"], case["nrhs"]
        b, f = _one(n, k, False)  # FP64: the factors are what is read
        if case["prec"] != "f64":
            b, f = b + 4.0 * n * n, 2.0 * f  # FP32 factors, and A for the residual: a solve and a residual
    else:
        held = _held(case) if kind == "serve" else 0
        parts = [_one(n, k, i >= held) for i, (n, k) in enumerate(_sizes(case))]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ what an output may be off by
def tolerance(case):
    """Measured against exact() over several seeds of every listed case and of drawn ones, times about four; the
    condition number of a general (uniform) matrix is of order n with a heavy tail, so its seeds differ by up to
    a hundred.  General matrices: FP64 solves up to 7e-11 off, refined FP32 factors up to 4e-9.  Dominant ones:
    FP64 solves 2.4e-15; a refined solution stops anywhere below a scaled residual of 16, which bounds its error by
    about 16 n 2^-53 (condition numbers of 1 to 4; seen: up to 1.4e-12 at n = 1500)."""
    if case["kind"] in ("solve", "again") and case["prec"] == "f64":
        return {"rel": 1e-9 if case["shift"] == 0.0 else 1e-13}
    if case.get("shift", 0.25) == 0.0:
        return {"rel": 2e-8}
    return {"rel": 64.0 * case.get("n", case.get("nmax")) * 2.0 ** -53}


# ------------------------------------------------------------------ the same in 64 bits
def _exact(A, B, shift):
    n = A.shape[0]
    if n <= 20000:
        return torch.linalg.solve(A, B)
    # diagonally dominant and too large to factor in a few seconds: x <- x + (b - A x) / (shift n), whose error
    # shrinks by about 2 sqrt(n / 12) / (shift n) a step
    X = B / (shift * n)
    for _ in range(14):
        X = X + (B - A @ X) / (shift * n)
    return X


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "refine", "again"):
        g = _gen(seed)
        A, B = _matrix(case, g), _rhs(case["n"], case["nrhs"], g)
        x = _exact(A, B, case["shift"])
        return {"x": x, "ipiv": None} if kind == "solve" else {"x": x}
    A, B, X, xbuf = _systems(case, seed)
    for a, b, x in zip(A, B, X):
        x.copy_(torch.linalg.solve(a, b))
    return {"x": xbuf, "info": None} if kind == "batch" else {"x": xbuf, "status": None}
