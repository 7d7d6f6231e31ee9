"""Offline sweep of the block width nb: prints the rows that csrc/nb_table.h, the
table that lu_factor(nb = 0) and lu_fact_bytes read, is chosen from.

    python -m paper_2202_13995_gb300.tune [--out PATH] [--reps K]

nb is the block width of the paper's blocked iteration (its LOCAL_MEM_BLOCK
blocking parameter): the width of each factored block column and the inner
dimension of the trailing update.  For each factorization kind (plain FP64, FP64
with the split tensor-core update, BF16/FP16 mixed with refinement, FP32) and each
size bucket, the sweep times whole solves (factor + solve or refinement, CUDA events
on the library's stream, the best of K after a warm-up) on the seeded HPL-shaped
matrices of the benchmarks and names the fastest candidate.  The table takes that,
or a narrower width within 3 percent of it that the neighbouring sizes prefer.  The
choice depends on (kind, n) only, so a request's result never depends on what else
runs.  Rebuild the library after a change (__graft_entry__.build()).
"""
from __future__ import annotations

import argparse
import sys
import time

# kind -> (lu precision, split update, diagonal shift / n, candidates)
KINDS = {
    "f64": ("f64", False, 0.0, (32, 64, 96, 128, 192, 256)),
    "f64_split": ("f64", True, 0.0, (64, 128, 192, 256)),
    "mixed": ("bf16", False, 0.25, (64, 128, 192, 256, 384, 512)),
    "f32": ("f32", False, 0.25, (64, 128, 192, 256, 384, 512)),
}
KIND_ID = {"f64": 0, "f64_split": 1, "mixed": 2, "f32": 3}
# size buckets (upper bounds) and the size each is measured at; the plain FP64
# solve at n = 32768 takes seconds and keeps the n = 16384 choice
BUCKETS = [(800, 600), (1280, 1024), (3072, 2048), (4608, 4096), (7168, 5800), (12288, 8192), (24576, 16384),
           (1 << 30, 32768)]
SKIP = {("f64", 32768)}


def time_solve(ctx, stream, kind, n, nb, reps):
    import torch
    from paper_2202_13995_gb300 import inputs as I
    from paper_2202_13995_gb300 import lu
    prec, split, shift, _ = KINDS[kind]
    A = I.hpl_matrix_torch(n, 3, diag_shift=shift * n, device="cuda")
    B = I.hpl_rhs_torch(n, 1, 3, device="cuda")
    X = lu.colmajor_empty(n, 1)

    def one():
        f = ctx.factor(A, prec, nb, sync=False, ozaki=split)
        if prec in ("bf16", "fp16", "f32"):
            f.refine(A, B, X, 16.0, 50)
        else:
            X.copy_(B)
            f.solve_(X)
        f.free()

    one()
    best = float("inf")
    for _ in range(reps):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        one()
        e1.record(stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    del A, B, X
    torch.cuda.empty_cache()
    return best


def sweep(reps: int):
    import torch
    from paper_2202_13995_gb300 import lu
    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream()
    ctx = lu.Context(stream)
    rows = []  # (kind, nmax, n, {nb: ms}, best nb)
    for kind, (_, _, _, cands) in KINDS.items():
        prev = None
        for nmax, n in BUCKETS:
            if (kind, n) in SKIP:
                rows.append((kind, nmax, n, {}, prev))
                continue
            times = {}
            for nb in cands:
                if nb > n:
                    continue
                t0 = time.time()
                times[nb] = time_solve(ctx, stream, kind, n, nb, reps)
                print(f"{kind:9s} n={n:6d} nb={nb:4d}: {times[nb]:10.3f} ms  ({time.time() - t0:.1f} s)", flush=True)
            prev = min(times, key=times.get)
            rows.append((kind, nmax, n, times, prev))
    ctx.close()
    return rows


def table_rows(rows):
    """The rows as kNbTable's lines, with the fastest width of each."""
    out = []
    for kind, nmax, n, times, best in rows:
        tt = ", ".join(f"nb {k}: {v:.3f}" for k, v in sorted(times.items())) or f"not measured: n = {n} keeps the smaller size's choice"
        out.append(f"    {{{KIND_ID[kind]}, {nmax}, {best}}},  // {kind}, measured at n = {n}: {tt}")
    return "\n".join(out) + "\n"


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--out", help="also write the rows to this file")
    ap.add_argument("--reps", type=int, default=2)
    args = ap.parse_args()
    text = table_rows(sweep(args.reps))
    print(text, end="")
    if args.out:
        with open(args.out, "w") as f:
            f.write(text)


if __name__ == "__main__":
    sys.exit(main())
