"""Offline sweep of the block width nb: writes csrc/nb_table.h, the table that
lu_factor(nb = 0) and lu_fact_bytes read.

    python -m paper_2202_13995_gb300.tune [--out PATH] [--reps K]

nb is the block width of the paper's blocked iteration (its LOCAL_MEM_BLOCK
blocking parameter): the width of each factored block column and the inner
dimension of the trailing update.  For each factorization kind (plain FP64, FP64
with the split tensor-core update, BF16/FP16 mixed
with refinement, FP32) and each size bucket, the sweep times whole solves
(factor + solve or refinement, CUDA events on the library's stream, the best
of K after a warm-up) on the seeded HPL-shaped matrices of the benchmarks and
keeps the fastest candidate.  The choice depends on (kind, n) only, so a
request's result never depends on what else runs.  Rebuild the library
afterwards (__graft_entry__.build()).
"""
from __future__ import annotations

import argparse
import os
import sys
import time

HERE = os.path.dirname(os.path.abspath(__file__))
TABLE = os.path.join(HERE, "csrc", "nb_table.h")

# kind -> (lu precision, split update, diagonal shift / n, candidates)
KINDS = {
    "f64": ("f64", False, 0.0, (64, 128, 192, 256)),
    "f64_split": ("f64", True, 0.0, (64, 128, 192, 256)),
    "mixed": ("bf16", False, 0.25, (64, 128, 256, 384, 512)),
    "f32": ("f32", False, 0.25, (64, 128, 256, 384, 512)),
}
KIND_ID = {"f64": 0, "f64_split": 1, "mixed": 2, "f32": 3}
# size buckets (upper bounds) and the size each is measured at; the plain FP64
# solve at n = 32768 takes seconds and keeps the n = 16384 choice
BUCKETS = [(800, 600), (1280, 1024), (3072, 2048), (4608, 4096), (7168, 6000), (12288, 8192), (24576, 16384),
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
            best = min(times, key=times.get)
            rows.append((kind, nmax, n, times, best))
            prev = best
    ctx.close()
    return rows


def write_table(rows, path: str, command: str, device: str):
    lines = [
        "// Block width nb of lu_factor(nb = 0), by factorization kind and size:",
        "// the fastest candidate of an offline sweep of whole solves (factor +",
        "// solve or refinement) on the benchmarks' seeded matrices.  Generated by",
        f"//   {command}",
        f"// on {device}; times in ms (best of the repetitions after a warm-up).",
        "#pragma once",
        "",
        "namespace gb {",
        "",
        "// kind: 0 FP64 (CUDA-core update), 1 FP64 (split tensor-core update),",
        "// 2 BF16 / FP16 mixed, 3 FP32.  The first entry of the kind whose nmax",
        "// is at least n applies.",
        "struct NbEntry {",
        "  int kind, nmax, nb;",
        "};",
        "",
        "constexpr NbEntry kNbTable[] = {",
    ]
    for kind, nmax, n, times, best in rows:
        tt = ", ".join(f"nb {k}: {v:.3f}" for k, v in sorted(times.items())) or f"not measured: n = {n} keeps the smaller size's choice"
        lines.append(f"    {{{KIND_ID[kind]}, {nmax}, {best}}},  // {kind}, measured at n = {n}: {tt}")
    lines += ["};", "", "}  // namespace gb", ""]
    with open(path, "w") as f:
        f.write("\n".join(lines))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--out", default=TABLE)
    ap.add_argument("--reps", type=int, default=2)
    args = ap.parse_args()
    import torch
    rows = sweep(args.reps)
    cmd = "python -m paper_2202_13995_gb300.tune" + (f" --reps {args.reps}" if args.reps != 2 else "")
    write_table(rows, args.out, cmd, torch.cuda.get_device_name(0))
    print(f"wrote {args.out}")


if __name__ == "__main__":
    sys.exit(main())
