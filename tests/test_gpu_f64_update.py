"""The plain FP64 factorization's trailing update (certified split products,
with the FP64 CUDA cores where the certificate fails or the update is small):
factors against the oracle at the edges of the rule that chooses it, and the
componentwise backward error of badly scaled, banded and sparse systems, which
a split update without the certificate loses."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_2202_13995_gb300 import inputs as I

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2202_13995_gb300 import lu
    c = lu.Context()
    yield c
    torch.cuda.synchronize()
    c.close()


def _dev(a):
    import torch
    from paper_2202_13995_gb300 import lu
    t = lu.colmajor_empty(a.shape[0], a.shape[1])
    t.copy_(torch.from_numpy(np.asfortranarray(a)))
    return t


# one step, the first size that takes the split update, the last that does not, ragged last blocks,
# widths below, at and above the certificate's least and most
@pytest.mark.parametrize("n,nb", [(703, 64), (704, 64), (705, 64), (705, 63), (600, 65), (1030, 64), (777, 128),
                                  (900, 256), (1000, 257),
                                  # the top solve in halves: from 3000 columns on, blocks of 256
                                  (3255, 256), (3256, 256), (3301, 256), (3301, 255)])
@pytest.mark.parametrize("nopiv", [False, True])
def test_factors_at_the_edges_of_the_rule(ctx, n, nb, nopiv):
    A = I.hpl_matrix(n, 300 + n + nb, diag_shift=n / 4 if nopiv else 0.0)
    f = ctx.factor(_dev(A), "f64", nb, nopiv=nopiv)
    LUo, ipo, info = O.getrf(A)
    assert f.info == info == 0
    assert np.array_equal(f.ipiv().cpu().numpy(), ipo)
    assert np.abs(f.lu().cpu().numpy() - LUo).max() <= 256 * n * U * np.abs(LUo).max()
    f.free()


def _system(kind, n, rng):
    A = rng.random((n, n)) - 0.5
    i = np.arange(n)
    if kind == "row_scaled":
        A *= 10.0 ** (30 * rng.random((n, 1)) - 15)
    elif kind == "rows_far_apart":
        A *= 10.0 ** (200 * rng.random((n, 1)) - 100)
    elif kind == "column_scaled":
        A *= 10.0 ** (30 * rng.random((1, n)) - 15)
    elif kind == "banded":
        A = A * (np.abs(i[:, None] - i[None, :]) < 40) + 2 * np.eye(n)
    elif kind == "sparse":
        A = A * (rng.random((n, n)) < 0.02) + 2 * np.eye(n)
    elif kind == "half_scaled":
        A[: n // 2] *= 1e-12
    return A


@pytest.mark.parametrize("n,nb", [(1100, 64), (1100, 128), (3301, 256)])
@pytest.mark.parametrize("kind", ["row_scaled", "rows_far_apart", "column_scaled", "banded", "sparse", "half_scaled"])
def test_componentwise_backward_error(ctx, kind, n, nb):
    """|b - A x| <= c (|A||x| + |b|) row by row.  Partial pivoting gives
    |b - A x| <= 3 n u |P^T L||U||x| (N. Higham, Accuracy and Stability of Numerical
    Algorithms, theorem 9.4); the factor beside the rows' own sums is the oracle's."""
    rng = np.random.default_rng(17)
    A = _system(kind, n, rng)
    x0 = rng.random((n, 1)) - 0.5
    B = A @ x0
    f = ctx.factor(_dev(A), "f64", nb)
    X = _dev(B)
    f.solve_(X)
    x = X.cpu().numpy()
    LUo, ipo, info = O.getrf(A)
    assert f.info == info == 0
    p = np.arange(n)
    for j, q in enumerate(ipo):
        p[j], p[q - 1] = p[q - 1], p[j]
    L, R = np.tril(LUo, -1) + np.eye(n), np.triu(LUo)
    bound = np.empty((n, 1))
    bound[p] = 3 * n * U * (np.abs(L) @ (np.abs(R) @ np.abs(x)))
    r = np.abs((B.astype(np.longdouble) - A.astype(np.longdouble) @ x.astype(np.longdouble)).astype(float))
    assert (r <= bound + U * np.abs(B)).all(), float((r / (bound + U * np.abs(B))).max())
    f.free()


@pytest.mark.parametrize("nopiv", [False, True])
@pytest.mark.parametrize("s", [1e-295, 1e-302, 1e-307])
def test_blocks_far_apart(ctx, s, nopiv):
    """Two clusters with a coupling so small that its products with itself underflow
    (the split's scale 2^(e_i + f_j - 54) is then below every FP64 number)."""
    n, nb = 900, 64
    A = I.hpl_matrix(n, 3, diag_shift=n / 4)
    A[:450, 450:] *= s
    A[450:, :450] *= s
    f = ctx.factor(_dev(A), "f64", nb, nopiv=nopiv)
    LUo, ipo, info = O.getrf(A)
    assert f.info == info == 0
    assert np.array_equal(f.ipiv().cpu().numpy(), ipo)
    assert np.abs(f.lu().cpu().numpy() - LUo).max() <= 256 * n * U * np.abs(LUo).max()
    f.free()


@pytest.mark.parametrize("w", [1, 31, 32, 33, 64, 100, 257, 512])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 130])
def test_top_solve_edges(ctx, w, N):
    """L^-1 X by substitution in FP64: |x - x_ref| <= 2 w u |L^-1| |L| |x| (both
    round each of at most w terms; Higham, theorem 8.5)."""
    import torch
    from paper_2202_13995_gb300 import lu
    rng = np.random.default_rng(w * 1000 + N)
    M = rng.random((w, w + N)) - 0.5
    M[:, :w] *= 4.0 / (4.0 + w)
    Md = torch.from_numpy(M.copy()).cuda()
    # (the C entry itself: Context.step_trsm takes a one-row operand's width for its row stride)
    assert lu.load().lu_step_trsm(ctx._h, lu._prec("f64"), w, N, C.c_void_p(Md.data_ptr()), w + N,
                                  C.c_void_p(Md.data_ptr() + 8 * w), w + N) == 0
    ctx.stream.synchronize()
    L = np.tril(M[:, :w], -1) + np.eye(w)
    want = O.trsm_unit_lower(L, M[:, w:])
    bound = 2 * w * U * (np.abs(np.linalg.inv(L)) @ (np.abs(L) @ np.abs(want))) + U * np.abs(want)
    got = Md.cpu().numpy()
    assert (np.abs(got[:, w:] - want) <= bound).all()
    assert np.array_equal(got[:, :w], M[:, :w])


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (7, 33, 5), (86, 86, 64), (384, 384, 63), (550, 550, 32), (554, 1000, 33),
                                   (1088, 1088, 31), (1089, 1089, 64)])
def test_small_update_edges(ctx, m, n, k):
    """C - A B: within k u (|A||B|) + u |C - A B| of the compensated update on either side."""
    import torch
    rng = np.random.default_rng(m + n + k)
    A, B, Cm = rng.random((m, k)) - 0.5, rng.random((k, n)) - 0.5, rng.random((m, n)) - 0.5
    C = torch.from_numpy(Cm.copy()).cuda()
    ctx.step_gemm(C, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), "f64")
    ref = O.gemm_update_dot2(Cm, A, B)
    bound = (k + 1) * U * (np.abs(A) @ np.abs(B)) + 2 * U * (np.abs(Cm) + np.abs(ref))
    assert (np.abs(C.cpu().numpy() - ref) <= bound).all()


def test_non_finite_entries_are_reported(ctx):
    from paper_2202_13995_gb300 import lu
    for bad in (np.nan, np.inf):
        for at in ((900, 5), (3, 900), (800, 700)):
            A = I.hpl_matrix(1000, 5)
            A[at] = bad
            with pytest.raises(lu.LuError) as e:
                ctx.factor(_dev(A), "f64", 64)
            assert e.value.code == lu.LU_ERANGE


@pytest.mark.parametrize("nopiv", [False, True])
@pytest.mark.parametrize("n,nb", [(900, 64), (3300, 256)])
def test_update_on_the_fp64_cores_by_flag(ctx, n, nb, nopiv):
    """LU_FACTOR_DFMA: the oracle's factors, without one split launch (the cast phase), where the
    default splits."""
    A = I.hpl_matrix(n, 31 + n, diag_shift=n / 4 if nopiv else 0.0)
    LUo, ipo, info = O.getrf(A)
    casts = {}
    for dfma in (False, True):
        ctx.profile(True)
        ctx.profile_read()
        f = ctx.factor(_dev(A), "f64", nb, nopiv=nopiv, dfma=dfma)
        casts[dfma] = ctx.profile_read()["cast"][1]
        ctx.profile(False)
        assert f.info == info == 0
        assert np.array_equal(f.ipiv().cpu().numpy(), ipo)
        assert np.abs(f.lu().cpu().numpy() - LUo).max() <= 256 * n * U * np.abs(LUo).max()
        f.free()
    assert casts[True] == 0 < casts[False]


def test_flag_combinations_that_are_refused(ctx):
    from paper_2202_13995_gb300 import lu
    A = _dev(I.hpl_matrix(64, 1))
    for prec, kw in (("bf16", {}), ("f32", {}), ("f64", {"ozaki": True})):
        with pytest.raises(lu.LuError) as e:
            ctx.factor(A, prec, 0, dfma=True, **kw)
        assert e.value.code == -7


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(900, 5), (3, 900), (3, 3), (700, 850)])
def test_non_finite_entries_without_pivoting(ctx, bad, at):
    """Without pivoting nothing is searched and nothing refused: a non-finite entry spreads to the
    same entries by the certified update as by multiply-adds, across a zero row and column too."""
    n = 1000
    A = I.hpl_matrix(n, 5, diag_shift=n / 4)
    A[495, :495] = 0.0
    A[:505, 505] = 0.0
    A[at] = bad
    out = []
    for dfma in (False, True):
        f = ctx.factor(_dev(A), "f64", 64, nopiv=True, dfma=dfma)
        assert f.info == 0
        out.append(f.lu().cpu().numpy())
        f.free()
    ok = np.isfinite(out[1])
    assert not ok.all() and np.array_equal(np.isfinite(out[0]), ok)
    assert np.abs(out[0][ok] - out[1][ok]).max() <= 256 * n * U * np.abs(out[1][ok]).max()
