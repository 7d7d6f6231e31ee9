"""FP64 trailing update by error-free splitting on the BF16 tensor cores
(Ozaki scheme) against the oracle, through the C ABI.

Bars:
  - operands that the slices represent exactly (7-bit integers times a power
    of two): the update equals C - A B bit for bit (every step is exact);
  - any FP64 operands: |C_oz - C_ref| <= u ((0.35 k + 4) 2^(e_i + f_j)
    + (|A||B|)_ij) + 2u |C_ref|, C_ref the compensated (Dot2) update of the
    oracle, u = 2^-53 and 2^e_i, 2^f_j the powers of two just above the
    largest |A(i, :)| and |B(:, j)|: dropped slice pairs (p + q >= 8) < 0.222 k,
    splitting remainders < 0.126 k, the 15 rounded right shifts <= 3.82 (in
    units of u 2^(e_i + f_j)), then the conversion of the integer sum and the
    subtraction round once each;
  - the certified form: within the FP64 dot product's k u (|A||B|)_ij + u |C|
    everywhere, refusing exactly the blocks that its rule refuses;
  - the factorization with this update: the FP64 bars (pivots equal to the
    oracle's, factors and x within the roundoff bounds, scaled residual < 16).
"""
import numpy as np
import pytest

import oracle as O
from paper_2202_13995_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2202_13995_gb300 import lu
    c = lu.Context()
    yield c
    torch.cuda.synchronize()
    c.close()


def _rm(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _dev(a):
    import torch
    from paper_2202_13995_gb300 import lu
    a = np.asarray(a, dtype=np.float64)
    t = lu.colmajor_empty(a.shape[0], a.shape[1])
    t.copy_(torch.from_numpy(np.asfortranarray(a)))
    return t


def _expo(x, axis):
    """e with 2^(e-1) <= max|x| < 2^e along axis (0 for an all-zero line)."""
    mx = np.abs(x).max(axis=axis)
    e = np.zeros(mx.shape, dtype=np.int64)
    nz = mx > 0
    e[nz] = np.frexp(mx[nz])[1]
    return e


def _bound(Am, Bm, ref):
    k = Am.shape[1]
    sc = np.ldexp(1.0, (_expo(Am, 1)[:, None] + _expo(Bm, 0)[None, :]).astype(np.int64))
    return EPS * ((0.35 * k + 4) * sc + np.abs(Am) @ np.abs(Bm)) + 2 * EPS * np.abs(ref)


def _run(ctx, Cm, Am, Bm):
    c = _rm(Cm)
    ctx.step_gemm_ozaki(c, _rm(Am), _rm(Bm))
    return c.cpu().numpy()


# m = 32 takes the kernel's stacked form (four slices of A per 128-row box)
@pytest.mark.parametrize("m,n,k", [(300, 300, 256), (128, 128, 64), (1, 1, 1), (257, 130, 200), (129, 385, 33),
                                   (32, 300, 256), (32, 129, 200), (32, 1300, 64)])
def test_exact_on_sliceable_operands(ctx, m, n, k):
    rng = np.random.default_rng(m * 7 + n + k)
    Am = rng.integers(-127, 128, (m, k)) / 128.0 * 2.0 ** rng.integers(-3, 4, (m, 1))
    Bm = rng.integers(-127, 128, (k, n)) / 128.0 * 2.0 ** rng.integers(-3, 4, (1, n))
    Cm = rng.integers(-2 ** 20, 2 ** 20, (m, n)) * 2.0 ** -14
    want = Cm - Am @ Bm  # exact: every partial sum fits in 53 bits
    got = _run(ctx, Cm, Am, Bm)
    assert np.array_equal(got, want)
    assert ctx.status() == 0


@pytest.mark.parametrize("m,n,k", [(333, 333, 256), (200, 520, 37), (130, 140, 1), (640, 384, 256), (32, 520, 256),
                                   (32, 1000, 37)])
def test_error_bound_against_dot2(ctx, m, n, k):
    rng = np.random.default_rng(m + n + k)
    Am = I.uniform_np(30 + k, 0, np.arange(m * k, dtype=np.uint64)).reshape(m, k)
    Bm = I.uniform_np(30 + k, 1, np.arange(k * n, dtype=np.uint64)).reshape(k, n)
    Cm = rng.standard_normal((m, n))
    ref = O.gemm_update_dot2(Cm, Am, Bm)
    got = _run(ctx, Cm, Am, Bm)
    bound = _bound(Am, Bm, ref)
    err = np.abs(got - ref)
    assert (err <= bound).all(), float((err / bound).max())
    # the plain FP64 update (the oracle's) errs by the same order
    scale = k * np.ldexp(1.0, (_expo(Am, 1)[:, None] + _expo(Bm, 0)[None, :]).astype(np.int64))
    plain = np.abs(O.gemm_update(Cm, Am, Bm) - ref)
    assert (err / scale).max() <= 8 * max((plain / scale).max(), 2.0 ** -56)


def test_wide_dynamic_range_zero_lines(ctx):
    m, n, k = 260, 190, 256
    rng = np.random.default_rng(5)
    Am = rng.standard_normal((m, k)) * 2.0 ** rng.integers(-300, 300, (m, 1))
    Bm = rng.standard_normal((k, n)) * 2.0 ** rng.integers(-300, 300, (1, n))
    Am[7, :] = 0.0
    Bm[:, 11] = 0.0
    Am[9, 3] = 2.0 ** 40  # one dominant entry in a row
    Cm = rng.standard_normal((m, n))
    ref = O.gemm_update_dot2(Cm, Am, Bm)
    got = _run(ctx, Cm, Am, Bm)
    assert (np.abs(got - ref) <= _bound(Am, Bm, ref)).all()
    assert np.array_equal(got[7, :], Cm[7, :])
    assert np.array_equal(got[:, 11], Cm[:, 11])


@pytest.mark.parametrize("ea,eb", [(-500, -500), (-510, -540), (-520, -560), (-1000, -993), (-1000, -995), (-1020, -1020),
                                   (500, -1060)])
def test_products_at_the_end_of_the_exponent_range(ctx, ea, eb):
    """Products that are normal, subnormal or below every FP64 number, with an accumulator of
    their size and one that hides them: the bound of above plus two roundings of subnormals."""
    m, n, k = 160, 140, 64
    rng = np.random.default_rng(9)
    Am = np.ldexp(rng.random((m, k)) - 0.5, ea)
    Bm = np.ldexp(rng.random((k, n)) - 0.5, eb)
    for Cm in (np.ldexp(rng.random((m, n)) - 0.5, max(ea + eb, -1000)), rng.random((m, n)) - 0.5):
        LD = np.longdouble  # (the compensated update's own error terms underflow here)
        ref = (Cm.astype(LD) - Am.astype(LD) @ Bm.astype(LD))
        err = np.abs(_run(ctx, Cm, Am, Bm).astype(LD) - ref)
        sc = np.ldexp(LD(1.0), (_expo(Am, 1)[:, None] + _expo(Bm, 0)[None, :]).astype(np.int64))
        bound = LD(EPS) * ((0.35 * k + 4) * sc + np.abs(Am).astype(LD) @ np.abs(Bm).astype(LD) + 2 * np.abs(ref)) + \
            2 * np.ldexp(LD(1.0), -1074)
        assert (err <= bound).all()


def test_non_finite_operand_is_reported(ctx):
    from paper_2202_13995_gb300 import lu
    m, n, k = 64, 64, 16
    Am = np.ones((m, k))
    Am[3, 4] = np.nan
    c = _rm(np.zeros((m, n)))
    ctx.step_gemm_ozaki(c, _rm(Am), _rm(np.ones((k, n))))
    assert ctx.status() == lu.LU_ERANGE


def _lead(x, axis):
    """The magnitudes' leading base-128 digits of the lines along axis (of |x| 2^-e rounded to 56 bits)."""
    e = np.expand_dims(_expo(x, axis), axis)
    return np.floor(np.rint(np.ldexp(np.abs(x), 56 - e)) / 2.0 ** 49)


CERT_LINE = 6866  # (0.35 * 64 + 4) / 63 * 2^14


def _refused(Am, Bm):
    """Blocks of 32 x 64 with an element whose magnitude product is below the line (zero lines pass)."""
    m, n = Am.shape[0], Bm.shape[1]
    small = _lead(Am, 1) @ _lead(Bm, 0) < CERT_LINE
    small &= np.abs(Am).max(1)[:, None] > 0
    small &= np.abs(Bm).max(0)[None, :] > 0
    pad = np.zeros(((m + 31) // 32 * 32, (n + 63) // 64 * 64), dtype=bool)
    pad[:m, :n] = small
    return pad.reshape(pad.shape[0] // 32, 32, -1, 64).any(axis=(1, 3))


def _peaked(rng, m, k, s):
    """Rows of entries of size s with one of size 1: sum |a b| is far below the lines' maxima."""
    X = (rng.random((m, k)) - 0.5) * 2 * s
    X[np.arange(m), rng.integers(0, k, m)] = rng.choice([-1.0, 1.0], m) * (0.5 + 0.5 * rng.random(m))
    return X * 2.0 ** rng.integers(-30, 30, (m, 1))


# sizes of the smaller entries from "every block refused" to "none"; ragged blocks, k of 1 to 4 chunks
@pytest.mark.parametrize("m,n,k", [(333, 517, 64), (129, 65, 64), (32, 700, 100), (640, 640, 128), (300, 260, 256)])
def test_certificate_on_either_side_of_its_line(ctx, m, n, k):
    rng = np.random.default_rng(m + n + k)
    shares = []
    for s in np.array([0.02, 0.12, 0.13, 0.137, 0.14, 0.143, 0.146, 0.15, 0.16, 0.5]) * (64.0 / k) ** 0.5 * 1.3:
        Am, Bm = _peaked(rng, m, k, s), _peaked(rng, n, k, s).T.copy()
        Am[m // 3] = 0.0
        Bm[:, n // 2] = 0.0
        Cm = (rng.random((m, n)) - 0.5) * np.abs(Am).max(1)[:, None] * np.abs(Bm).max(0)[None, :]
        Cm[m // 3], Cm[:, n // 2] = 1.5, 2.5
        want = _refused(Am, Bm)
        ref = O.gemm_update_dot2(Cm, Am, Bm)
        bound = k * EPS * (np.abs(Am) @ np.abs(Bm)) * (1 + 1e-9) + 2 * EPS * np.abs(ref)
        c, d, w = _rm(Cm), _rm(Cm), _rm(Cm)
        listed, raised = ctx.step_gemm_cert(c, _rm(Am), _rm(Bm))
        assert listed == want.sum() and raised == (want.sum() * 10 > want.size * 9)
        got = c.cpu().numpy()
        assert (np.abs(got - ref) <= bound).all(), float((np.abs(got - ref) / np.maximum(bound, 1e-300)).max())
        assert np.array_equal(got[m // 3], Cm[m // 3]) and np.array_equal(got[:, n // 2], Cm[:, n // 2])
        # refused blocks are the multiply-add update's, bit for bit, and with the flag every block is
        ctx.step_gemm(d, _rm(Am), _rm(Bm), "f64")
        plain = d.cpu().numpy()
        mask = np.kron(want, np.ones((32, 64), dtype=bool))[:m, :n]
        assert np.array_equal(got[mask], plain[mask])
        listed, raised = ctx.step_gemm_cert(w, _rm(Am), _rm(Bm), whole=True)
        assert (listed, raised) == (0, False) and np.array_equal(w.cpu().numpy(), plain)
        shares.append(want.mean())
    assert shares[0] == 1.0 and shares[-1] == 0.0 and any(0 < x < 1 for x in shares), shares
    assert ctx.status() == 0


def test_certificate_and_non_finite_lines(ctx):
    """A line with an infinity or a NaN has its blocks refused, across a zero line too."""
    rng = np.random.default_rng(2)
    m, n, k = 100, 200, 64
    for bad in (np.nan, np.inf):
        Am, Bm, Cm = rng.random((m, k)) - 0.5, rng.random((k, n)) - 0.5, rng.random((m, n)) - 0.5
        Am[40, 3] = Bm[5, 150] = bad
        Am[90] = 0.0
        Bm[:, 20] = 0.0
        c, d = _rm(Cm), _rm(Cm)
        listed, raised = ctx.step_gemm_cert(c, _rm(Am), _rm(Bm))
        ctx.step_gemm(d, _rm(Am), _rm(Bm), "f64")
        # block row 1 (row 40: 4 blocks) and block column 2 (column 150: 4 blocks), one shared
        assert (listed, raised) == (7, False)
        assert np.array_equal(np.isfinite(c.cpu().numpy()), np.isfinite(d.cpu().numpy()))
        assert ctx.status() == 0


def test_k_out_of_range_is_rejected(ctx):
    from paper_2202_13995_gb300 import lu
    with pytest.raises(lu.LuError):
        ctx.step_gemm_ozaki(_rm(np.zeros((4, 4))), _rm(np.zeros((4, 257))), _rm(np.zeros((257, 4))))
    for k in (63, 257):
        with pytest.raises(lu.LuError) as e:
            ctx.step_gemm_cert(_rm(np.zeros((4, 4))), _rm(np.zeros((4, k))), _rm(np.zeros((k, 4))))
        assert e.value.code == -4


@pytest.mark.parametrize("n,nb", [(1, 64), (65, 64), (500, 64), (777, 100), (1500, 256), (2048, 128)])
def test_factor_solve_ozaki(ctx, n, nb):
    A = I.hpl_matrix(n, 40 + n)
    B = I.hpl_rhs(n, 1, 40 + n)
    f = ctx.factor(_dev(A), "f64", nb, ozaki=True)
    assert f.info == 0
    LUo, ipo, info = O.getrf(A, nb)
    assert np.array_equal(f.ipiv().cpu().numpy(), ipo)
    LUg = f.lu().cpu().numpy()
    assert np.abs(LUg - LUo).max() <= 256 * n * EPS * max(1.0, np.abs(LUo).max())
    x = _dev(B)
    f.solve_(x)
    xo = O.getrs(LUo, ipo, B)
    kappa = O.cond1_est(LUo, ipo, O.norm_one(A))
    xg = x.cpu().numpy()
    assert np.abs(xg - xo).max() / np.abs(xo).max() <= max(1e-10, 10 * kappa * EPS), kappa
    assert O.scaled_residual(A, xg, B)[0] < 16.0
    assert ctx.status() == 0


def test_ozaki_nopiv(ctx):
    n = 1024
    A = I.hpl_matrix(n, 9, diag_shift=n / 4.0)
    B = I.hpl_rhs(n, 2, 9)
    f = ctx.factor(_dev(A), "f64", 128, nopiv=True, ozaki=True)
    assert f.info == 0
    LUo, info = O.getrf_nopiv(A, 128)
    LUg = f.lu().cpu().numpy()
    assert np.abs(LUg - LUo).max() <= 256 * n * EPS * max(1.0, np.abs(LUo).max())
    x = _dev(B)
    f.solve_(x)
    assert (O.scaled_residual(A, x.cpu().numpy(), B) < 16.0).all()


def test_ozaki_flag_needs_f64(ctx):
    from paper_2202_13995_gb300 import lu
    A = _dev(I.hpl_matrix(64, 1))
    with pytest.raises(lu.LuError):
        ctx.factor(A, "bf16", 0, ozaki=True)
    with pytest.raises(lu.LuError):
        ctx.factor(A, "f64", 512, ozaki=True)


@pytest.mark.slow
def test_full_size_f64_ozaki_n16384(ctx):
    """n = 16384, nb = 256 with the split update: all 16384 pivots and x
    against the oracle's (the FP64 bars), the first block step's U rows, and
    the scaled residual of the solve."""
    import torch
    from tests.conftest import check_full_size_f64
    n, nb = 16384, 256
    Ad = I.hpl_matrix_torch(n, 2, device="cuda")
    bd = I.hpl_rhs_torch(n, 1, 2, device="cuda")
    f = ctx.factor(Ad, "f64", nb, ozaki=True)
    LUg = f.lu()
    x = bd.clone()
    f.solve_(x)
    torch.cuda.synchronize()
    xg = check_full_size_f64(f, x)
    A = Ad.cpu().numpy()
    O.set_threads(0)
    LU1, ip1, _ = O.getrf(A, nb, ksteps=1)
    U_rows = LUg[:nb, :].cpu().numpy()
    assert np.abs(U_rows - LU1[:nb, :]).max() <= 1e-12 * max(1.0, np.abs(LU1[:nb, :]).max())
    assert O.scaled_residual(A, xg, bd.cpu().numpy()[:, 0]) < 16.0
