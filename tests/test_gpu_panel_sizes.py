"""Panels at the edges of the shapes of the kernels that hold the panel in shared
memory (rows per CTA, CTAs per cluster, the sizes around the lines between the
cluster, the grid and the cooperative kernel), in arithmetic that is exact in FP32 and FP64, with a zero column and
with ties across CTAs: pivots, L and U equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (31, 31), (32, 5), (33, 33), (64, 64), (65, 17), (129, 100), (257, 3), (512, 64), (513, 63),
         (1025, 33), (2049, 128), (5625, 64), (5626, 64), (8192, 32), (8193, 32),
         (1562, 64), (1563, 64), (2187, 64), (2188, 64), (4865, 100), (6240, 128), (7001, 129), (9000, 512)]


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2202_13995_gb300 import lu
    c = lu.Context()
    yield c
    torch.cuda.synchronize()
    c.close()


def _exact_panel(m, w, seed, zero_col):
    # A = P^T L U with |l| < 1 and short dyadic entries: elimination is exact
    rng = np.random.default_rng(seed)
    L = np.tril(rng.integers(-7, 8, size=(m, w)) / 8.0, -1)
    L[np.arange(w), np.arange(w)] = 1.0
    U = np.triu(rng.integers(-8, 9, size=(w, w)).astype(np.float64))
    U[np.arange(w), np.arange(w)] = rng.integers(1, 9, size=w) * rng.choice([-1.0, 1.0], size=w)
    if zero_col is not None:
        U[:, zero_col] = U[zero_col, :] = 0.0
    return (L @ U)[rng.permutation(m)]


def _panel(ctx, P, prec):
    import torch
    Pd = torch.from_numpy(np.ascontiguousarray(P)).to("cuda", torch.float64 if prec == "f64" else torch.float32)
    w = P.shape[1]
    ipiv = torch.zeros(w, dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.step_panel(Pd, ipiv, info, prec)
    assert ctx.status() == 0
    return Pd.cpu().numpy().astype(np.float64), ipiv.cpu().numpy(), info.item()


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("m,w", SIZES)
def test_panel_at_size_edges(ctx, m, w, prec):
    for seed, zc in ((m + w, None), (m + 2 * w, w - 1)):
        P = _exact_panel(m, w, seed, zc)
        LUo, ipo, info_o = O.getf2(P)
        assert info_o == (0 if zc is None else zc + 1)
        LU, ipiv, info = _panel(ctx, P, prec)
        assert info == info_o
        assert np.array_equal(ipiv, ipo)
        assert np.array_equal(LU, LUo)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("m", [40, 700, 3000])
def test_ties_go_to_the_first_row(ctx, m, prec):
    """Equal magnitudes in different CTAs, either sign, in a column that an
    interchange has reordered: the pivot is the first of them."""
    P = np.zeros((m, 3))
    P[:, 0] = 0.5
    P[m // 3, 0], P[m - 1, 0] = -2.0, 2.0
    P[:, 1] = np.where(np.arange(m) % 7 == 3, -4.0, 4.0)
    P[:, 2] = np.arange(m) % 5
    LUo, ipo, _ = O.getf2(P)
    assert ipo[0] == m // 3 + 1
    LU, ipiv, _ = _panel(ctx, P, prec)
    assert np.array_equal(ipiv, ipo)
    d = np.abs(LU - LUo).max()
    assert d <= 8 * (2.0 ** -53 if prec == "f64" else 2.0 ** -24) * np.abs(LUo).max()


def test_permutation_record_reaches_the_other_columns(ctx):
    """A factorization whose panels fit the cluster kernel: P A = L U with the
    interchanges applied to every column, for widths around its row groups."""
    import torch
    from paper_2202_13995_gb300 import inputs as I
    for n, nb in ((97, 32), (300, 33), (700, 64), (1111, 96)):
        A = I.hpl_matrix(n, 7 + n)
        f = ctx.factor(torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t(), "f64", nb)
        LUo, ipo, info_o = O.getrf(A, nb)
        assert f.info == info_o == 0
        assert np.array_equal(f.ipiv().cpu().numpy(), ipo)
        d = np.abs(f.lu().cpu().numpy() - LUo).max()
        assert d <= 256 * n * 2.0 ** -53 * np.abs(LUo).max()
        f.free()


@pytest.mark.parametrize("n,nb,prec", [(8300, 1, "f32"), (8300, 2, "f32"), (6400, 16, "f64")])
def test_permutation_record_of_narrow_grid_panels(ctx, n, nb, prec):
    """Panels of few columns on the grid, where the permutation record's count is zeroed
    and counted up within a column or two: |P A - L U| <= n u |L||U| (Higham, theorem 9.3)
    in every column, which a row missing from the record would break by O(1)."""
    import torch
    from paper_2202_13995_gb300 import inputs as I
    A = I.hpl_matrix_torch(n, 19 + nb, device="cuda")
    f = ctx.factor(A, prec, nb)
    assert f.info == 0
    p = np.arange(n)
    for j, q in enumerate(f.ipiv().cpu().numpy()):
        p[j], p[q - 1] = p[q - 1], p[j]
    LU = f.lu().double()
    f.free()
    if prec == "f32":
        A = A.float().double()
    L, R = torch.tril(LU, -1), torch.triu(LU)
    L.diagonal().fill_(1.0)
    d = (A[torch.from_numpy(p).cuda()] - L @ R).abs()
    u = 2.0 ** -24 if prec == "f32" else 2.0 ** -53
    assert bool((d <= n * u * (L.abs() @ R.abs())).all())
