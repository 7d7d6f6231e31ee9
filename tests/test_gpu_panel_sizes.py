"""Panels at the edges of the cluster kernel's shapes (rows per CTA, CTAs per
cluster, the last size that fits and the first that goes to the cooperative
kernel), in arithmetic that is exact in FP32 and FP64, with many ties and with
zero columns: pivots, L and U equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (31, 31), (32, 5), (33, 33), (64, 64), (65, 17), (129, 100), (257, 3), (512, 64), (513, 63),
         (1025, 33), (2049, 128), (5625, 64), (5626, 64), (8192, 32), (8193, 32)]


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2202_13995_gb300 import lu
    c = lu.Context()
    yield c
    torch.cuda.synchronize()
    c.close()


def _exact_panel(m, w, seed, zero_col):
    # entries of L in {0, +-1/2, +-1} and of U in {+-1, +-2}, banded: every product and
    # sum is a short dyadic number, and magnitudes tie in nearly every column
    rng = np.random.default_rng(seed)
    L = np.tril(rng.integers(-2, 3, size=(m, w)) / 2.0, -1)
    L[np.arange(w), np.arange(w)] = 1.0
    U = np.triu(rng.choice([-2.0, -1.0, 1.0, 2.0], size=(w, w)))
    U = np.where(np.triu(np.ones((w, w)), 6) > 0, 0.0, U)
    if zero_col is not None:
        U[:, zero_col] = 0.0
    return (L @ U)[rng.permutation(m)]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("m,w", SIZES)
def test_panel_at_size_edges(ctx, m, w, prec):
    import torch
    for seed, zc in ((m + w, None), (m + 2 * w, w // 2)):
        P = _exact_panel(m, w, seed, zc)
        LUo, ipo, info_o = O.getf2(P)
        # (the elimination stays exact: the oracle's FP64 factors are FP32 numbers)
        if not np.array_equal(LUo, LUo.astype(np.float32).astype(np.float64)):
            assert prec == "f64" or zc is not None
            if prec == "f32":
                continue
        Pd = torch.from_numpy(np.ascontiguousarray(P)).to("cuda", torch.float64 if prec == "f64" else torch.float32)
        ipiv = torch.zeros(w, dtype=torch.int32, device="cuda")
        info = torch.zeros(1, dtype=torch.int32, device="cuda")
        ctx.step_panel(Pd, ipiv, info, prec)
        assert ctx.status() == 0
        assert info.item() == info_o
        assert np.array_equal(ipiv.cpu().numpy(), ipo)
        assert np.array_equal(Pd.cpu().numpy().astype(np.float64), LUo)


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
