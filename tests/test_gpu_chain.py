"""The mixed factorization's two streams and dependent launches at the sizes where
they begin and end: the last columns' lookahead (2200 rows left), and the block
column's launches that start before their predecessor has ended (up to 4864 rows
below).  The lookahead changes the order of launches, not of any sum, so the
factors agree bit for bit with those of a context without it."""
import os

import numpy as np
import pytest

from paper_2202_13995_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nopiv", [False, True])
@pytest.mark.parametrize("n,nb", [(2455, 256), (2456, 256), (2457, 256), (4992, 128), (4993, 128), (5121, 256)])
def test_factor_bits_without_lookahead(monkeypatch, n, nb, nopiv):
    import torch
    from paper_2202_13995_gb300 import lu
    A = I.hpl_matrix_torch(n, 11 + n, diag_shift=n / 4, device="cuda")
    out = []
    for off in (False, True):
        if off:
            monkeypatch.setenv("GB300LU_NO_LOOKAHEAD", "1")
        with lu.Context() as ctx:
            f = ctx.factor(A, "bf16", nb, nopiv=nopiv)
            out.append(f.lu().cpu().numpy())
            B = I.hpl_rhs_torch(n, 1, 5, device="cuda")
            X = lu.colmajor_empty(n, 1)
            iters, resid = f.refine(A, B, X, 16.0, 50)
            assert float(np.max(resid)) < 16.0
            f.free()
            torch.cuda.synchronize()
    assert np.array_equal(out[0], out[1])
