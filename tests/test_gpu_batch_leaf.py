"""Narrow panels of the batched LU, one per warp with their rows in registers:
every group size of the update (1 to 4, 5 to 8, 9 to 16, 17 to 32 rows below
the block; past 32 the whole CTA), widths up to 8, both precisions, and pivots
so large or small that quotients leave the range of the reciprocal's product.

Banded matrices in their natural order, diagonally dominant: factors with
entries of order one per row scale and growth below 2, so the substitution's
rounding stays below 1e-12 in FP64 and 1e-4 in FP32.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _banded(n, band, seed, scale):
    g = np.random.default_rng([seed, band])
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    A = np.where(np.abs(i - j) <= band, g.uniform(-1.0, 1.0, (n, n)), 0.0)
    A[np.arange(n), np.arange(n)] = (2 * band + 2.0) * np.where(g.uniform(size=n) < 0.5, -1.0, 1.0)
    return sp.csc_matrix(A * scale)


@pytest.mark.parametrize("band", [1, 4, 5, 8, 9, 16, 17, 31, 32, 33, 45])
@pytest.mark.parametrize("width", [1, 3, 8])
@pytest.mark.parametrize("prec,scale", [("fp64", 1.0), ("fp64", 1e-200), ("fp32", 1.0), ("fp32", 1e25),
                                        ("fp32", 1e-25)])
def test_banded_factors_match_oracle(band, width, prec, scale):
    mats = [_banded(n, band, n, scale) for n in (band + 1, 97, 130)]
    arrs = [inputs.csc_arrays(A) for A in mats]
    b = spx.batch_analyze([(cp, ri) for cp, ri, _ in arrs], ordering=spx.SPX_ORDER_NATURAL, max_width=width)
    vals = np.concatenate([v for _, _, v in arrs])
    rhs = np.concatenate([inputs.rhs(A.shape[0], 1, 7).ravel() for A in mats])
    X, _ = b.run(vals, rhs, precision=prec)
    bound, o = (1e-12 if prec == "fp64" else 1e-4), 0
    for s, A in enumerate(mats):
        F = oracle.lu(A, b.perm(s))
        Lx, Ut = b.factor_on_pattern(s, F.sym.Lp, F.sym.Li)
        assert np.linalg.norm(Lx - F.Lx) <= bound * np.linalg.norm(F.Lx), s
        assert np.linalg.norm((Ut - F.Ut) / scale) <= bound * np.linalg.norm(F.Ut / scale), s
        n = A.shape[0]
        x, r = X[o:o + n], rhs[o:o + n]
        assert oracle.backward_error(sp.csc_matrix(A / scale), x * scale, r) <= (1e-13 if prec == "fp64" else 1e-4)
        o += n
    b.free()
