"""Diagonal blocks wider than 64 columns: factored in fixed point
(csrc/fxblock.cuh), or in FP64 where fixed point cannot hold the block.
Dense matrices, so that the root panels are as wide as max_width allows.

Fixed point rounds at 2^-60 of sqrt(a_ii a_jj), so the FP64 factor meets the
bounds of the FP64 kernels (1e-12) whatever the rows' scales; a pivot that is
not positive is reported at the same column, and replaced in the
single-precision modes, as by the FP64 kernels that take 64 columns at most.
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


def _dense(n, seed, scale=None, cond=None):
    g = np.random.default_rng([seed, 0])
    q, _ = np.linalg.qr(g.standard_normal((n, n)))
    d = np.exp(g.uniform(0.0, np.log(cond or 100.0), n))
    A = (q * d) @ q.T
    if scale is not None:
        A = A * scale[:, None] * scale[None, :]
    A = np.tril(A)
    return sp.csc_matrix(A + np.tril(A, -1).T)


def _factor(A, width, prec):
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_NATURAL, max_width=width)
    h.factorize(vals, prec)
    return h


@pytest.mark.parametrize("n,width", [(65, 128), (72, 128), (97, 97), (128, 128), (152, 152), (153, 160), (160, 160),
                                     (300, 152)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_wide_blocks_match_oracle(n, width, prec):
    A = _dense(n, n)
    h = _factor(A, width, prec)
    F = oracle.cholesky(A, h.perm())
    Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
    bound = 1e-12 if prec == "fp64" else 1e-4
    assert np.linalg.norm(Lx - F.Lx) <= bound * np.linalg.norm(F.Lx)
    B = inputs.rhs(n, 2, 1)
    X, info = h.solve(B)
    assert oracle.backward_error(A, X, B) <= (1e-13 if prec == "fp64" else 1e-12)
    h.free()


@pytest.mark.parametrize("spread", [1e3, 1e60])
def test_rows_of_very_different_scales(spread):
    g = np.random.default_rng(3)
    scale = np.exp(g.uniform(-np.log(spread), np.log(spread), 128))
    A = _dense(128, 4, scale)
    h = _factor(A, 128, "fp64")
    F = oracle.cholesky(A, h.perm())
    Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
    assert np.max(np.abs(Lx - F.Lx) / scale[F.sym.Li]) <= 1e-12 * 10.0   # entries of L are at most 10 row scales
    h.free()


@pytest.mark.parametrize("col", [0, 77, 127])
def test_failed_pivot_is_reported_and_replaced(col):
    A = sp.lil_matrix(_dense(128, 5))
    A[col, col] = -1.0
    A = sp.csc_matrix(A)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_NATURAL, max_width=128)
    with pytest.raises(spx.SpxError) as e:
        h.factorize(vals, "fp64")
    assert e.value.status == spx.SPX_ERR_NOT_SPD and h.info()["bad_col"] == col
    h.factorize(vals, "fp32")
    assert h.info()["npivot_repl"] >= 1
    h.free()


def test_nearly_singular_block():
    """A pivot near 2^-46 of its diagonal: below what fixed point takes."""
    A = _dense(96, 6).toarray()
    L = np.linalg.cholesky(A)
    L[50, 50] = np.sqrt(A[50, 50]) * 2.0 ** -23
    A = L @ L.T
    A = np.tril(A)
    A = sp.csc_matrix(A + np.tril(A, -1).T)
    h = _factor(A, 96, "fp64")
    F = oracle.cholesky(A, h.perm())
    Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
    M = sp.csc_matrix((Lx, F.sym.Li, F.sym.Lp)).toarray()
    P = A.toarray()[np.ix_(h.perm(), h.perm())]
    assert np.linalg.norm(M @ M.T - P) <= 1e-14 * np.linalg.norm(P)
    h.free()
