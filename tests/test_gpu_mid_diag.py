"""Diagonal blocks of 33 to 64 columns on the level walk: factored in fixed
point (csrc/fxblock.cuh), or in FP64 where fixed point cannot hold the block (a
scaled inverse of 8 or more, a pivot that is tiny or not positive).  Dense
matrices, so that the panels are as wide as max_width allows.

Fixed point rounds at 2^-60 of sqrt(a_ii a_jj) and the inverse at 2^-56, so the
factor meets the bounds of the FP64 kernels (1e-12; FP32: 1e-4).
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


def _dense(n, seed, cond=100.0, spread=1.0):
    g = np.random.default_rng([seed, 1])
    q, _ = np.linalg.qr(g.standard_normal((n, n)))
    scale = np.exp(g.uniform(-np.log(spread), np.log(spread), n)) if spread > 1.0 else np.ones(n)
    A = np.tril((q * np.exp(g.uniform(0.0, np.log(cond), n))) @ q.T * scale[:, None] * scale[None, :])
    return sp.csc_matrix(A + np.tril(A, -1).T), scale


def _factor(A, prec):
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_NATURAL, max_width=64, queue_panels=-1)
    h.factorize(vals, prec)
    return h


# cond 1e6: scaled inverses far past 8, so the FP64 way
@pytest.mark.parametrize("n", [33, 40, 57, 63, 64, 100, 190])
@pytest.mark.parametrize("prec,cond,spread", [("fp64", 100.0, 1.0), ("fp64", 1e6, 1.0), ("fp64", 100.0, 1e30),
                                              ("fp32", 100.0, 1.0), ("fp32", 100.0, 1e6)])
def test_blocks_match_oracle(n, prec, cond, spread):
    A, scale = _dense(n, n, cond, spread)
    h = _factor(A, prec)
    F = oracle.cholesky(A, h.perm())
    Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
    rows = scale[F.sym.Li]
    bound = 1e-12 if prec == "fp64" else 1e-4
    assert np.linalg.norm((Lx - F.Lx) / rows) <= bound * np.linalg.norm(F.Lx / rows)
    if spread == 1.0:
        B = inputs.rhs(n, 2, 1)
        X, _ = h.solve(B)
        assert oracle.backward_error(A, X, B) <= (1e-13 if prec == "fp64" else 1e-12)
    h.free()


@pytest.mark.parametrize("col", [0, 31, 32, 63])
def test_failed_pivot_is_reported_and_replaced(col):
    A = sp.lil_matrix(_dense(64, 5)[0])
    A[col, col] = -1.0
    cp, ri, vals = inputs.csc_arrays(sp.csc_matrix(A))
    h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_NATURAL, max_width=64, queue_panels=-1)
    with pytest.raises(spx.SpxError) as e:
        h.factorize(vals, "fp64")
    assert e.value.status == spx.SPX_ERR_NOT_SPD and h.info()["bad_col"] == col
    h.factorize(vals, "fp32")
    assert h.info()["npivot_repl"] >= 1
    h.free()
