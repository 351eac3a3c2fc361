"""Diagonal blocks in LU form, by block columns of eight with the inverses by
block rows (csrc/lublock.cuh), against the oracle: widths at and next to the
edges of a block column, of a warp and of the widest panel, in FP64 and FP32,
and replaced pivots.  Dense diagonally dominant matrices: growth below 2, so
1e-12 in FP64 and 1e-4 in FP32.
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


def _dense(n, seed):
    g = np.random.default_rng([seed, 2])
    A = g.uniform(-1.0, 1.0, (n, n))
    A[np.arange(n), np.arange(n)] = 1.5 * n * np.where(g.uniform(size=n) < 0.5, -1.0, 1.0)
    return sp.csc_matrix(A)


@pytest.mark.parametrize("n,width", [(1, 64), (7, 64), (8, 64), (9, 64), (16, 64), (31, 64), (33, 64), (64, 64),
                                     (65, 96), (97, 160), (160, 160), (200, 64), (330, 160)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_lu_blocks_match_oracle(n, width, prec):
    A = _dense(n, n)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "lu", ordering=spx.SPX_ORDER_NATURAL, max_width=width)
    h.factorize(vals, prec)
    F = oracle.lu(A, h.perm())
    Lx, Ut = h.factor_on_pattern(F.sym.Lp, F.sym.Li, lu=True)
    bound = 1e-12 if prec == "fp64" else 1e-4
    assert np.linalg.norm(Lx - F.Lx) <= bound * np.linalg.norm(F.Lx)
    assert np.linalg.norm(Ut - F.Ut) <= bound * np.linalg.norm(F.Ut)
    B = inputs.rhs(n, 2, 1)
    X, _ = h.solve(B)
    assert oracle.backward_error(A, X, B) <= (1e-13 if prec == "fp64" else 1e-12)
    h.free()


@pytest.mark.parametrize("col", [0, 7, 8, 40])
def test_small_pivot_is_replaced(col):
    A = sp.lil_matrix(_dense(41, 3))
    A[col, :] = 0.0
    A[:, col] = 0.0
    A[col, col] = 1e-300
    A = sp.csc_matrix(A)
    A.data[A.data == 0.0] = 1e-300
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "lu", ordering=spx.SPX_ORDER_NATURAL, max_width=64)
    h.factorize(vals, "fp64")
    assert h.info()["npivot_repl"] == 1
    h.free()
