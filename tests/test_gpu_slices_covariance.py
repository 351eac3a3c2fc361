"""FP64 Cholesky by slices on smooth covariance matrices, whose diagonal blocks
are ill-conditioned: elimination inside a block leaves pivots far below the
diagonal entries.  Both paths' panel TRSM is a product with the block's inverse,
so what either may lose grows with the block's condition; the slices may lose
no more than FP64 multiply-adds: entry (i, j) of L L^T against A's, in units of
sqrt(a_ii a_jj), is within twice the error of the general path plus 4 units of
rounding, and every matrix that the general path factors is factored.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _covariance(n, nugget, seed, spread):
    """exp(-|x - y|^2 / (2 0.3^2)) over random points of the unit square, and the unknowns' scales."""
    g = np.random.default_rng([seed, n])
    x = g.uniform(0.0, 1.0, (n, 2))
    d2 = ((x[:, None, :] - x[None, :, :]) ** 2).sum(2)
    A = np.exp(-d2 / (2 * 0.3 ** 2)) + nugget * np.eye(n)
    s = np.exp(g.uniform(-spread, spread, n))
    A = np.tril(A * s[:, None] * s[None, :])
    return A + np.tril(A, -1).T


@pytest.mark.parametrize("width,general", [(64, 1 << 30), (128, 0)])   # general: the queue, the levels on the CUDA cores
@pytest.mark.parametrize("nugget", [1e-4, 1e-8, 1e-10])
@pytest.mark.parametrize("seed,spread", [(1, 0.0), (2, 0.0), (3, 0.0), (4, 10.0)])
def test_smooth_covariance(width, general, nugget, seed, spread):
    n = 256
    A = _covariance(n, nugget, seed, spread)
    cp, ri, vals = inputs.csc_arrays(sp.csc_matrix(A))
    root = np.sqrt(np.diag(A))
    err = {}
    for region in (-1, general):
        h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_NATURAL, max_width=width, queue_panels=region)
        p = h.perm()
        Lp = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
        Li = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
        h.factorize(vals, "fp64")
        L = sp.csc_matrix((h.factor_on_pattern(Lp, Li), Li, Lp), shape=(n, n)).toarray()
        err[region] = np.max(np.abs(L @ L.T - A[np.ix_(p, p)]) / np.outer(root[p], root[p]))
        h.set_profiling(True)
        h.factorize(vals, "fp64")
        h.set_profiling(False)
        assert (h.kernel_stats()["update_tc"]["launches"] > 0) == (region == -1)
        h.free()
    assert err[-1] <= 2 * err[general] + 4 * 2.0 ** -53, err
