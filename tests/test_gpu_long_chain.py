"""Matrices whose panel tree is one long chain (a band in natural order): the
captured factorization's graph stays linear in the levels, so that the first
factorization costs little more than a repeated one.  A side stream that was
forked at every level without a launch made every node depend on all earlier
levels: half a million edges for 1,300 levels, 20 s to instantiate (633 levels:
2.3 s).
"""
import time

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


def _band(n, half, seed):
    g = np.random.default_rng(seed)
    L = sp.diags([np.full(n, 2.0 * half)] + [g.uniform(-1, 1, n - k) for k in range(1, half + 1)],
                 [-k for k in range(half + 1)], format="csc")
    return sp.csc_matrix(L + sp.tril(L, -1).T)


@pytest.mark.parametrize("half", [10, 64, 130])
@pytest.mark.parametrize("method,prec", [("llt", "fp64"), ("llt", "fp32"), ("llt", "tf32"), ("ldlt", "fp64"), ("ldlt", "bf16")])
def test_first_factorization_of_a_chain(method, prec, half):
    A = _band(1600, half, 1)
    cp, ri, vals = inputs.csc_arrays(A)
    warm = spx.analyze(*inputs.csc_arrays(_band(300, half, 2))[:2], method, ordering=spx.SPX_ORDER_NATURAL,
                       max_width=64, queue_panels=-1)
    warm.factorize(inputs.csc_arrays(_band(300, half, 2))[2], prec)      # kernels loaded
    warm.free()
    h = spx.analyze(cp, ri, method, ordering=spx.SPX_ORDER_NATURAL, max_width=64, queue_panels=-1)
    t = []
    for _ in range(3):
        t0 = time.perf_counter()
        h.factorize(vals, prec)
        t.append(time.perf_counter() - t0)
    assert t[0] <= 10 * t[1] + 0.3, t
    B = inputs.rhs(A.shape[0], 2, 1)
    X, _ = h.solve(B)
    assert oracle.backward_error(A, X, B) <= (1e-13 if prec == "fp64" else 1e-12)
    h.free()
