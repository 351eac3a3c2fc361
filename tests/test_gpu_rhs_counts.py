"""Solves with every number of right-hand sides that picks another form of the
sweeps (csrc/sweep.cu): FP64 by single columns in groups (up to 4), by blocks of
8 columns in 1 to 4 groups, with several passes a group (over 32); FP32 by 4
columns and by 16; panels of one to three 64-column blocks; Cholesky, LU, LDL^T.

FP64 solutions meet the FP64 backward error bound (1e-13); FP32 factors without
refinement are compared with the same factor's solutions column by column (sums
in another order: 1e-4), and refined to 1e-12.  A right-hand side that is not
finite leaves the others as they are.
"""
import numpy as np
import pytest

import oracle
from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


CASES = {
    "llt_64": (lambda: inputs.diffusion_3d(13, 12, 11, 1), "llt", dict(ordering=1, grid=(13, 12, 11), max_width=64)),
    "llt_128": (lambda: inputs.diffusion_3d(14, 14, 14, 2), "llt", dict(ordering=1, grid=(14, 14, 14))),
    "llt_150": (lambda: inputs.elasticity_27pt(6, 6, 7, 3), "llt", dict(ordering=1, grid=(6, 6, 7), dof=3, max_width=150)),
    "lu_64": (lambda: inputs.convection_diffusion_2d(40, 4)[0], "lu", dict(ordering=1, grid=(40, 40), max_width=64)),
    "lu_100": (lambda: inputs.random_spd_graph(500, 6, 5), "lu", dict(max_width=100)),
    "ldlt": (lambda: inputs.quasi_definite_3d(8, 7, 9, 6), "ldlt", dict(ordering=1, grid=(8, 7, 9), dof=2, max_width=64)),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_every_form_of_the_sweeps(name, prec):
    make, method, opts = CASES[name]
    A = make()
    n = A.shape[0]
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, method, **opts)
    h.factorize(vals, prec)
    B = inputs.rhs(n, 37, 7)
    plain = spx.default_refine(mode=0)
    one = np.stack([h.solve(np.ascontiguousarray(B[:, c]), refine=plain)[0] for c in range(B.shape[1])], 1)
    for nrhs in (1, 2, 4, 5, 8, 9, 16, 17, 37):
        Bn = np.asfortranarray(B[:, :nrhs])
        X, _ = h.solve(Bn, refine=plain)
        if prec == "fp64":
            assert oracle.backward_error(A, X, Bn) <= 1e-13
        else:
            assert np.max(np.linalg.norm(X - one[:, :nrhs], axis=0) / np.linalg.norm(one[:, :nrhs], axis=0)) <= 1e-4
            X, info = h.solve(Bn, refine=spx.default_refine(tol=1e-12))
            assert info["converged"] and oracle.backward_error(A, X, Bn) <= 1e-12
    h.free()


@pytest.mark.parametrize("nrhs", [3, 6, 20])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_a_column_that_is_not_finite_stays_alone(nrhs, prec):
    make, method, opts = CASES["llt_64"]
    A = make()
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, method, **opts)
    h.factorize(vals, prec)
    B = inputs.rhs(A.shape[0], nrhs, 3)
    plain = spx.default_refine(mode=0)
    X0, _ = h.solve(B, refine=plain)
    B[5, 1] = np.nan
    X1, _ = h.solve(B, refine=plain)
    keep = [c for c in range(nrhs) if c != 1]
    assert np.isnan(X1[:, 1]).all()
    bound = 1e-12 if prec == "fp64" else 1e-4
    assert np.linalg.norm(X1[:, keep] - X0[:, keep]) <= bound * np.linalg.norm(X0[:, keep])
    h.free()
