"""FP64 factorizations whose TRSM and updates run on the tensor cores by
error-free slices (csrc/slices.cuh), against the oracle and against the
CUDA-core path of the task queue, at the edges of their tiles: panels of one
to 150 columns (several digit blocks), heights around 64 and 128 rows, graph
orderings, Cholesky and LDL^T.

The slices' own error is below a chain of FP64 multiply-adds (slices.cuh), so
the factor meets the bounds of the FP64 factor (1e-12 relative, Frobenius and
largest entry) and its error is at most twice the CUDA-core path's plus 4
units of rounding (the order of the reductions differs between two runs).
"""
import numpy as np
import pytest

import oracle
from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu
SLICES, QUEUE = -1, 1 << 30      # queue_panels: every level on its own / the whole tree in the queue


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


CASES = {
    "one_wide": (lambda: inputs.diffusion_3d(8, 8, 8, 1), "llt", dict(ordering=1, grid=(8, 8, 8), max_width=64)),
    "ragged_24": (lambda: inputs.diffusion_3d(13, 9, 11, 2), "llt", dict(ordering=1, grid=(13, 9, 11), max_width=24)),
    "width_17": (lambda: inputs.diffusion_3d(16, 15, 14, 3), "llt", dict(ordering=1, grid=(16, 15, 14), max_width=17)),
    "two_blocks": (lambda: inputs.diffusion_3d(16, 16, 16, 4), "llt", dict(ordering=1, grid=(16, 16, 16))),
    "three_blocks": (lambda: inputs.elasticity_27pt(7, 7, 7, 5), "llt",
                     dict(ordering=1, grid=(7, 7, 7), dof=3, max_width=150)),
    "graph": (lambda: inputs.random_spd_graph(900, 5, 6), "llt", dict()),
    "contrast": (lambda: inputs.diffusion_3d(14, 13, 12, 7, sigma=4.0), "llt",
                 dict(ordering=1, grid=(14, 13, 12), max_width=64)),
    "ldlt": (lambda: inputs.quasi_definite_3d(10, 9, 8, 8), "ldlt", dict(ordering=1, grid=(10, 9, 8), dof=2, max_width=64)),
    "ldlt_33": (lambda: inputs.quasi_definite_3d(9, 9, 9, 9), "ldlt", dict(ordering=1, grid=(9, 9, 9), dof=2, max_width=33)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_slices_match_oracle_and_general_path(name):
    make, method, opts = CASES[name]
    A = make()
    cp, ri, vals = inputs.csc_arrays(A)
    err, F = {}, None
    for region in (SLICES, QUEUE):
        h = spx.analyze(cp, ri, method, queue_panels=region, **opts)
        F = F or (oracle.cholesky if method == "llt" else oracle.ldlt)(A, h.perm())
        h.factorize(vals, "fp64")
        Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
        err[region] = _rel(Lx, F.Lx)
        assert err[region] <= 1e-12 and np.max(np.abs(Lx - F.Lx)) <= 1e-12 * np.max(np.abs(F.Lx))
        B = inputs.rhs(A.shape[0], 2, 1)
        X, _ = h.solve(B)
        assert oracle.backward_error(A, X, B) <= 1e-13
        if region == SLICES:
            h.set_profiling(True)
            h.factorize(vals, "fp64")
            h.set_profiling(False)
            assert h.kernel_stats()["update_tc"]["launches"] > 0
        h.free()
    assert err[SLICES] <= 2 * err[QUEUE] + 4 * 2.0 ** -53


@pytest.mark.parametrize("power", [-900, -400, 400, 900])
def test_slices_scale_with_powers_of_two(power):
    """Rows of extreme exponents: the factor of 2^power A is 2^(power / 2) L
    up to the order of the reductions."""
    g = (12, 11, 10)
    A = inputs.diffusion_3d(*g, 3)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=1, grid=g, max_width=64, queue_panels=SLICES)
    F = oracle.cholesky(A, h.perm())
    h.factorize(vals * 2.0 ** power, "fp64")
    Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li) * 2.0 ** (-power // 2)
    assert _rel(Lx, F.Lx) <= 1e-12
    h.free()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_values_fail_as_on_the_general_path(bad):
    g = (12, 11, 10)
    A = inputs.diffusion_3d(*g, 3)
    cp, ri, vals = inputs.csc_arrays(A)
    got = []
    for region in (SLICES, QUEUE):
        h = spx.analyze(cp, ri, "llt", ordering=1, grid=g, max_width=64, queue_panels=region)
        v = vals.copy()
        j = int(h.perm()[30])               # an off-diagonal entry of an early column
        e = [k for k in range(cp[j], cp[j + 1]) if ri[k] != j]
        for k in e:
            v[k] = bad
            i = ri[k]
            v[[q for q in range(cp[i], cp[i + 1]) if ri[q] == j][0]] = bad
        with pytest.raises(spx.SpxError) as ex:
            h.factorize(v, "fp64")
        got.append((ex.value.status, h.info()["bad_col"]))
        h.free()
    assert got[0] == got[1]
