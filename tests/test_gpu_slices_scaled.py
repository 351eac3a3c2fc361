"""FP64 slices on symmetric systems whose unknowns have very different scales:
S A S with S diagonal, of powers of two, so that the exact factors are known to
the last bit from the unscaled system's (Cholesky: S L; LDL^T: S L S^-1 and
S D S), and multiply-adds in FP64 commit the same relative errors on both.  So
the scaled-back factor meets the bounds of the unscaled one: 1e-12 relative, and
at most twice the task queue's error (FP64 multiply-adds) plus 4 units of
rounding; the scaled-back solution has a backward error of at most 1e-13.
"""
import numpy as np
import pytest
import scipy.sparse as sp

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


def _scales(kind, n):
    """Exponents of the unknowns' scales: a random spread, or one of each node's two unknowns in another unit."""
    if isinstance(kind, int):
        return np.random.default_rng([kind, n]).integers(-kind, kind + 1, n)
    k, both = int(kind[1:]), np.zeros(n, np.int64)
    both[1::2] = -k
    return both


@pytest.mark.parametrize("kind", [7, 14, 20, "p20", "p30"])
@pytest.mark.parametrize("grid,width,method", [((10, 9, 8), 64, "ldlt"), ((9, 9, 9), 33, "ldlt"),
                                               ((13, 12, 11), 64, "llt"), ((12, 12, 12), 128, "llt")])
def test_scaled_unknowns(grid, width, method, kind):
    ldlt = method == "ldlt"
    A = inputs.quasi_definite_3d(*grid, 8) if ldlt else inputs.diffusion_3d(*grid, 8)
    n = A.shape[0]
    s = np.ldexp(1.0, _scales(kind, n))
    S = sp.diags(s)
    scaled = sp.csc_matrix(S @ A @ S)
    cp, ri, vals = inputs.csc_arrays(scaled)
    err, F = {}, None
    for region in (SLICES, QUEUE):
        if region == QUEUE and width > 64:
            continue
        h = spx.analyze(cp, ri, method, ordering=1, grid=grid, dof=2 if ldlt else 1, max_width=width,
                        queue_panels=region, pivot_tau=0.0)
        p = h.perm()
        F = F or (oracle.ldlt(A, p, tau=0.0) if ldlt else oracle.cholesky(A, p))
        h.factorize(vals, "fp64")
        Lx = h.factor_on_pattern(F.sym.Lp, F.sym.Li)
        sp_, col = s[p], np.repeat(np.arange(n), np.diff(F.sym.Lp))
        if ldlt:
            Lx = np.where(F.sym.Li == col, Lx / sp_[col] ** 2, Lx / sp_[F.sym.Li] * sp_[col])
        else:
            Lx = Lx / sp_[F.sym.Li]
        err[region] = np.linalg.norm(Lx - F.Lx) / np.linalg.norm(F.Lx)
        B = inputs.rhs(n, 2, 1)
        X, _ = h.solve(s[:, None] * B)
        be = oracle.backward_error(A, s[:, None] * X, B)
        h.free()
        assert err[region] <= 1e-12 and be <= 1e-13, (region, err[region], be)
    if QUEUE in err:
        assert err[SLICES] <= 2 * err[QUEUE] + 4 * 2.0 ** -53, err
