"""Selected inversion by error-free slices (csrc/update_sl.cu) at the edges of
its tiles: boxes whose panels have one to a few 64-row blocks below them, ragged
widths, strong contrast, against the oracle's selected inverse; the
log-determinant over fewer and more panels than its blocks and threads.
Tolerances are the repository's for the FP64 path (1e-12 relative, Frobenius);
with contrast exp(4 g) each entry against sqrt(Z_ii Z_jj), the scale that the
rounding of Z is relative to.
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


@pytest.mark.parametrize("grid,width,sigma", [((3, 3, 3), 64, 1.0), ((9, 8, 7), 17, 1.0), ((12, 11, 10), 64, 1.0),
                                              ((14, 13, 12), 48, 1.0), ((16, 15, 14), 64, 1.0), ((11, 12, 10), 64, 4.0)])
def test_selected_inverse_matches_oracle(grid, width, sigma):
    A = inputs.diffusion_3d(*grid, 5, sigma=sigma)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=1, grid=grid, max_width=width)
    F = oracle.cholesky(A, h.perm())
    h.factorize(vals, "fp64")
    h.selected_inverse()
    Z = h.selected_inverse_on_pattern(F.sym.Lp, F.sym.Li)
    Zo = oracle.selected_inverse(F)
    if sigma == 1.0:
        assert np.linalg.norm(Z - Zo) <= 1e-12 * np.linalg.norm(Zo)
    d = np.sqrt(Zo[F.sym.Lp[:-1]])
    col = np.repeat(np.arange(len(d)), np.diff(F.sym.Lp))
    assert np.max(np.abs(Z - Zo) / (d[col] * d[F.sym.Li])) <= 1e-11
    ld = h.logdet()
    want = 2.0 * np.sum(np.log(F.Lx[F.sym.Lp[:-1]]))
    assert abs(ld - want) <= 1e-12 * np.sum(np.abs(np.log(F.Lx[F.sym.Lp[:-1]])))
    h.free()
