"""Selected inversion where levels on the tensor cores (at least 4e6 multiply-adds)
and levels on the FP64 unit follow one another, panels of one to several 64-row
blocks, ragged widths, against the oracle's selected inverse: 1e-12 relative
(Frobenius), the repository's bound for the FP64 path, and 1e-11 an entry in units
of sqrt(Z_ii Z_jj).
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


@pytest.mark.parametrize("grid,width", [((10, 10, 10), 64), ((17, 16, 15), 64), ((20, 19, 18), 64), ((20, 19, 18), 33),
                                        ((20, 20, 20), 16), ((22, 13, 12), 48), ((90, 80, 1), 64)])
def test_selected_inverse_across_the_line(grid, width):
    A = inputs.diffusion_3d(*grid, 5) if grid[2] > 1 else inputs.laplacian_2d(*grid[:2])
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=1, grid=grid, max_width=width)
    F = oracle.cholesky(A, h.perm())
    h.factorize(vals, "fp64")
    h.selected_inverse()
    Z = h.selected_inverse_on_pattern(F.sym.Lp, F.sym.Li)
    Zo = oracle.selected_inverse(F)
    assert np.linalg.norm(Z - Zo) <= 1e-12 * np.linalg.norm(Zo)
    d = np.sqrt(Zo[F.sym.Lp[:-1]])
    col = np.repeat(np.arange(len(d)), np.diff(F.sym.Lp))
    assert np.max(np.abs(Z - Zo) / (d[col] * d[F.sym.Li])) <= 1e-11
    h.free()
