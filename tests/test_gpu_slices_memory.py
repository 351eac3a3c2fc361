"""Memory of the FP64 slices' operand copies: only the rows that the tensor cores
read, at 14 bytes an element of the panel's width rounded up to 16, 32 or whole
64-column blocks.
"""
import numpy as np
import pytest
import torch

from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


CASES = {
    "grid_64": (lambda: inputs.diffusion_3d(30, 30, 30, 1), "llt", dict(ordering=1, grid=(30, 30, 30), max_width=64)),
    "graph_128": (lambda: inputs.diffusion_3d(28, 27, 26, 2), "llt", dict()),
    "ldlt": (lambda: inputs.quasi_definite_3d(20, 20, 20, 3), "ldlt",
             dict(ordering=1, grid=(20, 20, 20), dof=2, max_width=64)),
}


def _copy_bytes(h, method):
    P = h.panels()
    w, m = P["width"].astype(np.int64), (P["height"] - P["width"]).astype(np.int64)
    cols = np.where(w <= 16, 16, np.where(w <= 32, 32, (w + 63) // 64 * 64))
    return 14 * int(np.sum(m * cols)) * (2 if method == "ldlt" else 1)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("name", list(CASES))
def test_operand_copy_is_as_wide_as_its_panels(name):
    make, method, opts = CASES[name]
    cp, ri, vals = inputs.csc_arrays(make())
    h = spx.analyze(cp, ri, method, queue_panels=-1, **opts)
    h.factorize(vals, "fp32")              # everything that does not depend on the precision
    before = _free()
    h.factorize(vals, "fp64")
    used = before - _free()
    fac = h.info()["factor_bytes"]
    # the storage that FP64 takes more of (the factor, LDL^T's second copy, the diagonal blocks' inverses), an
    # eighth for columns of blocks that end unevenly, exponents and lists; allocations round up to 2 MiB
    assert used <= (1.2 if method == "ldlt" else 0.6) * fac + 1.125 * _copy_bytes(h, method) + (32 << 20), (used, fac)
    h.free()
