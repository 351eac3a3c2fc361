"""Memory of the FP64 slices' operand copies: only the rows that the tensor cores
read, at 14 bytes an element of the panel's width rounded up to 16, 32 or whole
64-column blocks; given back when the handle needs the memory elsewhere or the
factor's precision changes, and not made where they would leave too little.
"""
import numpy as np
import pytest
import torch

import oracle
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


class _Filled:
    """Device memory taken up but for `left` bytes."""

    def __init__(self, left):
        self.blocks = []
        while True:
            room = _free() - left
            if room < (4 << 20):
                break
            self.blocks.append(torch.empty(room - (2 << 20), dtype=torch.uint8, device="cuda"))

    def release(self):
        self.blocks.clear()
        torch.cuda.empty_cache()


def _grid(queue_panels=-1):
    A = inputs.diffusion_3d(30, 30, 30, 1)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=1, grid=(30, 30, 30), max_width=64, queue_panels=queue_panels)
    return A, vals, h


def _sliced(h, vals):
    h.set_profiling(True)
    h.factorize(vals, "fp64")
    h.set_profiling(False)
    return h.kernel_stats()["update_tc"]["launches"] > 0


def _warm():
    """Every kernel of the calls below loaded (a first launch takes device memory)."""
    A, vals, h = _grid(1 << 30)
    h.factorize(vals, "fp32")
    h.factorize(vals, "fp64")
    h.selected_inverse()
    h.solve(inputs.rhs(A.shape[0], 40, 1))
    h.free()
    A, vals, h = _grid()
    h.factorize(vals, "fp64")
    h.selected_inverse()
    h.free()


def test_copies_are_given_back_when_memory_is_short():
    _warm()
    A, vals, h = _grid()
    h.factorize(vals, "fp64")
    fill = _Filled(48 << 20)                       # less than the selected inverse's first array
    try:
        h.selected_inverse()
        X, _ = h.solve(inputs.rhs(A.shape[0], 2, 1))
    finally:
        fill.release()
    assert oracle.backward_error(A, X, inputs.rhs(A.shape[0], 2, 1)) <= 1e-13
    assert _sliced(h, vals)                        # there is room again
    X, _ = h.solve(inputs.rhs(A.shape[0], 2, 1))
    assert oracle.backward_error(A, X, inputs.rhs(A.shape[0], 2, 1)) <= 1e-13
    h.free()


def test_copies_are_not_made_where_they_leave_too_little():
    _warm()
    A, vals, h = _grid()
    h.factorize(vals, "fp32")
    fac64 = 2 * h.info()["factor_bytes"]
    fill = _Filled(fac64 + _copy_bytes(h, "llt") + (96 << 20))   # the FP64 factor and the copies, no selected inverse
    try:
        h.factorize(vals, "fp64")
        h.selected_inverse()
        X, _ = h.solve(inputs.rhs(A.shape[0], 16, 1))
    finally:
        fill.release()
    assert oracle.backward_error(A, X, inputs.rhs(A.shape[0], 16, 1)) <= 1e-13
    assert _sliced(h, vals)
    before = _free()
    h.factorize(vals, "fp32")                      # the copies go with the FP64 factor
    assert _free() - before >= _copy_bytes(h, "llt")
    h.free()
