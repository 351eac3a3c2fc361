"""The batched kernel's forms for one to four CTAs an SM (different registers, the
same arithmetic): equal results up to the order of atomic sums, whichever one a
batch's size or spx_batch_set_config picks.  Small systems of two to five a side
(single-panel roots, few rows below a panel) beside larger ones.  Bounds: those of
a backward-stable solve (FP64 1e-13; FP32, unrefined, 1e-4).
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


def _batch(sides):
    mats = [inputs.convection_diffusion_2d(k, 100 + i)[0] for i, k in enumerate(sides)]
    arrs = [inputs.csc_arrays(A) for A in mats]
    b = spx.batch_analyze([(cp, ri) for cp, ri, _ in arrs], grids=[(k, k, 1) for k in sides],
                          ordering=spx.SPX_ORDER_GRID, max_width=64)
    return mats, b, np.concatenate([v for _, _, v in arrs]), \
        np.concatenate([inputs.rhs(A.shape[0], 1, 7).ravel() for A in mats])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("leaf", [0, 8, 16])
def test_every_occupancy_solves(prec, leaf):
    mats, b, vals, rhs = _batch([2, 3, 4, 5, 2, 3, 9, 17, 30, 2, 5])
    for ctas in (1, 2, 3, 4):
        b.set_config(ctas_per_sm=ctas, leaf_width=leaf)
        X, _ = b.run(vals, rhs, precision=prec)
        assert b.info()["ctas_per_sm"] == min(ctas, 2 if prec == "fp64" else 4)
        o = 0
        for A in mats:
            n = A.shape[0]
            assert oracle.backward_error(A, X[o:o + n], rhs[o:o + n]) <= (1e-13 if prec == "fp64" else 1e-4)
            o += n
    b.free()


@pytest.mark.parametrize("count", [1, 300, 304, 305, 456, 457, 700])
def test_default_occupancy_holds_the_batch(count):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mats, b, vals, rhs = _batch([2 + i % 3 for i in range(count)])
    X, _ = b.run(vals, rhs, precision="fp32", refine=spx.default_refine(tol=1e-12))
    assert b.info()["ctas_per_sm"] == min(4, max(2, -(-count // sms)))
    o = 0
    for A in mats:
        n = A.shape[0]
        assert oracle.backward_error(A, X[o:o + n], rhs[o:o + n]) <= 1e-12
        o += n
    b.free()
