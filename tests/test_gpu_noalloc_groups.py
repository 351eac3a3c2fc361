"""spx_solve_noalloc's column groups (as many as spx_solve's where their counters
fit the 16 MiB buffer): counts around each kernel's group size, and the last ones
that leave room for the counters of four groups, three, two and one.  Against
spx_solve without refinement: 1e-12 relative, as the orders of the sums differ.
"""
import numpy as np
import pytest

from paper_1405_2636_gb300 import inputs, spx

pytestmark = pytest.mark.gpu
BUFFER = 16 << 20


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    import __graft_entry__

    __graft_entry__.build()
    assert _t.cuda.is_available()
    return _t


@pytest.fixture(scope="module")
def system(torch):
    g = (17, 16, 15)
    A = inputs.diffusion_3d(*g, 3)
    cp, ri, vals = inputs.csc_arrays(A)
    h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_GRID, grid=g, max_width=64)
    h.factorize(vals, "fp64")
    yield A.shape[0], h
    h.free()


def _noalloc(torch, h, B, X):
    st = spx.load().spx_solve_noalloc(h._h, B.shape[1], B.data_ptr(), h.n, X.data_ptr(), h.n,
                                      torch.cuda.current_stream().cuda_stream)
    assert st == spx.SPX_OK, spx.load().spx_last_error(h._h)


def _columns(torch, n, nrhs):
    B = torch.from_numpy(np.ascontiguousarray(inputs.rhs(n, nrhs, 3).reshape(n, nrhs).T)).cuda().t()
    return B, torch.full((nrhs, n), float("nan"), dtype=torch.float64, device="cuda").t()


@pytest.mark.parametrize("nrhs", [1, 3, 4, 5, 8, 9, 16, 17, 24, 25, 33, "full"])
def test_matches_solve(torch, system, nrhs):
    n, h = system
    counters = 16 * h.info()["npanels"]
    if nrhs == "full":
        nrhs = (BUFFER - counters - 12) // (32 * n)      # the most columns that one group's counters allow
    B, X = _columns(torch, n, nrhs)
    _noalloc(torch, h, B, X)
    torch.cuda.synchronize()
    assert h.info()["noalloc_timeout"] == 0
    ref = h.solve(B if nrhs > 1 else B[:, 0], refine=spx.default_refine(mode=0))[0].reshape(X.shape)
    assert float((X - ref).norm() / ref.norm()) <= 1e-12


@pytest.mark.parametrize("groups", [1, 2, 3])
def test_fewer_groups_where_counters_do_not_fit(torch, groups):
    """Sizes at which the counters of `groups` groups fit and of one more do not."""
    for side in range(60, 110):                          # plane grids: many panels beside few rows
        cp, ri, vals = inputs.csc_arrays(inputs.laplacian_2d(side, side + 1))
        n = side * (side + 1)
        h = spx.analyze(cp, ri, "llt", ordering=spx.SPX_ORDER_GRID, grid=(side, side + 1, 1), max_width=8)
        counters = 16 * h.info()["npanels"]
        fits = [k for k in range(33, BUFFER // (32 * n) + 1)
                if 32 * n * k + groups * counters + 12 <= BUFFER < 32 * n * k + (groups + 1) * counters + 12]
        if fits:
            break
        h.free()
    assert fits
    h.factorize(vals, "fp64")
    B, X = _columns(torch, n, fits[0])
    _noalloc(torch, h, B, X)
    torch.cuda.synchronize()
    assert h.info()["noalloc_timeout"] == 0
    ref = h.solve(B, refine=spx.default_refine(mode=0))[0]
    assert float((X - ref).norm() / ref.norm()) <= 1e-12
    h.free()


@pytest.mark.parametrize("nrhs", [4, 16])
def test_takes_no_longer_than_solve(torch, system, nrhs):
    """One group, whatever the columns, took 2.3 times (4 columns) and 1.5 times (16) as long as spx_solve."""
    n, h = system
    B, X = _columns(torch, n, nrhs)
    ms = {}
    for name, call in (("noalloc", lambda: _noalloc(torch, h, B, X)),
                       ("solve", lambda: h.solve(B, refine=spx.default_refine(mode=0)))):
        t = []
        for _ in range(30):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ms[name] = np.median(t[5:])
    assert ms["noalloc"] <= 1.25 * ms["solve"], ms
