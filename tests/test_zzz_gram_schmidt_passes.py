"""Gram-Schmidt passes of the windowed solves at the basis sizes where their kernels change: rows per tile, columns
per thread, one or two stages in shared memory; row counts that are no multiple of a tile, windows of unequal size."""
import numpy as np
import pytest

import workloads as W
from oracle import eigen, stencil

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wire():
    w = W.make_wire(9, 11, 19, 0.5, 5, 7)  # 1881 rows: 25 past a tile of 32, 9 past 16, 1 past 8
    A = stencil.dense_A(w.nx, w.ny, w.nz, w.h, w.V, w.gamma_L, w.gamma_R)
    eps, _ = eigen.dense_spectrum(A)
    return w, eps


# basis size, block, mixed precision
@pytest.mark.parametrize("m,block,mixed", [
    (30, 1, False), (32, 2, False),              # columns within one warp
    (64, 2, False), (66, 2, False), (65, 1, False),
    (128, 2, False), (130, 2, False), (129, 1, False),
    (256, 2, False), (258, 2, False), (257, 1, False),
    (510, 2, False), (520, 1, False),            # past 512: single vectors, one stage
    (64, 1, True), (130, 2, True), (258, 2, True), (510, 2, True), (520, 1, True),
])
def test_pass_widths(wire, m, block, mixed):
    import paper_1606_01139_gb300 as swi
    w, eps = wire
    sigma = [float(eps.real[6]), float(eps.real[30])]
    n_req = [4, 6]
    tol = 2e-6 if mixed else 1e-11
    kw = dict(precision=swi.PREC_MIXED) if mixed else {}
    with swi.Context(w.nx, w.ny, w.nz, w.h, **kw) as ctx:
        ctx.set_potential(w.V)
        ctx.set_absorber(w.gamma_L, w.gamma_R)
        ctx.set_windows(sigma, n_req)
        info = ctx.solve(block=block, rel_tol=tol, max_basis=m, max_matvecs=60000)
        got = ctx.eigenvalues()
    assert info["status"] in ("SWI_OK", "SWI_HOLES"), info
    # a pair's residual is at most tol ||A||_G; eigenvalue condition numbers stay below ~100
    dist = np.abs(got[:, None] - eps[None, :]).min(1)
    assert dist.max() < tol * info["anorm"] * 100
    for s, n in zip(sigma, n_req):
        near = eps[np.argsort(np.abs(eps - s), kind="stable")[:n - 2]]
        assert np.abs(near[:, None] - got[None, :]).min(1).max() < tol * info["anorm"] * 100
