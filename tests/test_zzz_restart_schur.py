"""The restart's projected Schur step (FP32 Schur form, kept subspace corrected to double-single accuracy) at the
orders where its kernels change: register and shared-memory limits of the reduction, the chase and the kept block."""
import numpy as np
import pytest

import workloads as W
from oracle import eigen, stencil

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wire():
    w = W.make_wire(9, 10, 20, 0.5, 5, 11)
    A = stencil.dense_A(w.nx, w.ny, w.nz, w.h, w.V, w.gamma_L, w.gamma_R)
    eps, _ = eigen.dense_spectrum(A)
    return w, eps


# basis, kept vectors, request, block, imaginary part of the shift
@pytest.mark.parametrize("m,keep,n_req,block,im", [
    (48, 18, 8, 2, 0.0),     # smallest order that takes this form
    (97, 40, 12, 1, 0.0),
    (160, 88, 24, 2, 0.0),   # last order of five register columns; kept block at its three-column limit
    (168, 98, 24, 2, -0.05),  # matrix beyond shared memory in the reduction
    (236, 150, 40, 2, 0.0),  # packed matrix beyond shared memory in the chase
    (258, 60, 30, 1, 0.0),   # sixteen register columns
    (430, 300, 60, 2, 0.0),  # kept block beyond 256
    (508, 40, 24, 2, 0.0),
])
def test_restart_step_orders(wire, m, keep, n_req, block, im):
    import paper_1606_01139_gb300 as swi
    w, eps = wire
    sigma = float(eps.real[20])
    near = eps[np.argsort(np.abs(eps - (sigma + 1j * im)), kind="stable")]
    with swi.Context(w.nx, w.ny, w.nz, w.h) as ctx:
        ctx.set_potential(w.V)
        ctx.set_absorber(w.gamma_L, w.gamma_R)
        if im:
            ctx.set_windows_complex(np.array([sigma + 1j * im]), [n_req])
        else:
            ctx.set_windows([sigma], [n_req])
        info = ctx.solve(block=block, rel_tol=1e-11, max_basis=m, keep=keep, max_matvecs=40000)
        got = ctx.eigenvalues()
        wi = ctx.window_info()[0]
    assert info["status"] == "SWI_OK", info
    assert wi["restarts"] >= 1 and wi["schur_retries"] == 0
    # every delivered pair is an eigenvalue (rel_tol x ||A||_G x an eigenvalue condition of ~100), and the wanted
    # ones are there
    dist = np.abs(got[:, None] - eps[None, :]).min(1)
    assert dist.max() < 1e-11 * info["anorm"] * 100
    miss = np.abs(near[:n_req - 2, None] - got[None, :]).min(1)
    assert miss.max() < 1e-11 * info["anorm"] * 100
