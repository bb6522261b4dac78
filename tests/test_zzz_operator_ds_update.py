"""The double-single operator follows a potential or absorbers that are set anew, between applications and before a
solve of each block width."""
import numpy as np
import pytest

import workloads as W
from oracle import eigen, stencil

pytestmark = pytest.mark.gpu


def test_operator_follows_new_v_and_gamma():
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(8, 9, 12, 0.5, 3, 5)
    rng = np.random.default_rng(2)
    X = rng.standard_normal((w.N, 3)) + 1j * rng.standard_normal((w.N, 3))
    sig = np.array([0.1, -0.4, 0.7])
    tol = 64 * 2.0 ** -46 * 6.0
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        for V, gl in ((w.V, w.gamma_L), (2.0 * w.V, w.gamma_L), (2.0 * w.V, 3.0 * w.gamma_L), (w.V, 3.0 * w.gamma_L)):
            c.set_potential(V)
            c.set_absorber(gl, w.gamma_R)
            Y = c.apply_ds(X, sig)
            Yo = stencil.apply_A(X, w.nx, w.ny, w.nz, w.h, V, gl, w.gamma_R) - X * sig[None, :]
            assert np.abs(Y - Yo).max() <= tol * stencil.gershgorin_norm(w.h, V, gl, w.gamma_R)


@pytest.mark.parametrize("block", [1, 2, 4])
def test_solve_follows_a_new_potential(block):
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(8, 9, 12, 0.5, 3, 5)
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        for V in (w.V, 1.5 * w.V):
            c.set_potential(V)
            c.set_windows([float(V.min())], [4])
            info = c.solve(block=block, rel_tol=1e-10, max_matvecs=20000)
            assert info["status"] == "SWI_OK", info
            eps, _ = eigen.dense_spectrum(stencil.dense_A(w.nx, w.ny, w.nz, w.h, V, w.gamma_L, w.gamma_R))
            got = c.eigenvalues()
            # residual tolerance x ||A||_G x a condition number below ~100
            assert np.abs(got[:, None] - eps[None, :]).min(1).max() <= 1e-10 * info["anorm"] * 100
