"""complex64 operator on both sides of the rule between its fitted-tile and its TMA-staged kernel: thin and odd grids,
one to four columns, one and several z chunks; ragged 32 x 8 tiles with a partial column group for the staged one."""
import numpy as np
import pytest

import workloads as W
from oracle import stencil

pytestmark = pytest.mark.gpu

C64_TOL = 64 * 2.0 ** -24  # 37 products and sums in FP32 relative to ||A||_G max|X|


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("shape,nvec", [
    ((6, 20, 7), 1), ((45, 37, 30), 2), ((17, 16, 91), 2),    # two columns per block
    ((9, 13, 6), 3), ((200, 6, 9), 4), ((33, 70, 11), 4),     # four, thin tiles
    ((70, 45, 49), 6), ((97, 41, 25), 10),                    # TMA-staged: ragged tiles and column groups
])
def test_apply_c64(shape, nvec, bc):
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(*shape, 0.5, 4, 3)
    rng = np.random.default_rng(17 + nvec)
    X = (rng.standard_normal((w.N, nvec)) + 1j * rng.standard_normal((w.N, nvec))).astype(np.complex64)
    sig = rng.uniform(-2.0, 1.0, nvec)
    with swi.Context(*shape, 0.5, bc=bc) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        Y = c.apply_c64(X, sig)
    Xd = X.astype(np.complex128)
    sig32 = sig.astype(np.float32).astype(np.float64)
    Yo = stencil.apply_A(Xd, w.nx, w.ny, w.nz, w.h, w.V, w.gamma_L, w.gamma_R, bc=bc) - Xd * sig32[None, :]
    an = stencil.gershgorin_norm(w.h, w.V, w.gamma_L, w.gamma_R)
    assert np.max(np.abs(Y - Yo)) <= C64_TOL * an * np.max(np.abs(X))
