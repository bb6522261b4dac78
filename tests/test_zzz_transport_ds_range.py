"""Adjoint of T(E) in double-single where its operands leave the range of a float: absorbers so weak that the products
of the projections would vanish, on one side or both; and sums past the 1,024 terms that stay in double-single.

Bounds as in test_zzz_transport_ds.py: a double-single product is exact to 2^-47 of its magnitude, a chain of k
additions to k 2^-48 of the sum of the magnitudes (k at most 1,100 before the FP64 sums)."""
import numpy as np
import pytest

import workloads as W
from oracle import transport

pytestmark = pytest.mark.gpu


def _adjoint(n, nE, sL, sR, shape):
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(*shape, 0.5, 3, 9)
    rng = np.random.default_rng(100 + n)
    U = (rng.standard_normal((w.N, n)) + 1j * rng.standard_normal((w.N, n))) / np.sqrt(2.0 * w.N)
    eps = np.sort(rng.uniform(-1.0, 0.5, n)) - 1j * rng.uniform(0.01, 0.2, n)
    E = np.linspace(-1.1, 0.6, nE)
    wts = rng.standard_normal(nE)
    gL, gR = sL * w.gamma_L, sR * w.gamma_R
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(gL, gR)
        c.set_eigenpairs(eps, U)
        dV, _ = c.grad(E, wts)
    Ua = np.abs(U)
    Rt, Lt = (x.real for x in transport.projections(Ua, gL, gR))
    Mt = np.zeros_like(Rt)
    for En, we in zip(E, wts):
        ga = np.abs(1.0 / (En - eps))
        Mt += abs(we) * (ga[:, None] * Rt * ga[None, :]) @ (Lt.T * ga[None, :])
    Qt = 2.0 * np.sum((Ua @ Mt) * Ua, axis=1)
    u = 2.0 * (2 * 1100 + 3 * n + nE + 16) * 2.0 ** -48
    return dV, transport.grad_V_spectral(eps, U, gL, gR, E, wts), u * Qt + 2.0 ** -90 * Qt.max()


# absorber scales left and right (the projections themselves are double-single: they hold their digits to ~1e-27)
@pytest.mark.parametrize("sL,sR", [(1e-20, 1e-20), (1e-25, 1e-25), (1e-25, 1.0), (1e-3, 1e-22)])
def test_weak_absorbers(sL, sR):
    dV, want, tol = _adjoint(37, 5, sL, sR, (7, 6, 63))
    assert np.abs(want).max() > 0
    assert np.all(np.abs(dV - want) <= tol)


# a tile of 32 pairs, then one pair, past the limit; 1,176 rows
@pytest.mark.parametrize("n,nE", [(1056, 1), (1025, 2)])
def test_long_sums(n, nE):
    dV, want, tol = _adjoint(n, nE, 1.0, 1.0, (6, 7, 28))
    assert np.all(np.abs(dV - want) <= tol)
