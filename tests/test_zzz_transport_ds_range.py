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


def test_rounding_of_long_sums():
    """1,000 pairs on 216 rows, absorbers on one plane each (36 terms per projection): the double-single sums over the
    pairs set the error.  With a renormalisation every 8 terms a sum of k terms is off by ~0.3 sqrt(k) 2^-48 of their
    root sum of squares (2,000 real terms in M, ~1,000 in the quadratic form: 13 and 10; ~19 with the splits and the
    projections); without, by 0.08 k 2^-48 (160 and 80)."""
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(6, 6, 6, 0.5, 1, 1)
    n, rng = 1000, np.random.default_rng(5)
    U = (rng.standard_normal((w.N, n)) + 1j * rng.standard_normal((w.N, n))) / np.sqrt(2.0 * w.N)
    eps = np.sort(rng.uniform(-1.0, 0.5, n)) - 1j * rng.uniform(0.05, 0.2, n)
    E, wts = np.array([-0.7, -0.2, 0.3]), np.array([1.0, 0.7, 1.3])
    plane = np.arange(w.N) // 36
    gL, gR = 0.5 * (plane == 0), 0.5 * (plane == 5)
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(gL, gR)
        c.set_eigenpairs(eps, U)
        dV, _ = c.grad(E, wts)
    want = transport.grad_V_spectral(eps, U, gL, gR, E, wts)
    R, L = transport.projections(U, gL, gR)
    g2 = 1.0 / np.abs(E[:, None] - eps[None, :]) ** 2
    M2 = sum(we ** 2 * (ge[:, None] * np.abs(R) ** 2 * ge[None, :]) @ (np.abs(L.T) ** 2 * ge[None, :])
             for we, ge in zip(wts, g2))
    U2 = np.abs(U) ** 2
    rss = 2.0 * np.sqrt(np.sum((U2 @ M2) * U2, axis=1))
    assert np.sqrt(np.mean(((dV - want) / rss) ** 2)) <= 60 * 2.0 ** -48
