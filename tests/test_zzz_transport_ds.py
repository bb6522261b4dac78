"""Double-single contractions of T(E) and its adjoint against the oracle at the edges of their 32-wide tiles, one and
several energy groups, ragged row counts, and absorbers weak enough that the adjoint's M is far below 1.

Bounds: a double-single product is exact to 2^-47 of its magnitude and a chain of k additions to k 2^-48 of the sum of
the magnitudes (k at most 1,024 before the FP64 sums), so the sums' magnitudes times (2 * 1,100 + 3 n + nE + 16) 2^-48,
doubled for the complex parts; entries below 2^-90 of the largest may lose their tails to the range of a float."""
import numpy as np
import pytest

import workloads as W
from oracle import transport

pytestmark = pytest.mark.gpu

U48 = 2.0 ** -48
CHAIN = 1100


# pairs, energies, absorber scale
@pytest.mark.parametrize("n,nE,scale", [(1, 1, 1.0), (31, 3, 1.0), (32, 64, 1.0), (33, 70, 1.0), (65, 2, 1.0),
                                        (130, 9, 1.0), (33, 5, 1e-9)])
def test_transport_tiles(n, nE, scale):
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(7, 6, 63, 0.5, 3, 9)  # 2,646 rows: 22 past a tile; both absorbers vanish over part of them
    rng = np.random.default_rng(100 + n)
    U = (rng.standard_normal((w.N, n)) + 1j * rng.standard_normal((w.N, n))) / np.sqrt(2.0 * w.N)
    eps = np.sort(rng.uniform(-1.0, 0.5, n)) - 1j * rng.uniform(0.01, 0.2, n)
    E = np.linspace(-1.1, 0.6, nE)
    wts = rng.standard_normal(nE)
    wts[nE // 2] = 0.0 if nE > 1 else 1.0
    gL, gR = scale * w.gamma_L, scale * w.gamma_R
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(gL, gR)
        c.set_eigenpairs(eps, U)
        T = c.transmission(E)
        dV, dE = c.grad(E, wts)
    Ua = np.abs(U)
    Rt, Lt = (x.real for x in transport.projections(Ua, gL, gR))
    Wt = Rt * Lt
    S, Sd, Mt = [], [], np.zeros_like(Rt)
    for En, we in zip(E, wts):
        ga = np.abs(1.0 / (En - eps))
        S.append(ga @ Wt @ ga)
        Sd.append((ga * ga) @ Wt @ ga)
        Mt += abs(we) * (ga[:, None] * Rt * ga[None, :]) @ (Lt.T * ga[None, :])
    S, Sd = np.array(S), np.array(Sd)
    Qt = 2.0 * np.sum((Ua @ Mt) * Ua, axis=1)
    u = 2.0 * (2 * CHAIN + 3 * n + nE + 16) * U48
    tol = lambda q: u * q + 2.0 ** -90 * q.max()
    assert np.all(np.abs(T - transport.transmission_spectral(eps, U, gL, gR, E)) <= tol(S))
    assert np.all(np.abs(dE - wts * transport.grad_E_spectral(eps, U, gL, gR, E)) <= tol(2.0 * Sd * np.abs(wts).max()))
    assert np.all(np.abs(dV - transport.grad_V_spectral(eps, U, gL, gR, E, wts)) <= tol(Qt))
