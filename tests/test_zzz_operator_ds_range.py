"""Double-single operator on operands outside the range of its fast split: NaN and infinite entries and shifts reach
exactly the outputs that they reach in 64 bits, and values in the largest binade of a float keep their digits."""
import numpy as np
import pytest

import workloads as W
from oracle import stencil

pytestmark = pytest.mark.gpu


def _apply(w, h, bc, X, sig):
    import paper_1606_01139_gb300 as swi
    with swi.Context(w.nx, w.ny, w.nz, h, bc=bc) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        Y = c.apply_ds(X, sig)
    with np.errstate(all="ignore"):
        Yo = stencil.apply_A(X, w.nx, w.ny, w.nz, h, w.V, w.gamma_L, w.gamma_R, bc=bc) - X * sig[None, :]
    return Y, Yo


@pytest.mark.parametrize("h", [0.5, 2.0])
@pytest.mark.parametrize("bc", [0, 1])
def test_non_finite_operands(h, bc):
    w = W.make_wire(14, 13, 15, h, 3, 5)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((w.N, 6)) + 1j * rng.standard_normal((w.N, 6))
    at = (7 * 13 + 6) * 14 + 5
    X[at, 0] = complex(np.nan, 1.0)
    X[at, 1] = complex(1.0, -np.inf)
    X[2, 2] = complex(np.inf, np.nan)  # near a corner: its mirror points too
    X[at, 3] = 1e300                   # beyond the floats: an infinity
    sig = rng.uniform(-1.0, 1.0, 6)
    sig[4] = np.nan
    Y, Yo = _apply(w, h, bc, X, sig)
    Yo[:, 3] = np.where(np.abs(Yo[:, 3]) > 1e200, np.inf, Yo[:, 3])
    assert np.array_equal(np.isfinite(Y), np.isfinite(Yo))
    assert not np.isfinite(Y[:, 4]).any() and np.isfinite(Y[:, 5]).all()
    good = np.isfinite(Yo)
    # 37 products and sums of ~2^-47 each
    tol = 64 * 2.0 ** -46 * stencil.gershgorin_norm(h, w.V, w.gamma_L, w.gamma_R) * 6.0
    assert np.abs(np.where(good, Y - np.where(good, Yo, 0), 0)).max() <= tol


@pytest.mark.parametrize("value", [2.0 ** 127, -1.7 * 2.0 ** 127, 1.3 * 2.0 ** -74, 1.3 * 2.0 ** -100])
def test_edges_of_the_float_range(value):
    h = 2.0  # every weight below 1.2: no output beyond the floats
    w = W.make_wire(14, 13, 15, h, 3, 5)
    X = np.zeros((w.N, 2), complex)
    at = (7 * 13 + 11) * 14 + 12  # off the wells
    X[at, 0], X[at, 1] = value, 1j * value
    Y, Yo = _apply(w, h, 0, X, np.zeros(2))
    tail = 2.0 ** -140  # the floats' last denormals
    assert np.abs(Y - Yo).max() <= 64 * 2.0 ** -46 * abs(value) * 2.0 + tail
    assert np.abs(Yo).max() > 0.5 * abs(value)
