"""FP32 contractions on both sides of one 64-wide tile (a single tile contracts M itself, more take its symmetric part),
to the bounds of test_zzz_contraction_f32.py."""
import numpy as np
import pytest

import workloads as W
from test_zzz_contraction_f32 import _check, _ctx, swi  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 64, 65, 128])
def test_one_tile_and_more(swi, n):  # noqa: F811
    w = W.make_wire(7, 6, 63, 0.5, 3, 9)  # 2,646 rows: 22 past a block of 64
    rng = np.random.default_rng(n)
    U = (rng.standard_normal((w.N, n)) + 1j * rng.standard_normal((w.N, n))) / np.sqrt(2.0 * w.N)
    eps = np.sort(rng.uniform(-1.0, 0.5, n)) - 1j * rng.uniform(0.01, 0.2, n)
    E = np.linspace(-1.1, 0.6, 7)
    wts = rng.standard_normal(len(E))
    with _ctx(swi, w) as c:
        c.set_eigenpairs(eps, U)
        c.set_contraction(swi.CONTRACT_F32)
        T = c.transmission(E)
        dV, dE = c.grad(E, wts)
    _check(eps, U, w, E, wts, T, dV, dE)
