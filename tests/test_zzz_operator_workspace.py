"""The double-single operator's padded copy is not held by a context after a solve."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [2, 4])
def test_solve_gives_the_padded_copy_back(block):
    import torch
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(64, 62, 100, 0.5, 8, 3)
    pad = 16 * block * (64 + 12) * (62 + 12) * (100 + 12)
    X = torch.randn(w.N, block, dtype=torch.complex128, device="cuda")
    room = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")  # for the results, in torch's own pool
    del room
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        c.set_windows([float(w.V.min())], [4])
        c.solve(block=block, rel_tol=1e-3, max_basis=40, max_matvecs=80)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        c.apply_ds(X, np.zeros(block))  # needs the copy, of the same size
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
    assert before - after >= 0.9 * pad
