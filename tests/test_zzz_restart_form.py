"""The form of the restart's Schur step that is tried first (FP32 Schur form, kept subspace corrected to double-single),
by itself against numpy, and in solves that count how often it gave up."""
import numpy as np
import pytest

import workloads as W
from oracle import eigen, stencil

pytestmark = pytest.mark.gpu


def _matrix(m, k, b, seed, bordered):
    """A projected matrix of A - sigma: values near zero and up to ~45, nearly normal; bordered: as after a restart (a
    triangle of order k, b coupling rows below it, a band to the right)."""
    rng = np.random.default_rng(seed)
    cplx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    near = rng.uniform(-0.5, 0.5, k) - 0.05j * rng.random(k)
    far = rng.uniform(1.0, 45.0, m - k) - 0.3j * rng.random(m - k)
    if not bordered:
        V = np.eye(m) + 0.1 * cplx(m, m) / np.sqrt(m)
        return V @ np.diag(np.concatenate([near, far])) @ np.linalg.inv(V)
    H = np.zeros((m, m), complex)
    H[:k, :k] = np.triu(cplx(k, k), 1) * (0.05 / np.sqrt(k)) + np.diag(near)
    H[:, k:] = np.triu(cplx(m, m - k), -(k + b)) * (0.1 / np.sqrt(m))
    H[k:k + b, :k] = 1e-3 * cplx(b, k)
    H[range(k, m), range(k, m)] += far
    return H


@pytest.fixture(scope="module")
def ctx():
    import paper_1606_01139_gb300 as swi
    w = W.make_wire(6, 6, 6, 0.5, 1, 1)
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        yield c


# orders and kept counts at the edges of the kernels' registers and shared memory, odd ones among them
@pytest.mark.parametrize("bordered", [False, True])
@pytest.mark.parametrize("m,keep,b,sig_im", [(48, 3, 1, 0.0), (49, 21, 2, 0.0), (97, 40, 1, 0.0), (128, 48, 16, 0.0),
                                             (160, 96, 2, 0.0), (161, 97, 5, -0.05), (237, 88, 2, 0.0),
                                             (256, 60, 1, 0.0), (257, 150, 2, 0.0), (430, 260, 2, 0.0),
                                             (512, 60, 2, -0.02)])
def test_kept_block(ctx, m, keep, b, sig_im, bordered):
    H = _matrix(m, keep, b, m + keep, bordered)
    T, Z, info = ctx.check_restart(H, np.zeros((b, m)), keep=keep, n_want=max(1, keep // 2), sig_im=sig_im)
    assert info[2] == 0, info
    k = int(info[0])
    assert keep <= k <= min(keep + 8, m - b)
    # double-single products: sums of up to 512 terms of 2^-47 each, a few of them
    tol = 1e-11 * np.linalg.norm(H)
    assert np.linalg.norm(H @ Z - Z @ T) <= tol
    assert np.abs(Z.conj().T @ Z - np.eye(k)).max() <= 1e-11
    assert np.all(np.tril(T, -1) == 0)
    if not bordered:  # well-conditioned values: the k nearest, one by one
        ev = np.linalg.eigvals(H)
        ev = ev[np.argsort(np.abs(ev - 1j * sig_im))[:k]]
        d = np.abs(np.diag(T)[:, None] - ev[None, :])
        assert max(d.min(0).max(), d.min(1).max()) <= 10 * tol


@pytest.fixture(scope="module")
def wire():
    w = W.make_wire(9, 10, 20, 0.5, 5, 11)
    eps, _ = eigen.dense_spectrum(stencil.dense_A(w.nx, w.ny, w.nz, w.h, w.V, w.gamma_L, w.gamma_R))
    return w, eps


# basis, kept vectors, request, block (3 and more: the wide-block solver)
@pytest.mark.parametrize("m,keep,n_req,block", [(48, 18, 8, 2), (97, 40, 12, 1), (160, 88, 24, 2), (236, 150, 40, 2),
                                                (48, 24, 8, 3), (85, 40, 12, 5), (256, 96, 16, 16)])
def test_solves_run_this_form(wire, m, keep, n_req, block):
    import paper_1606_01139_gb300 as swi
    w, eps = wire
    sigma = [float(eps.real[20]), float(eps.real[60])]
    wide = block > 2
    tol = 3e-11 if wide else 1e-11  # what the block solver's double-single products reach
    with swi.Context(w.nx, w.ny, w.nz, w.h) as c:
        c.set_potential(w.V)
        c.set_absorber(w.gamma_L, w.gamma_R)
        c.set_windows(sigma, [n_req, n_req])
        info = c.solve(block=block, rel_tol=tol, max_basis=m, keep=keep, max_matvecs=60000)
        got = c.eigenvalues()
        wi = c.window_info()
    # it may give up where the cut between kept and other values falls within FP32 rounding: seldom
    assert all(x["restarts"] >= 1 and x["schur_retries"] == 0 for x in wi), wi
    assert sum(x["schur_fallbacks"] for x in wi) <= sum(x["restarts"] for x in wi) // 8, wi
    # a pair's residual is at most tol ||A||_G (ten times that explicitly in the wide form); condition numbers below ~100
    bound = tol * info["anorm"] * 100
    assert np.abs(got[:, None] - eps[None, :]).min(1).max() < bound
    for s, x in zip(sigma, wi):
        if x["n_conv"] >= n_req:
            near = eps[np.argsort(np.abs(eps - s), kind="stable")[:n_req - 2]]
            assert np.abs(near[:, None] - got[None, :]).min(1).max() < bound


# 24 values wanted and kept of a matrix whose 24th and 25th distances differ by 4e-5 of ~1, with condition numbers up to
# thousands: FP32 rounding alone orders them wrongly on some of these seeds
@pytest.mark.parametrize("seed", range(24))
def test_cut_within_fp32_rounding(ctx, seed):
    m, keep = 120, 24
    rng = np.random.default_rng(seed)
    r = np.concatenate([np.linspace(0.02, 1.0, keep), [1.0 + 4e-5], np.linspace(1.5, 45.0, m - keep - 1)])
    s = np.where(rng.random(m) < 0.5, -1.0, 1.0)
    s[keep] = -s[keep - 1]
    th = s * r * np.exp(-0.05j * rng.random(m))
    T = np.triu(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)), 1) * 2.5 / np.sqrt(m)
    T[range(m), range(m)] = th[rng.permutation(m)]
    Q, _ = np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))
    Tk, _, info = ctx.check_restart(Q @ T @ Q.conj().T, np.zeros((1, m)), keep=keep, n_want=keep)
    if info[2] == 0:  # else it gave up, and the full-order step decides
        assert info[1] == keep
        d = np.abs(np.diag(Tk)[:, None] - th[None, :keep])
        assert d.min(0).max() <= 1e-6  # every one of the keep nearest is there


# the grid spacing sets the size of H (~1/h^2): the result scales with it
@pytest.mark.parametrize("e", [-60, -30, 30, 60])
@pytest.mark.parametrize("m,keep", [(97, 40), (257, 150)])
def test_scale_of_the_matrix(ctx, m, keep, e):
    H = _matrix(m, keep, 2, 7, False)
    f = 2.0 ** e
    T, Z, info = ctx.check_restart(H * f, np.zeros((2, m)), keep=keep)
    assert info[2] == 0, info
    k = int(info[0])
    tol = 1e-11 * np.linalg.norm(H)
    assert np.linalg.norm(H @ Z - Z @ (T / f)) <= tol
    assert np.abs(Z.conj().T @ Z - np.eye(k)).max() <= 1e-11
    ev = np.linalg.eigvals(H)
    ev = ev[np.argsort(np.abs(ev))[:k]]
    d = np.abs(np.diag(T)[:, None] / f - ev[None, :])
    assert max(d.min(0).max(), d.min(1).max()) <= 10 * tol
