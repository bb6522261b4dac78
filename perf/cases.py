"""Timed cases of the partitioned eigensolver: what a user's program calls, at the sizes it calls it with.

Five kinds of work, each through the package's public entry points:

* ``operator``: the shifted operator (A - sigma_c) X on a block of vectors that is already on the GPU, in
  double-single, native FP64 or complex64 arithmetic;
* ``solve``: windows from a known spectrum, the windowed solve, then T(E) and its gradient (``double``), or the
  reduced-precision windows alone (``mixed``);
* ``pairs``: eigenpairs restored from a previous run, T(E) over an energy grid and its gradient with respect to
  V(r), with FP64-class or FP32 contractions;
* ``refine``: restored pairs of FP32-class accuracy, taken through the FP64 residual-correction sweeps;
* ``batch``: several independent wires of uneven grids solved in one call.

The wires follow ``workloads/``: h = 0.5 bohr, wells of depth 1-3 Ha along z, planar Gaussian absorbers at both ends.
``operator`` uses wells on the wire axis.  The other kinds use potentials that depend on z alone (the
``separable_wire`` of ``workloads/``), whose eigenpairs are products of one-dimensional ones, so that the windows can
be placed, pairs supplied and the results checked at any size.
"""
import math

import numpy as np
import torch

import paper_1606_01139_gb300 as swi

H = 0.5              # grid spacing (bohr)
ABS_HEIGHT = 0.5     # absorbers: height (Ha) and standard deviation (bohr)
ABS_SIGMA = 2.0
FD = (-5369 / 1800, 12 / 7, -15 / 56, 10 / 189, -1 / 112, 2 / 1925, -1 / 16632)  # 12th-order second difference


def listed():
    return [
        # the smallest operator call: a probe of one small wire, two vectors
        dict(name="operator_ds_10x10x20", kind="operator", arith="ds", nx=10, ny=10, nz=20, nvec=2, bc=0),
        # one step of the 8-window solve of the 48x48x96 wire: 8 windows of 2 vectors
        dict(name="operator_ds_48x48x96", kind="operator", arith="ds", nx=48, ny=48, nz=96, nvec=16, bc=0),
        # the reduced-precision operator on the 96x96x192 wire, 16 vectors
        dict(name="operator_c64_96x96x192", kind="operator", arith="c64", nx=96, ny=96, nz=192, nvec=16, bc=0),
        # a ragged grid with an odd number of complex64 vectors and zero ghosts
        dict(name="operator_c64_odd", kind="operator", arith="c64", nx=45, ny=37, nz=91, nvec=7, bc=1),
        # the small wire: 48 pairs in 4 windows, T(E) at 32 energies
        dict(name="solve_10x10x20", kind="solve", precision="double", nx=10, ny=10, nz=20, n_wells=6, n_r=48, p=4,
             n_E=32),
        # a wire of the uneven batch on its own: odd axes, two windows
        dict(name="solve_23x19x62", kind="solve", precision="double", nx=23, ny=19, nz=62, n_wells=12, n_r=40, p=2,
             n_E=64),
        # the lowest pairs of the 48x48x96 wire: one window of long vectors
        dict(name="solve_48x48x96", kind="solve", precision="double", nx=48, ny=48, nz=96, n_wells=24, n_r=14, p=1,
             n_E=128),
        # the same wire with a reduced-precision window
        dict(name="solve_mixed_48x48x96", kind="solve", precision="mixed", nx=48, ny=48, nz=96, n_wells=24, n_r=20,
             p=1, n_E=0),
        # T(E) and its gradient from the 400 stored pairs of the 48x48x96 wire, 128 energies
        dict(name="pairs_f64_48x48x96", kind="pairs", contraction="f64", nx=48, ny=48, nz=96, n_wells=24, n=400,
             n_E=128),
        # the differentiation form: 1000 pairs of the 64x64x128 wire, 256 energies, FP32 contractions
        dict(name="pairs_f32_64x64x128", kind="pairs", contraction="f32", nx=64, ny=64, nz=128, n_wells=40, n=1000,
             n_E=256),
        # FP32-class pairs of a middle-sized wire sharpened by two correction sweeps
        dict(name="refine_24x22x48", kind="refine", nx=24, ny=22, nz=48, n_wells=12, n=48, n_E=32),
        # four uneven wires solved in one call
        dict(name="batch_uneven", kind="batch", systems=4, lo=16, hi=24, n_r=20, p=2, n_E=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _wells(rng, nz):
    return max(2, round(nz * H / rng.uniform(2.0, 5.0)))  # one well every 2 to 5 bohr


def draw(rng):
    kind = rng.choice(["operator", "operator", "operator", "solve", "solve", "pairs", "pairs", "refine", "batch"])
    if kind == "operator":
        arith = rng.choice(["ds", "c64", "f64"])
        while True:
            nx, ny, nz = _log_int(rng, 6, 96), _log_int(rng, 6, 96), _log_int(rng, 8, 192)
            nvec = _log_int(rng, 1, 40)
            if nx * ny * nz * nvec <= 96 * 96 * 192 * (16 if arith == "c64" else 4):
                return dict(kind=kind, arith=arith, nx=nx, ny=ny, nz=nz, nvec=nvec, bc=rng.choice([0, 0, 1]))
    if kind == "solve":
        nx, ny, nz = _log_int(rng, 10, 32), _log_int(rng, 10, 32), _log_int(rng, 20, 72)
        return dict(kind=kind, precision=rng.choice(["double", "double", "mixed"]), nx=nx, ny=ny + (ny == nx), nz=nz,
                    n_wells=_wells(rng, nz), n_r=rng.randint(8, 32), p=rng.randint(1, 2), n_E=rng.randint(8, 64))
    if kind == "pairs":
        n = _log_int(rng, 24, 500)
        nx, ny, nz = _log_int(rng, 12, 64), _log_int(rng, 12, 64), _log_int(rng, 24, 128)
        return dict(kind=kind, contraction=rng.choice(["f64", "f32"]), nx=nx, ny=ny, nz=nz, n_wells=_wells(rng, nz),
                    n=min(n, 400 if nx * ny * nz > 250000 else n), n_E=rng.randint(8, 160))
    if kind == "refine":
        nx, ny, nz = rng.randint(12, 28), rng.randint(12, 28), rng.randint(24, 64)
        return dict(kind=kind, nx=nx, ny=ny + (ny == nx), nz=nz, n_wells=_wells(rng, nz), n=rng.randint(16, 64),
                    n_E=rng.randint(8, 48))
    lo = rng.randint(12, 16)
    return dict(kind=kind, systems=rng.randint(2, 5), lo=lo, hi=lo + rng.randint(2, 8), n_r=rng.randint(8, 24),
                p=rng.randint(1, 2), n_E=rng.randint(4, 24))


# ---------------------------------------------------------------- wires
def _absorbers_z(nz):
    z = np.arange(nz) * H
    return (ABS_HEIGHT * np.exp(-z ** 2 / (2 * ABS_SIGMA ** 2)),
            ABS_HEIGHT * np.exp(-(z - z[-1]) ** 2 / (2 * ABS_SIGMA ** 2)))


def _wells_z(nz, n_wells, rng):
    """A chain of wells along z, evenly spaced but for a few per cent, as in an atomic wire."""
    z = np.arange(nz) * H
    step = nz * H / n_wells
    zw = (np.arange(n_wells) + 0.5 + rng.uniform(-0.03, 0.03, size=n_wells)) * step
    dw = rng.uniform(0.95, 1.05, size=n_wells)
    return -(dw[:, None] * np.exp(-(z[None, :] - zw[:, None]) ** 2 / 2.0)).sum(0)


def _over_grid(f, nx, ny):
    """A function of z on the grid (x fastest)."""
    return np.repeat(f, nx * ny)


def _context(nx, ny, nz, V, bc=0, mixed=False):
    gl, gr = _absorbers_z(nz)
    ctx = swi.Context(nx, ny, nz, H, bc=swi.BC_ZERO if bc else swi.BC_ODD,
                      precision=swi.PREC_MIXED if mixed else swi.PREC_F64)
    ctx.set_potential(V)
    ctx.set_absorber(_over_grid(gl, nx, ny), _over_grid(gr, nx, ny))
    return ctx


def _kinetic_1d(n):
    """-1/2 d^2/dx^2 on n points with odd-reflection ghosts, dense."""
    T = np.zeros((n, n))
    for i in range(n):
        for k in range(-6, 7):
            j, s = i + k, 1.0
            if j == -1 or j == n:
                continue
            if j < 0:
                j, s = -2 - j, -1.0
            elif j > n:
                j, s = 2 * n - j, -1.0
            T[i, j] -= s * FD[abs(k)] / (2 * H * H)
    return T


def _modes_1d(n):
    """Eigenvalues and orthonormal (sine) modes of _kinetic_1d(n)."""
    i = np.arange(1, n + 1)
    X = math.sqrt(2.0 / (n + 1)) * np.sin(math.pi * np.outer(i, i) / (n + 1))
    th = math.pi * i / (n + 1)
    lam = FD[0] + 2 * sum(FD[k] * np.cos(k * th) for k in range(1, 7))
    return -lam / (2 * H * H), X


def _wire(nx, ny, nz, n_wells, n, seed):
    """A wire with V(z): potential, and its spectrum sorted by real part with the 1D mode numbers of every pair.  Of
    up to eight draws of the wells the first with an open gap above the n lowest pairs, or the one with the widest:
    which pairs are the n lowest must not hang on rounding."""
    ex, X = _modes_1d(nx)
    ey, Y = _modes_1d(ny)
    gl, gr = _absorbers_z(nz)
    best = None
    for k in range(8):
        vz = _wells_z(nz, n_wells, np.random.default_rng([seed, k]))
        ez, Z = np.linalg.eig(_kinetic_1d(nz) + np.diag(vz - 1j * (gl + gr)))
        eps = (ez[:, None, None] + ey[None, :, None] + ex[None, None, :]).reshape(-1)
        order = np.argsort(eps.real, kind="stable")
        re = eps.real[order[[0, n - 1, n]]]
        open_gap = (re[2] - re[1]) * n / (re[2] - re[0])  # in units of the mean spacing
        if best is None or open_gap > best[0]:
            best = (open_gap, vz, Z, eps, order)
        if open_gap > 0.1:
            break
    _, vz, Z, eps, order = best
    Z = Z / np.sqrt((Z * Z).sum(0))  # z^T z = 1
    kz, ky, kx = np.unravel_index(order, (nz, ny, nx))
    return dict(nx=nx, ny=ny, nz=nz, V=_over_grid(vz, nx, ny), eps=eps[order], kx=kx, ky=ky, kz=kz, X=X, Y=Y, Z=Z,
                gl=gl, gr=gr)


def _windows(eps, n, p):
    """p windows of equal counts for the lowest n pairs: shift mid-run, requests that reach the whole run (by
    |eps - sigma|, as the windows select) and two pairs more."""
    sig, req = [], []
    edges = np.linspace(0, n, p + 1).astype(int)
    for a, b in zip(edges[:-1], edges[1:]):
        s = 0.5 * (eps.real[a] + eps.real[b - 1])
        d = np.abs(eps - s)
        sig.append(s)
        req.append(int((d <= d[a:b].max() * (1 + 1e-9)).sum()) + 2)
    return np.array(sig), np.array(req, dtype=np.int32)


def _pairs(w, n, device):
    """The n lowest eigenpairs, u^T u = 1, as torch tensors (eps [n], U [N, n])."""
    t = lambda a: torch.as_tensor(a, device=device)  # noqa: E731
    X, Y = t(w["X"][:, w["kx"][:n]]), t(w["Y"][:, w["ky"][:n]])
    Z = t(w["Z"][:, w["kz"][:n]])
    XY = (Y[:, None, :] * X[None, :, :]).reshape(-1, n)
    U = torch.empty(w["nz"], w["nx"] * w["ny"], n, dtype=torch.complex128, device=device)
    for k in range(w["nz"]):
        U[k] = XY * Z[k]
    return t(np.ascontiguousarray(w["eps"][:n])), U.reshape(-1, n)


def _energies(eps, n, n_E):
    """n_E energies between the levels: spread evenly over the middle thirds of the gaps that are no narrower than
    the mean one (on a level of a weakly absorbed state T(E) is a resonance without a width)."""
    re = eps.real[:n + 1]
    gap = np.diff(re)
    gap = np.where(gap * len(gap) >= re[-1] - re[0], gap, 0.0)
    ends = np.cumsum(gap)
    at = (np.arange(n_E) + 0.5) / n_E * ends[-1]
    k = np.minimum(np.searchsorted(ends, at, side="right"), len(gap) - 1)
    return re[k] + gap[k] / 3 + (at - (ends[k] - gap[k])) / 3


def _weights(n_E, seed):
    return np.random.default_rng(seed + 7).uniform(0.5, 1.5, n_E)


# ---------------------------------------------------------------- the cases
def _sub_systems(case, seed):
    rng = np.random.default_rng(1000 + case["systems"])  # the grids belong to the case, the wells to the seed
    out = []
    for s in range(case["systems"]):
        nx = int(rng.integers(case["lo"], case["hi"] + 1))
        ny = int(rng.integers(case["lo"], case["hi"] + 1))
        nz = 2 * int(rng.integers(case["lo"], case["hi"] + 1))
        out.append(_wire(nx, ny + (nx == ny), nz, max(2, round(nz * H / 3.0)), case["n_r"],
                         seed * 64 + s))
    return out


def _count(case):
    """Pairs of a solve, pairs or refine case."""
    return case["n_r"] if case["kind"] == "solve" else case["n"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "operator":
        nx, ny, nz, nvec = case["nx"], case["ny"], case["nz"], case["nvec"]
        x, y = (np.arange(nx) - (nx - 1) / 2) * H, (np.arange(ny) - (ny - 1) / 2) * H
        perp = np.exp(-(x[None, :] ** 2 + y[:, None] ** 2) / 2).reshape(-1)
        vz = _wells_z(nz, 12, np.random.default_rng(seed))
        V = (vz[:, None] * perp[None, :]).reshape(-1)
        ctx = _context(nx, ny, nz, V, bc=case["bc"], mixed=case["arith"] == "c64")
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.complex64 if case["arith"] == "c64" else torch.complex128
        X = torch.randn(nx * ny * nz, nvec, dtype=dt, device="cuda", generator=g)
        sigma = np.random.default_rng(seed + 1).uniform(-2.0, 0.6, nvec)
        return dict(kind=kind, arith=case["arith"], ctx=ctx, X=X, sigma=sigma, V=V)
    if kind == "batch":
        systems = []
        for w in _sub_systems(case, seed):
            n = case["n_r"]
            systems.append(dict(ctx=_context(w["nx"], w["ny"], w["nz"], w["V"]), win=_windows(w["eps"], n, case["p"]),
                                E=_energies(w["eps"], n, case["n_E"])))
        return dict(kind=kind, systems=systems, n_keep=case["n_r"])
    n = _count(case)
    w = _wire(case["nx"], case["ny"], case["nz"], case["n_wells"], n, seed)
    mixed = kind == "solve" and case["precision"] == "mixed"
    st = dict(kind=kind, ctx=_context(w["nx"], w["ny"], w["nz"], w["V"], mixed=mixed))
    if kind == "solve":
        st.update(mixed=mixed, n=n, win=_windows(w["eps"], n, case["p"]))
    else:
        st["eps"], st["U"] = _pairs(w, n, "cuda")
        if kind == "refine":
            g = torch.Generator(device="cuda").manual_seed(seed)
            st["U"] += 1e-6 / math.sqrt(w["V"].size) * torch.randn(st["U"].shape, dtype=torch.complex128,
                                                                  device="cuda", generator=g)
        elif case["contraction"] == "f32":
            st["ctx"].set_contraction(swi.CONTRACT_F32)
        st["f32"] = kind == "pairs" and case["contraction"] == "f32"
    if case["n_E"]:
        st.update(E=_energies(w["eps"], n, case["n_E"]), weights=_weights(case["n_E"], seed))
    return st


def _transport(st):
    ctx = st["ctx"]
    T = ctx.transmission(st["E"])
    dV = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
    dV, dE = ctx.grad(st["E"], st["weights"], dLdV_out=dV)
    return T, dV, dE


def run(state):
    kind = state["kind"]
    if kind == "operator":
        ctx = state["ctx"]
        f = {"ds": ctx.apply_ds, "f64": ctx.apply, "c64": ctx.apply_c64}[state["arith"]]
        return f(state["X"], state["sigma"])
    if kind == "batch":
        for s in state["systems"]:
            s["ctx"].set_windows(*s["win"])
        swi.solve_batch([s["ctx"] for s in state["systems"]], block=2, rel_tol=1e-12, n_keep=state["n_keep"],
                        max_matvecs=20000)
        return [dict(eps=s["ctx"].eigenvalues(), T=s["ctx"].transmission(s["E"])) for s in state["systems"]]
    ctx = state["ctx"]
    if kind == "solve":
        ctx.set_windows(*state["win"])
        if state["mixed"]:
            # single-precision pairs: their eigenvalues are passed on as such
            ctx.solve(block=2, rel_tol=2e-6, n_keep=state["n"], max_matvecs=4000)
            return dict(eps=ctx.eigenvalues().astype(np.complex64))
        ctx.solve(block=2, rel_tol=1e-12, n_keep=state["n"], max_matvecs=20000)
        T, dV, dE = _transport(state)
        return dict(eps=ctx.eigenvalues(), T=T, dV=dV, dE=dE)
    ctx.set_eigenpairs(state["eps"], state["U"])
    if kind == "refine":
        ctx.refine(max_sweeps=2)
    T, dV, dE = _transport(state)
    if kind == "refine":
        return dict(eps=ctx.eigenvalues(), T=T, dV=dV, dE=dE)
    if state["f32"]:  # single-precision contractions: the results are passed on in single precision
        return dict(T=T.astype(np.float32), dV=dV.float(), dE=dE.astype(np.float32))
    return dict(T=T, dV=dV, dE=dE)


# ---------------------------------------------------------------- the same results in 64 bits
def _axis(X, dim, zero):
    """-1/2 second difference along one grid axis of X [nz, ny, nx, nvec]."""
    n = X.shape[dim]
    i = torch.arange(-6, n + 6, device=X.device)
    s = torch.where((i < 0) | (i >= n), -1.0, 1.0).to(torch.float64)
    src = torch.where(i < 0, -2 - i, torch.where(i > n, 2 * n - i, i))
    dead = (i == -1) | (i == n) | (src < 0) | (src >= n)
    if zero:
        dead |= (i < 0) | (i >= n)
    s = torch.where(dead, 0.0, s)
    src = src.clamp(0, n - 1)
    shape = [1] * 4
    shape[dim] = n + 12
    P = X.index_select(dim, src) * s.view(shape)
    out = FD[0] * P.narrow(dim, 6, n)
    for k in range(1, 7):
        out = out + FD[k] * (P.narrow(dim, 6 - k, n) + P.narrow(dim, 6 + k, n))
    return out * (-1 / (2 * H * H))


def _exact_transport(w, n, E, wts, device):
    """T, dL/dV and dL/dE from the exact pairs: the projections of a z-only absorber couple pairs of equal x and y
    modes."""
    eps = w["eps"][:n]
    Z = w["Z"][:, w["kz"][:n]]
    same = (w["kx"][:n, None] == w["kx"][None, :n]) & (w["ky"][:n, None] == w["ky"][None, :n])
    R = (Z.T @ (w["gr"][:, None] * Z.conj())) * same
    L = (Z.T @ (w["gl"][:, None] * Z.conj())) * same
    W = R * L
    g = 1.0 / (np.asarray(E)[:, None] - eps[None, :])
    T = np.einsum("ek,ek->e", g @ W, g.conj()).real
    if wts is None:
        return T, None, None
    dE = -2 * np.einsum("ek,ek->e", (g * g) @ W, g.conj()).real * wts
    t = lambda a: torch.as_tensor(a, device=device)  # noqa: E731
    M = torch.zeros(n, n, dtype=torch.complex128, device=device)
    tR, tL, tg = t(R), t(L), t(g)
    # M_ac = sum_l R_al L_cl sum_e w_e g_ea g_ec conj(g_el): nonzero only where a, l and c share x and y modes
    for key in np.unique(w["kx"][:n] * 100000 + w["ky"][:n]):
        ix = t(np.nonzero(w["kx"][:n] * 100000 + w["ky"][:n] == key)[0])
        gi, Ri, Li = tg[:, ix], tR[ix][:, ix], tL[ix][:, ix]
        for e in range(len(E)):
            d = gi[e]
            M[ix[:, None], ix[None, :]] += wts[e] * (d[:, None] * ((Ri * d.conj()[None, :]) @ Li.T) * d[None, :])
    _, U = _pairs(w, n, device)
    dV = torch.empty(U.shape[0], dtype=torch.float64, device=device)
    for r in range(0, U.shape[0], 65536):
        u = U[r:r + 65536]
        dV[r:r + 65536] = 2 * ((u @ M) * u).sum(1).real
    return T, dV, dE


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "operator":
        st = prepare(case, seed)
        nx, ny, nz, nvec = case["nx"], case["ny"], case["nz"], case["nvec"]
        gl, gr = _absorbers_z(nz)
        V = torch.as_tensor(st["V"], device=dev).view(nz, ny, nx, 1)
        G = torch.as_tensor(gl + gr, device=dev).view(nz, 1, 1, 1)
        out = torch.empty(nx * ny * nz, nvec, dtype=torch.complex128, device=dev)
        for c in range(nvec):
            X = st["X"][:, c].to(torch.complex128).view(nz, ny, nx, 1)
            Y = sum(_axis(X, d, bool(case["bc"])) for d in range(3))
            out[:, c] = (Y + (V - float(st["sigma"][c]) - 1j * G) * X).reshape(-1)
        return out
    if kind == "batch":
        n = case["n_r"]
        return [dict(eps=w["eps"][:n], T=_exact_transport(w, n, _energies(w["eps"], n, case["n_E"]), None, dev)[0])
                for w in _sub_systems(case, seed)]
    n = _count(case)
    w = _wire(case["nx"], case["ny"], case["nz"], case["n_wells"], n, seed)
    if kind == "solve" and case["precision"] == "mixed":
        return dict(eps=w["eps"][:n])
    T, dV, dE = _exact_transport(w, n, _energies(w["eps"], n, case["n_E"]), _weights(case["n_E"], seed), dev)
    out = dict(T=T, dV=dV, dE=dE)
    if kind != "pairs":
        out["eps"] = w["eps"][:n]
    return out


# ---------------------------------------------------------------- the work of one pass
STENCIL_FLOPS = 116  # per point and vector: 18 neighbour pairs, the diagonal and the absorber


def _work_transport(N, n, n_E):
    flops = 2 * 8.0 * N * n * n + 8.0 * n_E * n * n * (n + 1) + 8.0 * N * n * n
    return 16.0 * N * n + 16.0 * N + 8.0 * N, flops


def _work_solve(N, n_r, p, item):
    # at least one basis of 2 n + 1 vectors per window: applications, Gram-Schmidt, rotation to the pairs
    k = max(1, n_r // p)
    m = 2 * k + 1
    return p * item * N * (m + k), p * N * (STENCIL_FLOPS * m + 8.0 * m * m + 8.0 * m * k)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for w in _sub_systems(case, 0):
            x, y = _work_solve(w["V"].size, case["n_r"], case["p"], 16.0)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    N = case["nx"] * case["ny"] * case["nz"]
    if kind == "operator":
        item = 8.0 if case["arith"] == "c64" else 16.0
        return {"bytes": N * (2 * item * case["nvec"] + item), "flops": float(STENCIL_FLOPS) * N * case["nvec"]}
    if kind == "solve":
        b, f = _work_solve(N, case["n_r"], case["p"], 8.0 if case["precision"] == "mixed" else 16.0)
        if case["n_E"] and case["precision"] == "double":
            x, y = _work_transport(N, case["n_r"], case["n_E"])
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    n = case["n"]
    b, f = _work_transport(N, n, case["n_E"])
    if kind == "refine":  # two sweeps: residuals, two-fold bases of the groups of 16, their pencils
        b, f = b + 2 * 16.0 * N * n, f + 2 * N * n * (4.0 * STENCIL_FLOPS + 8.0 * 6 * 32)
    return {"bytes": b, "flops": f}
