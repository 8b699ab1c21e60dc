"""The calls that users of this library make, over the sizes they make them at.

The library finds the k eigenpairs of A v = lambda B v nearest an interior
shift.  A program either calls a whole solve (plhr.solve,
plhr.hamiltonian_eigh) or drives the pieces itself: operator products,
applications of a preconditioner, projected Grams and the projected extraction
step.  The listed cases take one of each at the size of this repository's own
workloads (2D 32 x 32, 3D 128^3 Laplacians with absolute-value multigrid, the
64^3 Hamiltonian with the Teter-Payne-Allan preconditioner, the 64^3-element
trilinear finite elements) or a ragged neighbour of it; draw() spreads over the
ranges around them.

Blocks are n x columns, row-major FP64 (FP32 for the FP32 V-cycle), grid
points flattened x fastest.  Inputs come from the seed alone; exact() gives the
same results from plain torch or numpy in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1408_0042_gb300 as plhr

# A V-cycle's shift relative to the mesh: sqrt(sigma) h of the 128^3 workload
# (sigma = 1068.57, h = 1/129) is 0.2534.
_SIGMA_H2 = 1068.5711114200 / 129.0 ** 2


def listed():
    return [
        # One product with the smallest operator of the tests and of the 2D
        # workload: a call whose cost is its latency.
        {"name": "apply_lap2d_32x32", "fn": "apply", "op": "lap2d", "nx": 32, "ny": 32, "nz": 1, "cols": 6},
        # A V of the 128^3 workload (k + guard = 16 columns).
        {"name": "apply_lap3d_128", "fn": "apply", "op": "lap3d", "nx": 128, "ny": 128, "nz": 128, "cols": 16},
        # Stiffness and mass products of the generalized finite-element pencil
        # (64^3 elements, k = 8 and one guard column).
        {"name": "q1_pair_64", "fn": "q1", "nx": 64, "ny": 64, "nz": 64, "cols": 9},
        # T R in FP64, the form of the default all-FP64 solve, on the profiling
        # grid of the 3D workload.
        {"name": "avmg_f64_64", "fn": "avmg", "form": "f64", "nx": 64, "ny": 64, "nz": 64, "levels": 3, "cols": 16},
        # [S | Q_W] = T [...] of the FP32 phase of the 128^3 mixed solve.
        {"name": "avmg_f32_128", "fn": "avmg", "form": "f32", "nx": 128, "ny": 128, "nz": 128, "levels": 4,
         "cols": 32},
        # T R in double-word arithmetic on a box with three unequal axes and a
        # block some of whose columns are already locked.
        {"name": "avmg_dw_96x80x64", "fn": "avmg", "form": "dw", "nx": 96, "ny": 80, "nz": 64, "levels": 3,
         "cols": 11},
        # T R for the 64^3 Hamiltonian (k + guard = 10).
        {"name": "tpa_64", "fn": "tpa", "nx": 64, "ny": 64, "nz": 64, "cols": 10},
        # The Grams of the 64^3 Hamiltonian's FP64 solve, trial basis [V W S P]
        # with two locked columns.
        {"name": "gram_f64_64_m36", "fn": "gram", "form": "f64", "nx": 64, "ny": 64, "nz": 64, "kp": 10, "na": 8},
        # The Grams of the 128^3 workload's FP64-storage phase, full basis.
        {"name": "gram_dw_128_m64", "fn": "gram", "form": "dw", "nx": 128, "ny": 128, "nz": 128, "kp": 16, "na": 16},
        # One projected extraction of the 128^3 workload.
        {"name": "extract_m64", "fn": "extract", "kp": 16, "na": 16},
        # A whole all-FP64 call, forward and backward: eigenpairs of a
        # Hamiltonian and the gradient of a loss on them, tight tolerance.
        {"name": "ham_grad_48", "fn": "ham_grad", "nx": 48, "ny": 48, "nz": 48, "k": 6},
        # A whole mixed-precision call with multigrid: the eigenvalues nearest
        # the shift and the density of their eigenvectors, tight tolerance.
        {"name": "solve_mixed_112x96x80", "fn": "solve_mixed", "nx": 112, "ny": 96, "nz": 80, "levels": 4, "k": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges."""
    fn = rng.choice(["apply", "apply", "q1", "avmg", "avmg", "avmg", "tpa", "gram", "gram", "extract", "ham_grad",
                     "solve_mixed"])
    if fn == "apply":
        op = rng.choice(["lap2d", "lap3d", "ham"])
        cols = rng.randint(1, 24)
        if op == "lap2d":
            return {"fn": fn, "op": op, "nx": _log_int(rng, 24, 1400), "ny": _log_int(rng, 24, 1400), "nz": 1,
                    "cols": cols}
        return {"fn": fn, "op": op, "nx": _log_int(rng, 12, 128), "ny": _log_int(rng, 12, 128),
                "nz": _log_int(rng, 12, 128), "cols": min(cols, 16)}
    if fn == "q1":
        return {"fn": fn, "nx": _log_int(rng, 8, 64), "ny": _log_int(rng, 8, 64), "nz": _log_int(rng, 8, 64),
                "cols": rng.randint(1, 12)}
    if fn == "avmg":
        form = rng.choice(["f64", "f32", "dw"])
        levels = rng.choice([2, 3, 4]) if form == "f32" else rng.choice([2, 3])
        f = 2 ** (levels - 1)
        coarse = [rng.randint(5, 16) for _ in range(3)]
        return {"fn": fn, "form": form, "nx": f * coarse[0], "ny": f * coarse[1], "nz": f * coarse[2],
                "levels": levels, "cols": rng.randint(1, 32 if form == "f32" else 16)}
    if fn == "tpa":
        return {"fn": fn, "nx": _log_int(rng, 10, 80), "ny": _log_int(rng, 10, 80), "nz": _log_int(rng, 10, 80),
                "cols": rng.randint(1, 16)}
    if fn == "gram":
        kp = rng.randint(4, 16)
        return {"fn": fn, "form": rng.choice(["f64", "dw"]), "nx": _log_int(rng, 12, 128),
                "ny": _log_int(rng, 12, 128), "nz": _log_int(rng, 12, 128), "kp": kp, "na": rng.randint(1, kp)}
    if fn == "extract":
        kp = rng.randint(4, 16)
        return {"fn": fn, "kp": kp, "na": rng.randint(max(1, kp - 6), kp)}
    if fn == "ham_grad":
        return {"fn": fn, "nx": rng.randint(20, 48), "ny": rng.randint(20, 48), "nz": rng.randint(20, 48),
                "k": rng.randint(3, 5)}
    return {"fn": fn, "nx": 4 * rng.randint(8, 20), "ny": 4 * rng.randint(8, 16), "nz": 4 * rng.randint(8, 12),
            "levels": 3, "k": rng.randint(3, 6)}


# ----------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda")


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _lap(X, dims, h, periodic=False, scale=1.0):
    """Negative finite-difference Laplacian of a block (n x c, x fastest)."""
    d = [N for N in reversed(dims)]
    Y = X.reshape(*d, -1)
    out = 2.0 * len(d) * Y
    for a in range(len(d)):
        if periodic:
            out = out - torch.roll(Y, 1, a) - torch.roll(Y, -1, a)
        else:
            lo = Y.narrow(a, 0, d[a] - 1)
            hi = Y.narrow(a, 1, d[a] - 1)
            out.narrow(a, 1, d[a] - 1).sub_(lo)
            out.narrow(a, 0, d[a] - 1).sub_(hi)
    return (out * (scale / h ** 2)).reshape(X.shape)


def _modes(dims, cols, gen):
    """A block of Ritz-vector-like columns: a standing wave of random
    wavenumbers in each column with a tenth of noise."""
    n = int(np.prod(dims))
    X = torch.randn(n, cols, generator=gen, device=_dev(), dtype=torch.float64).mul_(0.1)
    Y = X.reshape(*reversed(dims), cols)
    wave = None
    for a, N in enumerate(reversed(dims)):
        q = torch.randint(1, max(2, N // 8 + 1), (cols,), generator=gen, device=_dev()).to(torch.float64)
        p = torch.arange(1, N + 1, device=_dev(), dtype=torch.float64)
        s = torch.sin(p[:, None] * q[None, :] * (math.pi / (N + 1)))
        s = s.reshape([N if b == a else 1 for b in range(len(dims))] + [cols])
        wave = s if wave is None else wave * s
    Y.add_(wave)
    return X


def _dims(case):
    return (case["nx"], case["ny"]) if case.get("nz", 1) == 1 else (case["nx"], case["ny"], case["nz"])


def _mesh(case):
    return 1.0 / (case["nx"] + 1)


def _apply_inputs(case, seed):
    dims, gen = _dims(case), _gen(seed)
    X = _modes(dims, case["cols"], gen)
    pot = -4.0 * torch.rand(X.shape[0], generator=gen, device=_dev(), dtype=torch.float64) if case["op"] == "ham" else None
    return X, pot


def _q1_inputs(case, seed):
    gen = _gen(seed)
    E = (case["nx"], case["ny"], case["nz"])
    X = _modes(tuple(e - 1 for e in E), case["cols"], gen)
    # the coefficient of the finite-element workload: 1 or 10 per element
    c = 1.0 + 9.0 * torch.randint(0, 2, (E[2], E[1], E[0]), generator=gen, device=_dev()).to(torch.float64)
    return E, X, c


def _avmg_inputs(case, seed):
    X = _modes(_dims(case), case["cols"], _gen(seed))
    return X.to(torch.float32) if case["form"] == "f32" else X


def _tpa_inputs(case, seed):
    gen = _gen(seed)
    X = _modes(_dims(case), case["cols"], gen)
    pot = -4.0 * torch.rand(X.shape[0], generator=gen, device=_dev(), dtype=torch.float64)
    return X, pot


def _gram_inputs(case, seed):
    """The trial basis [V W S P], its image and its T-harmonic image, block by
    block, columns as unevenly scaled as a converging iteration leaves them."""
    dims, gen, h = _dims(case), _gen(seed), _mesh(case)
    sigma = _SIGMA_H2 / h ** 2
    # T diagonal, so that U^T Q is symmetric as it is in the solver
    t = (h ** 2 / 6.0) * (0.7 + 0.6 * torch.rand(int(np.prod(dims)), 1, generator=gen, device=_dev(),
                                                 dtype=torch.float64))
    Z, AZ, Q = [], [], []
    for b, nc in enumerate((case["kp"], case["na"], case["na"], case["kp"])):
        z = _modes(dims, nc, gen)
        size = torch.rand(nc, generator=gen, device=_dev(), dtype=torch.float64)
        z.mul_(10.0 ** (-2.0 * size * (0, 3, 2, 1)[b]))
        az = _lap(z, dims, h)
        Z.append(z)
        AZ.append(az)
        Q.append((az - sigma * z).mul_(t))
    cs = torch.cat([1.0 / z.norm(dim=0) for z in Z])
    return Z, AZ, Q, sigma, cs


def _extract_inputs(case, seed):
    """Grams of a block iteration under way on a 48 x 40 Laplacian: V near the
    eigenvectors closest to sigma, W and S the preconditioned residuals, P
    earlier directions, T near |A - sigma|^{-1} and not commuting with A."""
    gen, nx, ny, h = _gen(seed), 48, 40, 1.0 / 49
    kp, na = case["kp"], case["na"]
    rnd = lambda *s: torch.randn(*s, generator=gen, device=_dev(), dtype=torch.float64)  # noqa: E731

    def axis(N):
        p = torch.arange(1, N + 1, device=_dev(), dtype=torch.float64)
        S = torch.sin(p[:, None] * p[None, :] * (math.pi / (N + 1))) * math.sqrt(2.0 / (N + 1))
        return S, (4.0 / h ** 2) * torch.sin(p * (math.pi / (2 * (N + 1)))) ** 2

    (Sx, mx), (Sy, my) = axis(nx), axis(ny)
    mu = (my[:, None] + mx[None, :]).reshape(-1)
    n, sigma = nx * ny, float(300.0 + 400.0 * torch.rand(1, generator=gen, device=_dev(), dtype=torch.float64))
    modes = lambda X: torch.einsum("ab,cd,bdk->ack", Sy, Sx, X.reshape(ny, nx, -1)).reshape(n, -1)  # noqa: E731
    M = rnd(n, 48)
    A = lambda X: _lap(X, (nx, ny), h)  # noqa: E731
    d = 1.0 / ((mu - sigma).abs() + 20.0)
    T = lambda X: modes(d[:, None] * modes(X)) + (2e-3 / n) * (M @ (M.T @ X))  # noqa: E731
    near = torch.argsort((mu - sigma).abs())[:kp]
    C = 0.02 * rnd(n, kp) * (d[:, None] / d.max())
    C[near, torch.arange(kp, device=_dev())] += 1.0
    V = modes(C)
    V = V / V.norm(dim=0)
    lam = (V * A(V)).sum(0)
    W = T(A(V) - V * lam)[:, :na]
    S = T(A(W) - W * lam[:na])
    P = T(rnd(n, kp))
    Z = torch.cat([V, W, S, P], 1)
    cs = 1.0 / Z.norm(dim=0)
    Zs = Z * cs
    U = A(Zs) - sigma * Zs
    Q = T(U)
    Guq = U.T @ Q
    Gzz = Zs.T @ Zs
    return 0.5 * (Gzz + Gzz.T), 0.5 * (Guq + Guq.T), Q.T @ Zs, cs


def _nearest(lam, sigma, count):
    return np.lexsort((lam, np.abs(lam - sigma)))[:count]


def _pick_shift(lam, k, lo, hi, inner):
    """A shift whose k nearest eigenvalues (sorted values lam, shifts between
    indices lo and hi) stand apart: the widest gap to the rest and, with inner,
    between themselves, in the units of the relative residual."""
    best, where = -1.0, None
    for i in range(lo, hi):
        w = lam[i:i + k]
        below = lam[i] - lam[i - 1] if i > 0 else np.inf
        above = lam[i + k] - lam[i + k - 1]
        # the shift has to see the window [i, i + k) as the k nearest, with room
        # for half the smaller outer gap, and no two at the same distance
        s = 0.5 * (w[0] + w[-1]) + 0.11 * min(below, above)
        gap = min(below, above)
        if inner and k > 1:
            gap = min(gap, 2.0 * np.min(np.diff(w)), 2.0 * np.min(np.diff(np.sort(np.abs(w - s)))))
        score = gap / max(abs(s), 1.0)
        if score > best:
            best, where = score, s
    return float(where)


def _ham_inputs(case, seed):
    """A separable potential (a quantum dot of three unequal axes: one Gaussian
    well with two shallow satellites per axis), so that plain numpy knows the
    eigenpairs."""
    rng = np.random.RandomState(seed % (1 << 31))
    dims = _dims(case)
    axes, evs, vecs = [], [], []
    for N, wide in zip(dims, (1.5, 2.1, 3.0)):
        x = np.arange(N, dtype=np.float64)
        v = np.zeros(N)
        for depth, width, where in ((rng.uniform(1.4, 1.8), wide * rng.uniform(0.9, 1.1), 0.5 + rng.uniform(-0.05, 0.05)),
                                    (rng.uniform(0.1, 0.3), rng.uniform(2.0, 3.0), rng.uniform(0.1, 0.3)),
                                    (rng.uniform(0.1, 0.3), rng.uniform(2.0, 3.0), rng.uniform(0.7, 0.9))):
            r = np.abs(x - where * N)
            r = np.minimum(r, N - r)
            v -= depth * np.exp(-r * r / (2.0 * width * width))
        H = np.diag(v + 1.0)
        i = np.arange(N)
        H[i, (i + 1) % N] -= 0.5
        H[(i + 1) % N, i] -= 0.5
        e, y = np.linalg.eigh(H)
        axes.append(v)
        evs.append(e)
        vecs.append(y)
    V = (axes[2][:, None, None] + axes[1][None, :, None] + axes[0][None, None, :]).ravel()
    lam = (evs[2][:, None, None] + evs[1][None, :, None] + evs[0][None, None, :]).ravel()
    low = np.sort(np.partition(lam, 60)[:60])
    k = case["k"]
    sigma = _pick_shift(low, k, 1, 5, True)
    w = rng.uniform(0.5, 1.5, k)
    mask = (rng.uniform(size=V.size) < 0.5).astype(np.float64)
    return V, sigma, w, mask, evs, vecs, lam


def _mixed_inputs(case, seed):
    """A box whose edge varies with the seed, the shift in a clear gap."""
    rng = np.random.RandomState(seed % (1 << 31))
    dims, h = _dims(case), rng.uniform(0.9, 1.1) / (case["nx"] + 1)
    mus = [4.0 / h ** 2 * np.sin(np.arange(1, N + 1) * np.pi / (2.0 * (N + 1))) ** 2 for N in dims]
    lam = (mus[2][:, None, None] + mus[1][None, :, None] + mus[0][None, None, :]).ravel()
    low = np.sort(np.partition(lam, 120)[:120])
    sigma = _pick_shift(low, case["k"], 20, 60, False)
    return dims, h, sigma, mus, lam


# ----------------------------------------------------------------- the calls
def prepare(case, seed):
    fn = case["fn"]
    if fn == "apply":
        X, pot = _apply_inputs(case, seed)
        if case["op"] == "ham":
            A = plhr.Operator.hamiltonian(_dims(case), 1.0, pot)
        else:
            A = plhr.Operator.laplacian(_dims(case), _mesh(case))
        return {"fn": fn, "A": A, "X": X}
    if fn == "q1":
        E, X, c = _q1_inputs(case, seed)
        return {"fn": fn, "A": plhr.Operator.q1_stiffness(E, c), "B": plhr.Operator.q1_mass(E), "X": X}
    if fn == "avmg":
        h = _mesh(case)
        A = plhr.Operator.laplacian(_dims(case), h)
        T = plhr.AVMG(A, _SIGMA_H2 / h ** 2, levels=case["levels"], nu=2, transfer=1, coarse=1)
        return {"fn": fn, "form": case["form"], "T": T, "R": _avmg_inputs(case, seed)}
    if fn == "tpa":
        X, pot = _tpa_inputs(case, seed)
        A = plhr.Operator.hamiltonian(_dims(case), 1.0, pot)
        return {"fn": fn, "A": A, "T": plhr.TPA(A, -1.4, 2.6), "R": X}
    if fn == "gram":
        Z, AZ, Q, sigma, cs = _gram_inputs(case, seed)
        return {"fn": fn, "form": plhr.GRAM_DW if case["form"] == "dw" else plhr.GRAM_F64, "Z": Z, "AZ": AZ, "Q": Q,
                "sigma": sigma, "cs": cs}
    if fn == "extract":
        Gzz, Guq, Gqz, cs = _extract_inputs(case, seed)
        return {"fn": fn, "G": (Gzz, Guq, Gqz, cs), "kp": case["kp"]}
    if fn == "ham_grad":
        V, sigma, w, mask, _, _, _ = _ham_inputs(case, seed)
        t = lambda x: torch.from_numpy(x).to(_dev())  # noqa: E731
        return {"fn": fn, "V": t(V).requires_grad_(), "sigma": sigma, "w": t(w), "mask": t(mask), "k": case["k"],
                "dims": _dims(case)}
    dims, h, sigma, _, _ = _mixed_inputs(case, seed)
    A = plhr.Operator.laplacian(dims, h)
    T = plhr.AVMG(A, sigma, levels=case["levels"], nu=2, transfer=1, coarse=1)
    kp = case["k"] + 2
    v0 = torch.rand(A.n, kp, generator=_gen(seed), device=_dev(), dtype=torch.float64) - 0.5
    return {"fn": fn, "A": A, "T": T, "sigma": sigma, "k": case["k"], "v0": v0}


def run(state):
    fn = state["fn"]
    if fn == "apply":
        return state["A"].apply(state["X"])
    if fn == "q1":
        return state["A"].apply_pair(state["B"], state["X"])
    if fn == "avmg":
        T, R = state["T"], state["R"]
        return T.apply(R) if state["form"] == "f64" else T.apply_f32(R) if state["form"] == "f32" else T.apply_dw(R)
    if fn == "tpa":
        return state["T"].apply(state["R"])
    if fn == "gram":
        return plhr.gram(state["form"], state["Z"], state["AZ"], state["Q"], sigma=state["sigma"],
                         colscale=state["cs"])
    if fn == "extract":
        return plhr.tharm_extract(*state["G"], kp=state["kp"], nv=state["kp"])
    if fn == "ham_grad":
        V, mask = state["V"], state["mask"]
        lam, vecs = plhr.hamiltonian_eigh(V, state["dims"], 1.0, state["sigma"], state["k"], tol=_HAM_TOL,
                                          prec="tpa")
        loss = (state["w"] * lam).sum() + (mask[:, None] * vecs * vecs).sum()
        (grad,) = torch.autograd.grad(loss, V)
        return {"lam": lam.detach(), "grad": grad}
    lam, vecs, _ = plhr.solve(state["A"], state["sigma"], state["k"], T=state["T"], tol=_MIXED_TOL,
                              v_init=state["v0"], guard=2, precision=plhr.PRECISION_MIXED, raise_on_notconv=True)
    return {"lam": lam, "density": plhr.eigval_grad(vecs, np.ones(state["k"]))}


# Tolerances of the whole calls: as tight as a program asks that takes
# gradients or densities from the eigenvectors (their error is the residual
# over the gap to the next eigenvalue).
_HAM_TOL = 3e-11
_MIXED_TOL = 1e-10


# ----------------------------------------------------------------- the work
def work(case):
    fn = case["fn"]
    if fn == "extract":
        m = 2 * case["kp"] + 2 * case["na"]
        # the matrices in and the coefficients out; Hessenberg reduction (10/3 m^3)
        # and QR iteration (10 m^3) of the projected problem
        return {"bytes": 8.0 * (3 * m * m + m * case["kp"] + case["kp"] ** 2), "flops": 40.0 / 3.0 * m ** 3}
    if fn == "q1":
        n = float((case["nx"] - 1) * (case["ny"] - 1) * (case["nz"] - 1))
        c = case["cols"]
        return {"bytes": 8.0 * (3 * n * c + case["nx"] * case["ny"] * case["nz"]), "flops": 2.0 * 2 * 27 * n * c}
    n = float(case["nx"] * case["ny"] * case["nz"])
    d = len(_dims(case))
    if fn == "apply":
        return {"bytes": 16.0 * n * case["cols"] + (8.0 * n if case["op"] == "ham" else 0.0),
                "flops": (2.0 * d + 1) * n * case["cols"]}
    if fn == "avmg":
        # levels of the hierarchy above the coarsest: four sweeps and a residual
        # with B_l (two products where B_l is the polynomial), two transfers
        eb, c, flops, h = (4.0 if case["form"] == "f32" else 8.0), case["cols"], 0.0, _mesh(case)
        for s in range(case["levels"] - 1):
            poly = math.sqrt(_SIGMA_H2) * 2 ** s >= 2.0 * math.pi / 10.0
            flops += n / 8.0 ** s * c * ((4 if poly else 3.5) * (20 if poly else 9) + 4)
        return {"bytes": 2.0 * eb * n * c, "flops": flops}
    if fn == "tpa":
        return {"bytes": 16.0 * n * case["cols"], "flops": n * case["cols"] * (5.0 * math.log2(n) + 1)}
    if fn == "gram":
        m = 2 * case["kp"] + 2 * case["na"]
        return {"bytes": 8.0 * 3 * n * m, "flops": 2.0 * n * (m * (m + 1) + m * m)}
    # whole solves, per iteration the Grams, the update, two operator products
    # and the preconditioner; about 60 iterations for the Hamiltonian at its
    # tolerance, 30 for the Laplacian with multigrid
    kp = case["k"] + 2
    m = 4 * kp
    its = 60.0 if fn == "ham_grad" else 30.0
    per_point = 2.0 * (m * (m + 1) + m * m) + 4.0 * m * kp + 16.0 * kp + 400.0 * kp
    return {"bytes": 8.0 * n * (2 * kp + 1), "flops": its * n * per_point}


# ----------------------------------------------------------------- 64-bit results
def _q1_exact(case, seed):
    E, X, c = _q1_inputs(case, seed)
    h, cols = 1.0 / E[0], X.shape[1]
    k1 = np.array([[1.0, -1.0], [-1.0, 1.0]]) / h
    m1 = np.array([[2.0, 1.0], [1.0, 2.0]]) * h / 6.0
    # nodes with the boundary: (Ez + 1, Ey + 1, Ex + 1, cols)
    P = torch.zeros(E[2] + 1, E[1] + 1, E[0] + 1, cols, device=_dev(), dtype=torch.float64)
    P[1:-1, 1:-1, 1:-1] = X.reshape(E[2] - 1, E[1] - 1, E[0] - 1, cols)
    YA, YB = torch.zeros_like(P), torch.zeros_like(P)
    at = lambda q, i: q[(i >> 2):(i >> 2) + E[2], ((i >> 1) & 1):((i >> 1) & 1) + E[1], (i & 1):(i & 1) + E[0]]  # noqa: E731
    for i in range(8):
        for j in range(8):
            iz, iy, ix, jz, jy, jx = i >> 2, (i >> 1) & 1, i & 1, j >> 2, (j >> 1) & 1, j & 1
            K = (k1[iz, jz] * m1[iy, jy] * m1[ix, jx] + m1[iz, jz] * k1[iy, jy] * m1[ix, jx]
                 + m1[iz, jz] * m1[iy, jy] * k1[ix, jx])
            at(YA, i).add_(c[..., None] * at(P, j), alpha=float(K))
            at(YB, i).add_(at(P, j), alpha=float(m1[iz, jz] * m1[iy, jy] * m1[ix, jx]))
    return tuple(y[1:-1, 1:-1, 1:-1].reshape(-1, cols) for y in (YA, YB))


def _along(M, X, axis):
    """M applied along one axis of X."""
    return torch.movedim(torch.tensordot(M, X, dims=([1], [axis])), 0, axis)


def _vcycle(R, dims, h, sigma, levels):
    """The absolute-value multigrid V-cycle (Appendix A, Algorithm 4) with two
    Richardson sweeps, trilinear cell-centred transfers and the coarsest solve
    on the fine grid's spectrum."""
    def prolong(Nc):
        P = np.zeros((2 * Nc, Nc))
        for i in range(Nc):
            P[2 * i, i] = P[2 * i + 1, i] = 0.75
            if i > 0:
                P[2 * i, i - 1] = 0.25
            if i < Nc - 1:
                P[2 * i + 1, i + 1] = 0.25
        return torch.from_numpy(P).to(_dev())

    def cycle(r, dl, hl, left):
        shape = tuple(reversed(dl))
        if left == 1:
            X, denom = r.reshape(*shape, -1), None
            for a, (N0, N) in enumerate(zip(shape, reversed(dims))):
                p, m = np.arange(N0) + 0.5, np.arange(1, N0 + 1)
                S = np.sin(np.outer(p, m) * np.pi / N0)
                S /= np.linalg.norm(S, axis=0)
                mu = torch.from_numpy(4.0 / h ** 2 * np.sin(m * np.pi / (2.0 * (N + 1))) ** 2).to(_dev())
                mu = mu.reshape([N0 if b == a else 1 for b in range(len(shape))] + [1])
                denom = mu if denom is None else denom + mu
                X = _along(torch.from_numpy(S.T.copy()).to(_dev()), X, a)
            X = X / (denom - sigma).abs()
            for a, N0 in enumerate(shape):
                p, m = np.arange(N0) + 0.5, np.arange(1, N0 + 1)
                S = np.sin(np.outer(p, m) * np.pi / N0)
                S /= np.linalg.norm(S, axis=0)
                X = _along(torch.from_numpy(S).to(_dev()), X, a)
            return X.reshape(r.shape)
        lo, hi = -sigma, 4.0 * len(dl) / hl ** 2 - sigma
        poly = not math.sqrt(sigma) * hl < 2.0 * math.pi / 10.0
        c = 0.5 * max(abs(lo), abs(hi))
        beta = (max(lo * lo, hi * hi) + c * c) / (2.0 * c) if poly else 4.0 * len(dl) / hl ** 2

        def B(x):
            y = _lap(x, dl, hl)
            if not poly:
                return y
            y = y - sigma * x
            return (_lap(y, dl, hl) - sigma * y + c * c * x) / (2.0 * c)

        w = r / beta
        w = w + (r - B(w)) / beta
        res = (r - B(w)).reshape(*shape, -1)
        for a, N in enumerate(shape):
            res = _along(0.5 * prolong(N // 2).T, res, a)
        half = tuple(N // 2 for N in dl)
        wc = cycle(res.reshape(-1, r.shape[1]), half, 2.0 * hl, left - 1).reshape(*reversed(half), -1)
        for a, N in enumerate(shape):
            wc = _along(prolong(N // 2), wc, a)
        w = w + wc.reshape(w.shape)
        for _ in range(2):
            w = w + (r - B(w)) / beta
        return w

    return cycle(R, tuple(dims), h, levels)


def _tpa_exact(case, seed):
    X, _ = _tpa_inputs(case, seed)
    dims, shape = _dims(case), tuple(reversed(_dims(case)))
    mu = None
    for a, N in enumerate(shape):
        m = torch.arange(N, device=_dev(), dtype=torch.float64)
        e = (1.0 - torch.cos(2.0 * math.pi * m / N)).reshape([N if b == a else 1 for b in range(3)])
        mu = e if mu is None else mu + e
    x = mu / 2.6
    num = 27.0 + 18.0 * x + 12.0 * x ** 2 + 8.0 * x ** 3
    K = num / (num + 16.0 * x ** 4)
    F = torch.fft.fftn(X.reshape(*shape, -1), dim=(0, 1, 2))
    return torch.fft.ifftn(K[..., None] * F, dim=(0, 1, 2)).real.reshape(X.shape).contiguous()


def _gram_exact(case, seed):
    Z, AZ, Q, sigma, cs = _gram_inputs(case, seed)
    Z, AZ, Q = torch.cat(Z, 1), torch.cat(AZ, 1), torch.cat(Q, 1)
    U = (AZ - sigma * Z) * cs
    Z, Q = Z * cs, Q * cs
    return torch.stack([Z.T @ Z, U.T @ Q, Q.T @ Z])


def _extract_exact(case, seed):
    """The T-harmonic values nearest zero, a conjugate pair counted once."""
    Gzz, Guq, Gqz, _ = (x.cpu().numpy() for x in _extract_inputs(case, seed))
    L = np.linalg.cholesky(Guq)
    H = np.linalg.solve(L, np.linalg.solve(L, Gqz).T).T
    xi = 1.0 / np.linalg.eigvals(H)
    xi = xi[np.lexsort((xi.real, np.abs(xi)))]
    units, cols = [], 0
    for x in xi:
        if x.imag < 0:
            continue
        if cols >= case["kp"]:
            break
        units.append((x.real, x.imag))
        cols += 2 if x.imag > 0 else 1
    none = dict.fromkeys(("Cp", "Cvv", "tags", "partner", "status", "kept", "units"))
    return {**none, "xi": np.array(units)}


def _ham_exact(case, seed):
    V, sigma, w, mask, evs, vecs, lam = _ham_inputs(case, seed)
    k, shape = case["k"], tuple(reversed(_dims(case)))
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(_dev())  # noqa: E731
    idx = _nearest(lam, sigma, k)
    own = np.stack(np.unravel_index(idx, shape))
    Y = torch.stack([(t(vecs[2][:, a])[:, None, None] * t(vecs[1][:, b])[None, :, None]
                      * t(vecs[0][:, c])[None, None, :]).reshape(-1) for a, b, c in own.T], 1)
    L, all_lam, m = t(lam[idx]), t(lam.reshape(shape)), t(mask)
    grad = (Y * Y) @ t(w)
    for j in range(k):
        # sum over all other modes i of v_i (v_i . g) / (lambda_j - lambda_i)
        G = (2.0 * m * Y[:, j]).reshape(shape)
        for a in range(3):
            G = _along(t(vecs[2 - a].T), G, a)
        d = L[j] - all_lam
        d[tuple(own[:, j])] = float("inf")
        G = G / d
        for a in range(3):
            G = _along(t(vecs[2 - a]), G, a)
        grad = grad + Y[:, j] * G.reshape(-1)
    return {"lam": L, "grad": grad}


def _mixed_exact(case, seed):
    dims, h, sigma, mus, lam = _mixed_inputs(case, seed)
    shape = tuple(reversed(dims))
    idx = _nearest(lam, sigma, case["k"])
    dens = np.zeros(shape)
    for a in np.stack(np.unravel_index(idx, shape)).T:
        s = [np.sin(np.arange(1, N + 1) * (i + 1) * np.pi / (N + 1)) ** 2 * 2.0 / (N + 1) for N, i in zip(shape, a)]
        dens += s[0][:, None, None] * s[1][None, :, None] * s[2][None, None, :]
    return {"lam": lam[idx], "density": dens.ravel()}


def exact(case, seed):
    fn = case["fn"]
    if fn == "apply":
        X, pot = _apply_inputs(case, seed)
        if case["op"] == "ham":
            return _lap(X, _dims(case), 1.0, periodic=True, scale=0.5) + pot[:, None] * X
        return _lap(X, _dims(case), _mesh(case))
    if fn == "q1":
        return _q1_exact(case, seed)
    if fn == "avmg":
        h = _mesh(case)
        return _vcycle(_avmg_inputs(case, seed).to(torch.float64), _dims(case), h, _SIGMA_H2 / h ** 2,
                       case["levels"])
    if fn == "tpa":
        return _tpa_exact(case, seed)
    if fn == "gram":
        return _gram_exact(case, seed)
    if fn == "extract":
        return _extract_exact(case, seed)
    return _ham_exact(case, seed) if fn == "ham_grad" else _mixed_exact(case, seed)
