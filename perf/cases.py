"""The measured workloads of the library: what a program that solves A x = b with the two-grid
method has it do, through the public entry points of ``paper_2005_03070_gb300``.

A case names one of six uses (``op``):

  phase1   one coarse phase and its use: coarse GMRES-DR(m, k) for a fixed number of cycles
           (with the moved vectors, A Y and its factorisation), the coarse solution
           prolonged, its residual, and the first deflation projection.  The basis itself is
           defined only up to a rotation of its span, so the case returns what the program
           computes with it: x_c, and the projected x and r at full length.
  solve    a fine-grid solve with a deflation basis that the program already holds (the basis
           is reused across right-hand sides): BiCGStab-Proj, GMRES-Proj or IDR-Proj.
  twogrid  the whole step in the float32 + refinement form: float32 coarse phase,
           prolongation, float32 cycles refined in float64.
  basis    a saved basis loaded into a deflation handle: A Y and CholQR2.
  batch    many 2D instances x 8 right-hand sides: set-up and solve.
  adjoint  the differentiable solve: forward and backward through autograd.

Tolerances are tight (1e-12 or 1e-13) where a solution is returned, so that x is determined by
the problem and not by the rounding of one run; the coarse phases run a fixed number of
cycles, so that a pass is the same work whatever the rounding.
"""
import math

import numpy as np
import torch

from paper_2005_03070_gb300 import tg
from paper_2005_03070_gb300.autograd import two_grid_solve

BETA3 = (2.0, 1.0, 0.5)          # the 3D workload's convection
EXP2D = (40.0, 40.0, 5.0)        # -exp(5xy) Lap u + 40 u_x + 40 u_y


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest two-grid problem in use: launches and the m x m step count
        dict(name="phase1_cd2d_127", op="phase1", kind="cd2d", N=127, m=30, k=15, cycles=6),
        # an ordinary 2D grid; the 60-column coarse phase of the batched workload's instances
        dict(name="phase1_cd2d_511", op="phase1", kind="cd2d", N=511, m=60, k=20, cycles=6),
        # the headline 3D workload's coarse phase: coarse 127^3, GMRES-DR(60, 30), float64
        dict(name="phase1_cd3d_255", op="phase1", kind="cd3d", N=255, m=60, k=30, cycles=5),
        # the 32^4 U(1) lattice, complex128, GMRES-DR(80, 40) on 16^4
        dict(name="phase1_u1_32", op="phase1", kind="u1_4d", N=32, m=80, k=40, cycles=3),
        # a second right-hand side on the smallest problem, restarted every 60 products
        dict(name="solve_cd2d_127", op="solve", kind="cd2d", N=127, k=15, method="bicgstab", precision="f64",
             ncyc=0, rtol=1e-12),
        # a second right-hand side of the headline workload, BiCGStab(20)-Proj(30), float64
        dict(name="solve_cd3d_255", op="solve", kind="cd3d", N=255, k=30, method="bicgstab", precision="f64",
             ncyc=20, rtol=1e-13),
        # the whole headline step in the float32 + refinement form
        dict(name="twogrid_f32_cd3d_255", op="twogrid", kind="cd3d", N=255, m=60, k=30, cycles=10, ncyc=20,
             rtol=1e-13),
        # the paper's other fine-grid methods
        dict(name="gmres_cd3d_95", op="solve", kind="cd3d", N=95, k=30, method="gmres", precision="f64",
             ncyc=20, rtol=1e-12),
        dict(name="idr_exp2d_127", op="solve", kind="exp2d", N=127, k=30, method="idr", precision="f64", ncyc=20,
             rtol=1e-12),
        # a basis saved by an earlier run, loaded for the 3D workload's smaller grid
        dict(name="basis_cd3d_191", op="basis", kind="cd3d", N=191, k=30),
        # a cut of the batched workload (N_i odd, beta_i in [0.5, 4], 8 right-hand sides each)
        dict(name="batch_6", op="batch", count=6, nmin=127, nmax=511, m=60, k=20, cycles=12, ncyc=20, rtol=1e-12),
        # gradient of a loss through the variable-coefficient solve, forward and backward; the
        # coarse phases stop at 5 converged pairs of the 20 kept
        dict(name="adjoint_127", op="adjoint", kind="vark2d", N=127, m=40, k=20, nev=5, ncyc=20, rtol=1e-12),
    ]


def _odd(rng, lo, hi):
    """An odd size, spread over the logarithm of [lo, hi]."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v | 1))


def draw(rng):
    op = rng.choice(["phase1", "phase1", "phase1", "solve", "solve", "solve", "twogrid", "basis", "batch", "adjoint"])
    if op == "phase1":
        kind = rng.choice(["cd2d", "cd3d", "u1_4d"])
        N = _odd(rng, 63, 511) if kind == "cd2d" else _odd(rng, 31, 191) if kind == "cd3d" else 2 * rng.randint(5, 14)
        m, k = rng.choice([(24, 9), (30, 15), (40, 20), (60, 20), (60, 30), (73, 35)])
        return dict(op=op, kind=kind, N=N, m=m, k=k, cycles=rng.randint(2, 5))
    if op == "solve":
        method = rng.choice(["bicgstab", "bicgstab", "gmres", "idr"])
        precision = rng.choice(["f64", "f32_ir"]) if method == "bicgstab" else "f64"
        kind = rng.choice(["cd2d", "cd3d"])
        N = _odd(rng, 63, 255) if kind == "cd2d" else _odd(rng, 31, 191)
        if method == "gmres":
            N = min(N, 127)
        return dict(op=op, kind=kind, N=N, k=rng.randint(8, 30), method=method, precision=precision,
                    ncyc=rng.choice([0, 20]), rtol=1e-12)
    if op == "twogrid":
        kind = rng.choice(["cd2d", "cd3d"])
        N = _odd(rng, 63, 255) if kind == "cd2d" else _odd(rng, 31, 191)
        m, k = rng.choice([(30, 15), (40, 20), (60, 30)])
        return dict(op=op, kind=kind, N=N, m=m, k=k, cycles=rng.randint(6, 12), ncyc=20, rtol=1e-12)
    if op == "basis":
        kind = rng.choice(["cd2d", "cd3d"])
        N = _odd(rng, 63, 511) if kind == "cd2d" else _odd(rng, 31, 191)
        return dict(op=op, kind=kind, N=N, k=rng.randint(8, 40))
    if op == "batch":
        return dict(op=op, count=rng.randint(2, 6), nmin=63, nmax=rng.choice([127, 255, 383]), m=rng.choice([40, 60]),
                    k=20, cycles=rng.randint(6, 12), ncyc=20, rtol=1e-12)
    return dict(op="adjoint", kind="vark2d", N=_odd(rng, 63, 127), m=40, k=20, nev=5, ncyc=20, rtol=1e-12)


# ------------------------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 64 + stream) & 0x7FFFFFFFFFFF)
    return g


def _randn(seed, stream, n, dtype=torch.float64):
    return torch.randn(n, dtype=dtype, device="cuda", generator=_gen(seed, stream))


def _links(seed, L):
    """Random U(1) link phases, theta ~ U(-pi, pi)."""
    th = (2.0 * torch.rand(4, L ** 4, dtype=torch.float64, device="cuda", generator=_gen(seed, 2)) - 1.0) * math.pi
    return torch.polar(torch.ones_like(th), th)


def _hops(links, v, L):
    U = links.view(4, L, L, L, L)
    v = v.view(L, L, L, L)                       # dims (x3, x2, x1, x0)
    out = torch.zeros_like(v)
    for mu in range(4):
        d = 3 - mu
        out += U[mu] * torch.roll(v, -1, d) + torch.roll(U[mu].conj() * v, 1, d)
    return out.reshape(-1)


def _lattice_mass(links, L, seed):
    """m with the smallest eigenvalue of (m + 8) - hops near 1e-2: the top Ritz value of 80 plain
    Lanczos steps on the hops."""
    v = torch.complex(_randn(seed, 3, L ** 4), _randn(seed, 4, L ** 4))
    v /= torch.linalg.vector_norm(v)
    a, b, prev = [], [], torch.zeros_like(v)
    for _ in range(80):
        w = _hops(links, v, L) - (b[-1] * prev if b else 0.0)
        al = torch.vdot(v, w).real
        w = w - al * v
        a.append(al)
        b.append(torch.linalg.vector_norm(w))
        prev, v = v, w / b[-1]
    T = np.diag([float(x) for x in a])
    off = np.array([float(x) for x in b[:-1]])
    T += np.diag(off, 1) + np.diag(off, -1)
    return float(np.linalg.eigvalsh(T)[-1]) - 8.0 + 1e-2


def _kappa(seed, N):
    """exp of a smooth random field (unit variance, correlation length about 0.1) on the node grid."""
    x = torch.arange(N + 2, dtype=torch.float64, device="cuda") / (N + 1)
    p = torch.arange(1, 13, dtype=torch.float64, device="cuda")
    w = torch.exp(-0.5 * (p * math.pi * 0.1) ** 2 / 2)
    S = torch.cos(math.pi * p[:, None] * x[None, :] + 2 * math.pi * torch.rand(12, 1, dtype=torch.float64, device="cuda",
                                                                               generator=_gen(seed, 5))) * w[:, None]
    z = S.T @ torch.randn(12, 12, dtype=torch.float64, device="cuda", generator=_gen(seed, 6)) @ S
    return torch.exp(z / z.std()).reshape(-1).contiguous()


def _beta(kind):
    return BETA3 if kind == "cd3d" else EXP2D if kind == "exp2d" else (1.0,)


def _modes(kind, N, k):
    """The k coarse-grid eigenvectors of smallest eigenvalue of the constant-coefficient operator
    (products of sines, scaled along each convection direction), coarse (N-1)/2 points per axis."""
    Nc, dim = (N - 1) // 2, 3 if kind == "cd3d" else 2
    h = 1.0 / (Nc + 1)
    beta = (BETA3 if dim == 3 else (1.0, 0.0))[:dim]
    p = np.arange(1, min(Nc, 12) + 1)
    vals = []
    for b in beta:
        lo, hi = -1.0 / h ** 2 - b / (2 * h), -1.0 / h ** 2 + b / (2 * h)
        vals.append(2.0 / h ** 2 - 2.0 * math.sqrt(lo * hi) * np.cos(p * math.pi * h))
    grid = vals[0].reshape((-1,) + (1,) * (dim - 1))
    for a in range(1, dim):
        grid = grid + vals[a].reshape((1,) * a + (-1,) + (1,) * (dim - 1 - a))
    order = np.argsort(grid.reshape(-1), kind="stable")[:k]
    idx = np.stack(np.unravel_index(order, grid.shape), 1) + 1
    t = torch.arange(1, Nc + 1, dtype=torch.float64, device="cuda")
    out = []
    for q in idx:
        f = []
        for a, b in enumerate(beta):
            lo, hi = -1.0 / h ** 2 - b / (2 * h), -1.0 / h ** 2 + b / (2 * h)
            f.append((lo / hi) ** (t / 2) * torch.sin(math.pi * int(q[a]) * t * h))
        v = f[1][:, None] * f[0][None, :]
        if dim == 3:
            v = f[2][:, None, None] * v[None]
        out.append((v / torch.linalg.vector_norm(v)).reshape(-1))
    return torch.stack(out).contiguous()


def _batch_sizes(case, seed):
    g = np.random.default_rng([int(seed), 7])
    # the sizes belong to the case, the convections and right-hand sides to the seed
    q = np.linspace(0.0, 1.0, case["count"])
    Ns = [int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** v)) | 1 for v in q]
    return Ns, [float(b) for b in g.uniform(0.5, 4.0, case["count"])]


def _operator(case, seed):
    if case["kind"] == "u1_4d":
        links = _links(seed, case["N"])
        return tg.Operator("u1_4d", case["N"], links=links, mass=_lattice_mass(links, case["N"], seed))
    return tg.Operator(case["kind"], case["N"], _beta(case["kind"]))


def _vector(case, seed, stream, n):
    if case["kind"] == "u1_4d":
        return torch.complex(_randn(seed, stream, n), _randn(seed, stream + 1, n))
    return _randn(seed, stream, n)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        Ns, betas = _batch_sizes(case, seed)
        b = tg.Batch(Ns, betas)
        return dict(case=case, batch=b, rhs=_randn(seed, 10, b.total))
    if op == "adjoint":
        N = case["N"]
        kappa = _kappa(seed, N).requires_grad_(True)
        b = _randn(seed, 10, N * N).requires_grad_(True)
        return dict(case=case, kappa=kappa, b=b, grad=_randn(seed, 12, N * N))
    A = _operator(case, seed)
    st = dict(case=case, A=A, b=_vector(case, seed, 10, A.n))
    if op == "basis":
        # eigenvectors of the coarse grid, moved, with the errors of an earlier run
        Y = A.prolong(_modes(case["kind"], case["N"], case["k"]))
        st["Y"] = Y + 1e-3 * _randn(seed, 16, Y.numel()) * (torch.linalg.vector_norm(Y) / math.sqrt(Y.numel()))
    elif op == "solve":
        precision = case["precision"]
        if case["kind"] == "exp2d":
            st["defl"] = A.coarse_gmresdr(st["b"], 60, case["k"], rtolev=1e-6, max_cycles=20, precision=precision)[1]
        else:
            Y = A.prolong(_modes(case["kind"], case["N"], case["k"]))
            st["defl"] = A.defl_from_basis(Y, case["k"], precision=precision)
        if case["method"] == "idr":
            st["P"] = _randn(seed, 18, 4 * A.n).view(4, A.n)
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    op = case["op"]
    if op == "phase1":
        A = st["A"]
        # rtolev and rtol below reach: the given number of cycles runs
        xc, defl, _, _ = A.coarse_gmresdr(st["b"], case["m"], case["k"], rtolev=1e-15, rtol=1e-15,
                                          max_cycles=case["cycles"])
        x = A.prolong(xc)
        r = st["b"] - A.apply(x)
        defl.project(x, r)
        return {"xc": xc, "x": x, "r": r}
    if op == "solve":
        A = st["A"]
        x = torch.zeros_like(st["b"])
        restart = 60 if case["ncyc"] == 0 else 0
        if case["method"] == "idr":
            A.solve_idr(st["b"], x, st["P"], st["defl"], rtol=case["rtol"], ncyc=case["ncyc"], restart_mvps=restart)
        else:
            A.solve(st["b"], x, st["defl"], method=case["method"], precision=case["precision"], rtol=case["rtol"],
                    ncyc=case["ncyc"], restart_mvps=restart)
        return {"x": x}
    if op == "twogrid":
        A = st["A"]
        xc, defl, _, _ = A.coarse_gmresdr(st["b"], case["m"], case["k"], rtolev=1e-15, rtol=1e-15,
                                          max_cycles=case["cycles"], precision="f32_ir")
        x = A.prolong(xc)
        A.solve(st["b"], x, defl, precision="f32_ir", rtol=case["rtol"], ncyc=case["ncyc"], restart_mvps=0)
        return {"x": x}
    if op == "basis":
        defl = st["A"].defl_from_basis(st["Y"], case["k"])
        return {"Q": defl.copy(1), "AY": defl.copy(2), "R": defl.copy(3)}
    if op == "batch":
        B = st["batch"]
        B.setup(st["rhs"], m=case["m"], k=case["k"], rtolev=1e-15, rtol=1e-15, max_cycles=case["cycles"])
        x = torch.zeros_like(st["rhs"])
        B.solve(st["rhs"], x, rtol=case["rtol"], ncyc=case["ncyc"])
        return {"x": x}
    kappa, b = st["kappa"], st["b"]
    kappa.grad = b.grad = None
    x = two_grid_solve(kappa, b, case["N"], m=case["m"], k=case["k"], nev=case["nev"], rtol=case["rtol"],
                       ncyc=case["ncyc"])
    x.backward(st["grad"])
    return {"x": x.detach(), "dkappa": kappa.grad, "db": b.grad}


# ------------------------------------------------------------------------------- what a pass needs
def _sizes(case):
    N, kind = case["N"], case["kind"]
    d = {"u1_4d": 4, "cd3d": 3}.get(kind, 2)
    Nc = N // 2 if kind == "u1_4d" else (N - 1) // 2
    return N ** d, Nc ** d, 16 if kind == "u1_4d" else 8, {"u1_4d": 66, "cd3d": 14}.get(kind, 10)


def _gmresdr_flops(nc, m, k, cycles, per_op, cplx):
    """Arnoldi with two Gram-Schmidt passes (4 multiply-adds per basis entry), the operator, the
    restart recombinations."""
    f = 4 if cplx else 1
    steps = sum(8 * f * (j + 1) + per_op for j in range(m))
    steps += (cycles - 1) * (sum(8 * f * (j + 1) + per_op for j in range(k, m)) + 2 * f * (m + 1) * (k + 1))
    return float(nc) * steps


def _factor_flops(n, k, per_op, cplx):
    """A Y, and CholQR2: two symmetric Gram products and two triangular products."""
    return float(n) * (k * per_op + (4 if cplx else 1) * 4 * k * (k + 1))


def work(case):
    """Inputs read once and outputs written once; flops of the method: a solve is counted with
    the products it needs on these operators, about 1.3 N (2D) and 1.6 N (3D) with deflation."""
    op = case["op"]
    if op == "batch":
        Ns, _ = _batch_sizes(case, 0)
        n = sum(v * v for v in Ns)
        nc = sum(((v - 1) // 2) ** 2 for v in Ns)
        its = sum(v * v * 1.3 * v * (10 + 19) for v in Ns)
        return {"bytes": 2 * 8.0 * 8 * n,
                "flops": _gmresdr_flops(nc, case["m"], case["k"], case["cycles"], 10, False)
                + _factor_flops(n, case["k"], 10, False) + 8.0 * its}
    n, nc, es, per = _sizes(case)
    cplx = case["kind"] == "u1_4d"
    prods = (1.6 if case["kind"] == "cd3d" else 1.3) * case["N"]
    if op == "phase1":
        return {"bytes": float(es) * (3 * n + nc),
                "flops": _gmresdr_flops(nc, case["m"], case["k"], case["cycles"], per, cplx)
                + _factor_flops(n, case["k"], per, cplx) + (4 if cplx else 1) * 6.0 * case["k"] * n}
    if op == "solve":
        vec = {"bicgstab": 19, "idr": 30, "gmres": 8 * 10}[case["method"]]
        return {"bytes": 8.0 * n * (2 + 3 * case["k"]), "flops": n * prods * (per + vec)}
    if op == "twogrid":
        return {"bytes": 8.0 * 2 * n, "flops": _gmresdr_flops(nc, case["m"], case["k"], case["cycles"], per, False)
                + _factor_flops(n, case["k"], per, False) + n * prods * (per + 19)}
    if op == "basis":
        return {"bytes": 8.0 * 3 * case["k"] * n, "flops": _factor_flops(n, case["k"], per, False)}
    return {"bytes": 8.0 * 6 * n, "flops": 2 * (n * 2 * prods * (per + 19) + _factor_flops(n, case["k"], per, False))}


# ------------------------------------------------------------------------------- the same in plain float64
def _lap_apply(u, N, dim, beta):
    """Centred differences of -Lap u + beta . grad u on the unit square or cube, u (N, ..., N), x last."""
    h = 1.0 / (N + 1)
    y = (2.0 * dim / h ** 2) * u
    for a in range(dim):
        ax = dim - 1 - a
        lo = torch.narrow(u, ax, 0, N - 1)
        hi = torch.narrow(u, ax, 1, N - 1)
        torch.narrow(y, ax, 1, N - 1).add_(lo, alpha=-1.0 / h ** 2 - beta[a] / (2 * h))
        torch.narrow(y, ax, 0, N - 1).add_(hi, alpha=-1.0 / h ** 2 + beta[a] / (2 * h))
    return y


def _sine_solve(b, N, dim, beta):
    """x = A^-1 b through the closed-form eigenvectors (b: (..., N, ..., N), x last)."""
    h = 1.0 / (N + 1)
    t = torch.arange(1, N + 1, dtype=torch.float64, device=b.device)
    S = math.sqrt(2.0 * h) * torch.sin(math.pi * h * t[:, None] * t[None, :])
    lam, scale = 0.0, []
    for a in range(dim):
        lo, hi = -1.0 / h ** 2 - beta[a] / (2 * h), -1.0 / h ** 2 + beta[a] / (2 * h)
        shape = [1] * dim
        shape[dim - 1 - a] = N
        lam = lam + (2.0 / h ** 2 - 2.0 * math.sqrt(lo * hi) * torch.cos(math.pi * h * t)).reshape(shape)
        scale.append(((lo / hi) ** (t / 2)).reshape(shape))
    x = b.clone()
    for s in scale:
        x = x / s
    for _ in range(2):
        for a in range(dim):
            x = torch.movedim(torch.movedim(x, -1 - a, -1) @ S, -1, -1 - a)
        if _ == 0:
            x = x / lam
    for s in scale:
        x = x * s
    return x


def _block_solve(coef, b, N):
    """Direct solve of a 5-point system (coef: diag, west, east, south, north, each (N, N), y first)
    by block elimination over the rows of the grid; b (N, N, r)."""
    def line(j):
        return torch.diag(coef[0][j]) + torch.diag(coef[1][j, 1:], -1) + torch.diag(coef[2][j, :-1], 1)
    G, z = [], []
    for j in range(N):
        T, r = line(j), b[j]
        if j:
            T = T + coef[3][j][:, None] * G[-1]
            r = r - coef[3][j][:, None] * z[-1]
        s = torch.linalg.solve(T, torch.cat([torch.diag(-coef[4][j]), r], 1))
        G.append(s[:, :N])
        z.append(s[:, N:])
    x = [None] * N
    x[N - 1] = z[N - 1]
    for j in range(N - 2, -1, -1):
        x[j] = z[j] + G[j] @ x[j + 1]
    return torch.stack(x)


def _exp2d_coefs(N):
    h = 1.0 / (N + 1)
    t = torch.arange(1, N + 1, dtype=torch.float64, device="cuda") * h
    a = torch.exp(EXP2D[2] * t[None, :] * t[:, None]) / h ** 2
    cx, cy = EXP2D[0] / (2 * h), EXP2D[1] / (2 * h)
    return [4 * a, -a - cx, -a + cx, -a - cy, -a + cy]


def _vark_coefs(kappa, N, sgn):
    h = 1.0 / (N + 1)
    K = kappa.view(N + 2, N + 2)
    c = K[1:-1, 1:-1]
    w, e = (0.5 / h ** 2 * (c + K[1:-1, :-2]), 0.5 / h ** 2 * (c + K[1:-1, 2:]))
    s, n = (0.5 / h ** 2 * (c + K[:-2, 1:-1]), 0.5 / h ** 2 * (c + K[2:, 1:-1]))
    cb = sgn * 1.0 / (2 * h)
    return [w + e + s + n, -w - cb, -e + cb, -s, -n]


def _interp1(Nc):
    P = torch.zeros(2 * Nc + 1, Nc, dtype=torch.float64, device="cuda")
    for I in range(Nc):
        P[2 * I + 1, I] = 1.0
        P[2 * I, I] = P[2 * I + 2, I] = 0.5
    return P


def _plain_level(case, st_links, mass, fine):
    """(apply, prolong, restrict) of the plain float64 / complex128 problem, on flat vectors."""
    N = case["N"]
    if case["kind"] != "u1_4d":
        dim = 3 if case["kind"] == "cd3d" else 2
        beta = tuple(_beta(case["kind"])) + (0.0,) * 2
        Nc = (N - 1) // 2
        P = _interp1(Nc)

        def axes(v, M):
            for a in range(dim):
                v = torch.movedim(torch.movedim(v, -1 - a, -1) @ M.T, -1, -1 - a)
            return v.reshape(-1)
        return (lambda v: _lap_apply(v.view((N,) * dim), N, dim, beta).reshape(-1),
                lambda v: _lap_apply(v.view((Nc,) * dim), Nc, dim, beta).reshape(-1),
                lambda v: axes(v.view((Nc,) * dim), P), lambda v: axes(v.view((N,) * dim), P.T) / 2 ** dim)
    L, Lc = N, N // 2
    site = torch.arange(L ** 4, device="cuda")
    c = [(site // L ** a) % L for a in range(4)]
    y = [v - v % 2 for v in c]
    W = torch.ones(L ** 4, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        odd = c[mu] % 2 == 1
        at = y[0] + L * (y[1] + L * (y[2] + L * y[3]))
        W = torch.where(odd, W * st_links[mu][at], W)
        y[mu] = c[mu]
    w = 0.25 * W.conj()
    X = (c[0] // 2) + Lc * ((c[1] // 2) + Lc * ((c[2] // 2) + Lc * (c[3] // 2)))

    def pro(v):
        return w * v[X]

    def res(v):
        t = w.conj() * v
        out = torch.zeros(Lc ** 4, 2, dtype=torch.float64, device="cuda")
        return torch.view_as_complex(out.index_add_(0, X, torch.view_as_real(t)))

    def app(v):
        return (mass + 8.0) * v - _hops(st_links, v, L)
    return app, lambda v: res(app(pro(v))), pro, res


def _plain_phase1(case, seed):
    """GMRES-DR(m, k) for the case's cycles with full matrices, then the projection, in plain torch."""
    m, k = case["m"], case["k"]
    links = mass = None
    if case["kind"] == "u1_4d":
        links = _links(seed, case["N"])
        mass = _lattice_mass(links, case["N"], seed)
    Af, Ac, pro, res = _plain_level(case, links, mass, True)
    n, nc, _, _ = _sizes(case)
    b = res(_vector(case, seed, 10, n))
    cplx = b.is_complex()
    V = torch.zeros(m + 1, nc, dtype=b.dtype, device="cuda")
    nb = torch.linalg.vector_norm(b)
    V[0] = b / nb
    H = np.zeros((m + 1, m), dtype=complex if cplx else float)
    c = np.zeros(m + 1, dtype=H.dtype)
    c[0] = float(nb)
    xc, j0 = torch.zeros_like(b), 0

    def to(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    for cyc in range(case["cycles"]):
        for j in range(j0, m):
            w = Ac(V[j])
            for _ in range(2):
                hj = V[:j + 1].conj() @ w
                w = w - hj @ V[:j + 1]
                H[:j + 1, j] += hj.cpu().numpy()
            H[j + 1, j] = float(torch.linalg.vector_norm(w))
            V[j + 1] = w / H[j + 1, j].real
        d = np.linalg.lstsq(H, c, rcond=None)[0]
        rs = c - H @ d
        xc = xc + to(d) @ V[:m]
        f = np.linalg.solve(H[:m].conj().T, np.eye(m)[:, m - 1])
        h2 = abs(H[m, m - 1]) ** 2
        M = H[:m].copy()
        M[:, m - 1] += h2 * f
        th, G = np.linalg.eig(M)
        order = sorted(range(m), key=lambda i: (abs(th[i]), th[i].real, 0 if th[i].imag >= 0 else 1))
        kk = k
        if not cplx and th[order[k - 1]].imag > 0:
            kk = k + 1
        cols = []
        for i in order[:kk]:
            if cplx:
                cols.append(G[:, i])
            elif th[i].imag == 0:
                cols.append(G[:, i].real)
            elif th[i].imag > 0:
                cols += [G[:, i].real, G[:, i].imag]
        Pk = np.linalg.qr(np.stack(cols, 1))[0]
        z = np.concatenate([-h2 * f, [H[m, m - 1]]])
        P1 = np.linalg.qr(np.concatenate([np.concatenate([Pk, np.zeros((1, kk))]), z[:, None]], 1))[0]
        if cyc == case["cycles"] - 1:
            Y = to(Pk).T @ V[:m]
            break
        Hn = P1.conj().T @ H @ P1[:m, :kk]
        V[:kk + 1] = to(P1).T @ V
        # the restart direction once more against the kept span, as rounding leaves it
        V[kk] -= (V[:kk].conj() @ V[kk]) @ V[:kk]
        V[kk] /= torch.linalg.vector_norm(V[kk])
        H[:] = 0
        H[:kk + 1, :kk] = Hn
        c = np.concatenate([P1.conj().T @ rs, np.zeros(m - kk)])
        j0 = kk
    del V
    Yf = torch.stack([pro(v) for v in Y], 1)
    AY = torch.stack([Af(Yf[:, i]) for i in range(Yf.shape[1])], 1)
    x = pro(xc)
    r = _vector(case, seed, 10, n) - Af(x)
    Q, R = torch.linalg.qr(AY)
    q = Q.mH @ r
    x = x + Yf @ torch.linalg.solve_triangular(R, q[:, None], upper=True)[:, 0]
    return {"xc": xc, "x": x, "r": r - Q @ q}


def exact(case, seed):
    op, kind = case["op"], case.get("kind")
    if op == "batch":
        Ns, betas = _batch_sizes(case, seed)
        rhs = _randn(seed, 10, 8 * sum(v * v for v in Ns))
        out, at = [], 0
        for N, b in zip(Ns, betas):
            r = rhs[at:at + 8 * N * N].view(N, N, 8).permute(2, 0, 1)
            out.append(_sine_solve(r, N, 2, (b, 0.0)).permute(1, 2, 0).reshape(-1))
            at += 8 * N * N
        return {"x": torch.cat(out)}
    N = case["N"]
    n = _sizes(case)[0]
    if op == "adjoint":
        kappa, g = _kappa(seed, N), _randn(seed, 12, N * N)
        x = _block_solve(_vark_coefs(kappa, N, 1), _randn(seed, 10, n).view(N, N, 1), N)[..., 0]
        lam = _block_solve(_vark_coefs(kappa, N, -1), g.view(N, N, 1), N)[..., 0]
        X, Lm = (torch.nn.functional.pad(v, (1, 1, 1, 1)) for v in (x, lam))
        s = -0.5 * (N + 1) ** 2
        dk = torch.zeros_like(X)
        fx = s * (Lm[:, 1:] - Lm[:, :-1]) * (X[:, 1:] - X[:, :-1])
        fy = s * (Lm[1:] - Lm[:-1]) * (X[1:] - X[:-1])
        dk[:, 1:] += fx
        dk[:, :-1] += fx
        dk[1:] += fy
        dk[:-1] += fy
        return {"x": x.reshape(-1), "dkappa": dk.reshape(-1), "db": lam.reshape(-1)}
    if op == "phase1":
        return _plain_phase1(case, seed)
    if op == "basis":
        A = _operator(case, seed)
        Y = A.prolong(_modes(kind, N, case["k"]))          # an input of the case, made as in prepare()
        Y = (Y + 1e-3 * _randn(seed, 16, Y.numel()) * (torch.linalg.vector_norm(Y) / math.sqrt(Y.numel()))).view(-1, n)
        dim = 3 if kind == "cd3d" else 2
        beta = tuple(_beta(kind)) + (0.0,) * 2
        AY = torch.stack([_lap_apply(v.view((N,) * dim), N, dim, beta).reshape(-1) for v in Y])
        # Cholesky QR three times: orthonormal to rounding
        Q, R = AY, torch.eye(case["k"], dtype=torch.float64, device="cuda")
        for _ in range(3):
            C = torch.linalg.cholesky(Q @ Q.T)
            Q = torch.linalg.solve_triangular(C, Q, upper=False)
            R = C.T @ R
        return {"Q": Q, "AY": AY, "R": R.T.contiguous()}
    b = _vector(case, seed, 10, n)
    if kind == "exp2d":
        return {"x": _block_solve(_exp2d_coefs(N), b.view(N, N, 1), N).reshape(-1)}
    dim = 3 if kind == "cd3d" else 2
    return {"x": _sine_solve(b.view((N,) * dim), N, dim, tuple(_beta(kind)) + (0.0,) * 2).reshape(-1)}
