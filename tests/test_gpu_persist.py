"""One-launch BiCGStab and IDR cycles: the smallest grids (fewer points than blocks), the largest
basis their own projection takes and one more, every real operator kind, both projections, a
cycle longer than one launch, and caps.

Solutions are compared with a dense float64 solve of the operator's own columns.  A solve to a
relative residual of 1e-12 differs from it by at most 1e-12 times the condition number, below
1e5 on these grids."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _op(kind, N):
    from paper_2005_03070_gb300 import tg
    if kind == "vark2d":
        g = torch.Generator(device="cuda")
        g.manual_seed(N)
        kappa = torch.exp(torch.randn((N + 2) ** 2, dtype=torch.float64, device="cuda", generator=g) * 0.3)
        return tg.Operator(kind, N, (1.0,), kappa=kappa)
    return tg.Operator(kind, N, {"exp2d": (40.0, 40.0, 5.0)}.get(kind, (2.0, 1.0, 0.5)))


def _dense(A):
    eye = torch.eye(A.n, dtype=torch.float64, device="cuda")
    return torch.stack([A.apply(eye[i].contiguous()) for i in range(A.n)], 1)


@pytest.mark.parametrize("kind,N", [("cd2d", 3), ("cd2d", 5), ("cd2d", 13), ("cd2d", 31), ("vark2d", 17),
                                    ("exp2d", 15), ("cd3d", 3), ("cd3d", 7), ("cd3d", 11)])
@pytest.mark.parametrize("how", ["f64", "f32_ir", "idr", "idr_f32"])
def test_solution(kind, N, how):
    A = _op(kind, N)
    M = _dense(A)
    b = torch.randn(A.n, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    if how.startswith("idr"):
        P = torch.randn(min(4, A.n - 1), A.n, dtype=torch.float64, device="cuda")
        status, st = A.solve_idr(b, x, P, None, rtol=1e-12, ncyc=10, precision="f32_ir" if how == "idr_f32" else "f64")
    else:
        status, st = A.solve(b, x, None, precision=how, rtol=1e-12, ncyc=10, restart_mvps=0)
    ref = torch.linalg.solve(M, b)
    assert status == 0
    assert ((x - ref).norm() / ref.norm()).item() <= 1e-7
    assert abs(((b - M @ x).norm() / b.norm()).item() - st[0]["relres"]) <= 1e-13


@pytest.mark.parametrize("k", [1, 63, 64, 65])
@pytest.mark.parametrize("proj", ["minres", "galerkin"])
@pytest.mark.parametrize("precision", ["f64", "f32_ir"])
def test_projection_columns(k, proj, precision):
    A = _op("cd2d", 25)
    M = _dense(A)
    _, V = torch.linalg.eigh(0.5 * (M + M.T))
    d = A.defl_from_basis(V[:, :k].T.contiguous(), k, proj=proj, precision=precision)
    b = torch.randn(A.n, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    status, st = A.solve(b, x, d, precision=precision, rtol=1e-11, ncyc=0, restart_mvps=40, history=64)
    ref = torch.linalg.solve(M, b)
    assert status == 0 and ((x - ref).norm() / ref.norm()).item() <= 1e-7
    # the first history entry is the residual after the first projection
    r = b.clone()
    d.project(torch.zeros_like(b), r)
    assert abs(st[0]["history"][0][0] - (r.norm() / b.norm()).item()) <= (1e-12 if precision == "f64" else 1e-5)


@pytest.mark.parametrize("method", ["bicgstab", "idr"])
def test_longer_than_one_launch(method):
    """An indefinite Helmholtz problem that does not converge: the product cap ends a cycle that
    takes several launches, and the reported residual is the solution's."""
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd2d", 63, (0.0,), mass=-2500.0)
    b = torch.randn(A.n, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    if method == "idr":
        P = torch.randn(2, A.n, dtype=torch.float64, device="cuda")
        _, st = A.solve_idr(b, x, P, None, rtol=1e-15, ncyc=0, restart_mvps=2999, max_mvps=2999)
    else:
        _, st = A.solve(b, x, None, rtol=1e-15, ncyc=0, restart_mvps=2999, max_mvps=2999)
    rel = ((b - A.apply(x)).norm() / b.norm()).item()
    assert st[0]["mvps"] <= 2999 + 3
    assert abs(rel - st[0]["relres"]) <= 1e-12 * max(1.0, rel)
