"""The two-sweep Arnoldi run against the Arnoldi relation, through one coarse GMRES-DR cycle and
GMRES cycles: column counts around the kernels' groups (64 and 128 columns), row counts around
whole chunks, each basis type.

One cycle from v_0 = b_c / ||b_c|| minimises the residual over the Krylov space of dimension m; a
QR of that space in numpy gives the same x_c.  The space's basis is built there by Gram-Schmidt
twice, so both sides differ by rounding times the condition of the least squares, bounded by the
1e-9 (float64) and 2e-3 (float32 basis: eps 6e-8 times a condition below 3e4) used here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(A, b, m):
    """The residual minimiser over K_m(A_c, b_c), with A_c applied by the library (checked against
    the oracle elsewhere)."""
    from paper_2005_03070_gb300 import tg
    bc = A.restrict(b)
    V = torch.zeros(m + 1, A.nc, dtype=bc.dtype, device="cuda")
    V[0] = bc / bc.norm()
    H = np.zeros((m + 1, m), dtype=complex if bc.is_complex() else float)
    for j in range(m):
        w = A.apply(V[j].contiguous(), level=tg.TG_COARSE)
        for _ in range(2):
            h = V[:j + 1].conj() @ w
            w = w - h @ V[:j + 1]
            H[:j + 1, j] += h.cpu().numpy()
        H[j + 1, j] = w.norm().item()
        V[j + 1] = w / H[j + 1, j].real
    rhs = np.zeros(m + 1, dtype=H.dtype)
    rhs[0] = bc.norm().item()
    d = np.linalg.lstsq(H, rhs, rcond=None)[0]
    return torch.from_numpy(d).cuda() @ V[:m]


@pytest.mark.parametrize("kind,N,m", [("cd2d", 31, 20), ("cd2d", 33, 63), ("cd2d", 65, 64), ("cd2d", 127, 65),
                                      ("cd2d", 129, 130), ("cd3d", 33, 30), ("cd3d", 65, 12), ("u1_4d", 8, 40),
                                      ("u1_4d", 12, 66)])
@pytest.mark.parametrize("precision", ["f64", "f32_ir"])
def test_one_cycle(kind, N, m, precision):
    from paper_2005_03070_gb300 import tg
    if kind == "u1_4d" and precision == "f32_ir":
        pytest.skip("the lattice is complex128 only")
    g = torch.Generator(device="cuda")
    g.manual_seed(N + m)
    if kind == "u1_4d":
        th = 6.28 * torch.rand(4, N ** 4, dtype=torch.float64, device="cuda", generator=g)
        A = tg.Operator(kind, N, links=torch.polar(torch.ones_like(th), th), mass=0.3)
        b = torch.complex(*(torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g) for _ in range(2)))
    else:
        A = tg.Operator(kind, N, (2.0, 1.0, 0.5))
        b = torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g)
    xc, _, st, _ = A.coarse_gmresdr(b, m, m // 2 - 1, rtolev=1e-15, rtol=1e-15, max_cycles=1, precision=precision,
                                    want_defl=False)
    ref = _reference(A, b, m)
    assert ((xc - ref).norm() / ref.norm()).item() <= (1e-9 if precision == "f64" else 2e-3)


@pytest.mark.parametrize("N,m3,cap", [(33, 1, 7), (33, 20, 20), (65, 20, 45), (127, 70, 70)])
def test_gmres_cycles(N, m3, cap):
    """GMRES(m3) stopped by the product cap: never more products than the cap, and the residual of
    the last cycle is the recomputed one."""
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd2d", N, (1.0,))
    b = torch.randn(A.n, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    _, st = A.solve(b, x, None, method="gmres", rtol=1e-14, m3=m3, max_mvps=cap)
    assert st[0]["mvps"] == cap
    rel = ((b - A.apply(x)).norm() / b.norm()).item()
    assert abs(rel - st[0]["relres"]) <= 1e-12
    assert rel < 1.0
