"""Deflation set-up from bases whose columns differ in size.

Scaled by powers of two the whole set-up is exact: the Gram matrix, its Cholesky factor and the
products Y R^-1 change only in exponents, so Q (MinRes), V and A V's matrix H (Galerkin) come out
the same bit for bit and A Y and R scaled.  For other scales the factors reproduce every column
of A Y to 64 eps of its own norm, with eps = 2^-53 (sums of at most 70 terms rounded once or, in the
small product R = R2 R1, per term; what a float64 product loses)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _basis(kind, N, k):
    from paper_2005_03070_gb300 import tg
    g = torch.Generator(device="cuda").manual_seed(N + k)
    if kind == "u1_4d":
        th = 6.28 * torch.rand(4, N ** 4, dtype=torch.float64, device="cuda", generator=g)
        A = tg.Operator(kind, N, links=torch.polar(torch.ones_like(th), th), mass=0.3)
        return A, torch.complex(*(torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g) for _ in range(2)))
    A = tg.Operator(kind, N, (2.0, 1.0, 0.5))
    return A, torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g)


CASES = [("cd2d", 63, 9), ("cd2d", 65, 5), ("cd2d", 127, 17), ("cd3d", 17, 41), ("cd3d", 33, 70), ("u1_4d", 8, 6), ("u1_4d", 10, 33)]


@pytest.mark.parametrize("kind,N,k", CASES)
@pytest.mark.parametrize("proj", ["minres", "galerkin"])
@pytest.mark.parametrize("exps", [(0, -20, -40, -70), (0, 300, -300), (-200, 0, 1, 0, 77)])
def test_powers_of_two(kind, N, k, proj, exps):
    A, Y = _basis(kind, N, k)
    s = torch.tensor([2.0 ** exps[i % len(exps)] for i in range(k)], dtype=torch.float64, device="cuda")
    plain = [A.defl_from_basis(Y, k, proj=proj).copy(w) for w in range(4)]
    scaled = [A.defl_from_basis((Y * s[:, None]).contiguous(), k, proj=proj).copy(w) for w in range(4)]
    assert torch.equal(scaled[2], plain[2] * s[:, None])                     # A Y
    assert torch.equal(scaled[1], plain[1])                                  # Q or V
    want = plain[3] * s[:, None] if proj == "minres" else plain[3]           # R (rows: its columns) or H
    assert torch.equal(scaled[3], want)


@pytest.mark.parametrize("kind,N,k", CASES)
@pytest.mark.parametrize("spread", [1e2, 1e5, 1e8, 1e19])
def test_any_scales(kind, N, k, spread):
    A, Y = _basis(kind, N, k)
    g = torch.Generator(device="cuda").manual_seed(k)
    s = spread ** -torch.rand(k, dtype=torch.float64, device="cuda", generator=g)
    s[0], s[-1] = 1.0, 1.0 / spread
    d = A.defl_from_basis((Y * s[:, None]).contiguous(), k)
    Q, AY, R = d.copy(1), d.copy(2), d.copy(3)
    G = Q.conj() @ Q.T
    assert (G - torch.eye(k, device="cuda")).abs().max().item() <= 1e-13
    err = (R @ Q - AY).norm(dim=1) / AY.norm(dim=1)
    assert err.max().item() <= 64 * EPS
