"""Tensor-core split products (Out = In S and A^H B) through the deflation set-up, at the sizes
where they can go wrong: the row counts around the first split size and around whole tiles,
column counts around the 8-, 16- and 32-column blocks, rows of very different magnitude.

Tolerances, with eps = 2^-53: Q is orthonormal to 1e-13 as in the other set-up tests; the
factors reproduce A Y, and V^H A V the matrix H, to 64 eps of their norms (sums of at most 256
terms rounded once or, in the small products R = R2 R1, per term)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _setup(kind, N, k, proj, scale=None, seed=0):
    from paper_2005_03070_gb300 import tg
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if kind == "u1_4d":
        th = 6.28 * torch.rand(4, N ** 4, dtype=torch.float64, device="cuda", generator=g)
        A = tg.Operator(kind, N, links=torch.polar(torch.ones_like(th), th), mass=0.3)
        Y = torch.complex(*(torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g) for _ in range(2)))
    else:
        A = tg.Operator(kind, N, (2.0, 1.0, 0.5))
        Y = torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g)
    if scale is not None:
        Y = Y * scale(A.n)
    d = A.defl_from_basis(Y.contiguous(), k, proj=proj)
    return [d.copy(w) for w in range(4)]


# 63^2 = 3969 rows stay below the split, 65^2 = 4225 are above it with a partial tile, 127^2 has
# one row more than whole tiles, 8^4 whole tiles only
@pytest.mark.parametrize("kind,N", [("cd2d", 63), ("cd2d", 65), ("cd2d", 127), ("cd3d", 17), ("u1_4d", 8), ("u1_4d", 10)])
@pytest.mark.parametrize("k", [1, 4, 5, 8, 16, 17, 32, 33, 41, 70])
def test_cholqr2(kind, N, k):
    Y, Q, AY, R = _setup(kind, N, k, "minres")
    G = (Q.conj() @ Q.T).cpu().numpy()
    assert np.abs(G - np.eye(k)).max() <= 1e-13
    d = (R @ Q - AY).norm() / AY.norm()
    assert d.item() <= 64 * EPS


@pytest.mark.parametrize("kind,N,k", [("cd2d", 65, 7), ("cd3d", 17, 33), ("u1_4d", 8, 19), ("cd2d", 129, 130)])
def test_galerkin(kind, N, k):
    from paper_2005_03070_gb300 import tg
    Y, V, AY, H = _setup(kind, N, k, "galerkin")
    # A V = A Y (V^H Y)^-1 in the basis V of Y; H is stored transposed
    C = V.conj() @ Y.T
    AV = torch.linalg.solve(C.T, AY)
    want = (V.conj() @ AV.T).T
    cond = torch.linalg.cond(C).item()
    assert ((H - want).norm() / want.norm()).item() <= 64 * EPS * max(1.0, cond)


def test_row_magnitudes():
    """Rows scaled by 2^-200 .. 2^200 go through the row exponents, an infinity through plain
    float64: the set-up reports it as before."""
    from paper_2005_03070_gb300 import tg
    g = torch.Generator(device="cuda")
    g.manual_seed(3)

    def scale(n):
        return torch.exp2(torch.randint(-200, 201, (1, n), device="cuda", generator=g).double())
    Y, Q, AY, R = _setup("cd2d", 127, 12, "minres", scale)
    assert torch.isfinite(Q).all()
    # the largest rows carry the norm: the factors reproduce A Y relative to its rows
    rel = ((R @ Q - AY).abs().amax(0) / AY.abs().amax(0).clamp_min(1e-300))
    assert (R @ Q - AY).norm() / AY.norm() <= 64 * EPS
    assert torch.isfinite(rel).all()
    Y[3, 777] = float("inf")
    A = tg.Operator("cd2d", 127, (2.0, 1.0, 0.5))
    with pytest.raises(tg.TgError):
        A.defl_from_basis(Y.contiguous(), 12)
