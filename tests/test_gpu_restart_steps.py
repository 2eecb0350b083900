"""The restart kernel's least-squares, Hessenberg, eigenvector and Gram-Schmidt steps at the sizes
where their splits change (one or two columns, 32 and 33 rows, reflectors of two rows and of the
full block a restart leaves, real and complex) and on badly scaled matrices.

The matrices have the diagonal 1 .. m in random order and random entries of size 1 / sqrt(m)
elsewhere: eigenvectors of condition below 1e3 (computed for every case here), so float64 rounding
of the largest value moves values by at most 1e-12 of it and an invariant subspace's residual by no
more; the bounds are 1e-10."""
import numpy as np
import pytest

from oracle.gmresdr import harmonic_ritz as o_hritz, order_ritz, select_k

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hbar(m, k, cx, full, seed):
    g = np.random.default_rng(seed)
    H = g.standard_normal((m + 1, m))
    if cx:
        H = H + 1j * g.standard_normal((m + 1, m))
    keep = np.triu(np.ones((m + 1, m), dtype=bool), -1)
    if full:
        keep[:k + 1, :k] = True
    H = np.where(keep, H, 0.0) / np.sqrt(m)
    H[np.arange(m), np.arange(m)] = 1.0 + g.permutation(m)
    return H


@pytest.mark.parametrize("m,k", [(2, 1), (3, 1), (3, 2), (5, 4), (31, 16), (32, 8), (33, 32), (64, 33), (65, 20), (97, 48)])
@pytest.mark.parametrize("cx", [False, True])
@pytest.mark.parametrize("full,scale", [(False, 1.0), (True, 1.0), (True, 1e140), (True, 1e-140)])
def test_pairs(m, k, cx, full, scale):
    from paper_2005_03070_gb300 import tg
    H = _hbar(m, k, cx, full, 7 * m + k)
    th, basis, eres = tg.harmonic_ritz(torch.from_numpy((scale * H).T.copy()).cuda(), m, k, complex_=cx)
    th, basis = th.cpu().numpy() / scale, basis.cpu().numpy().T
    theta, G = o_hritz(H)
    idx = order_ritz(theta)
    # compared as sets: values of equal modulus may swap places
    d = np.abs(th[:, None] - theta[None, :])
    assert max(d.min(0).max(), d.min(1).max()) <= 1e-10 * np.abs(theta).max()
    n = basis.shape[1]
    assert n in (k, k + 1)
    assert np.max(np.abs(basis.conj().T @ basis - np.eye(n))) <= 1e-12
    # an invariant subspace of the harmonic matrix M: M B = B (B^H M B)
    Hm = H[:m]
    f = np.linalg.solve(Hm.conj().T, np.eye(m)[:, -1])
    M = Hm.astype(H.dtype).copy()
    M[:, -1] += abs(H[m, m - 1]) ** 2 * f
    B = basis[:m]
    assert np.linalg.norm(M @ B - B @ (B.conj().T @ (M @ B))) <= 1e-10 * np.linalg.norm(M)
