"""The Schur form where nearly every decision is a deflation: triangular matrices, whose values the
deflation search takes off one after the other without a sweep between, alone and with 2 x 2 blocks
of complex pairs among them.

With the last row of Hbar zero the harmonic matrix is H_m itself, and a triangular H_m passes the
Hessenberg reduction unchanged, so real values and the diagonal of complex matrices come back
exactly.  A block [a b; -b a] gives a +- i sqrt(b^2): two roundings, 4 eps of |b| allowed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _values(H, m, cx):
    from paper_2005_03070_gb300 import tg
    th, _, _ = tg.harmonic_ritz(torch.from_numpy(H.T.copy()).cuda(), m, max(1, m // 2), complex_=cx)
    return th.cpu().numpy()


@pytest.mark.parametrize("m", [2, 3, 31, 32, 33, 64, 97])
@pytest.mark.parametrize("cx", [False, True])
def test_triangular(m, cx):
    g = np.random.default_rng(m)
    H = np.zeros((m + 1, m), dtype=complex if cx else float)
    H[:m] = np.triu(g.standard_normal((m, m)), 1)
    d = 1.0 + g.permutation(m)
    if cx:
        H[:m] += 1j * np.triu(g.standard_normal((m, m)), 1)
        d = d * np.exp(0.25j * np.arange(m))
    H[np.arange(m), np.arange(m)] = d
    want = np.sort_complex(np.asarray(d, dtype=complex))
    for _ in range(10):
        assert np.array_equal(np.sort_complex(_values(H, m, cx)), want)


@pytest.mark.parametrize("m", [3, 32, 65])
@pytest.mark.parametrize("start", [0, 1])
def test_pairs_among_single_values(m, start):
    g = np.random.default_rng(m + start)
    H = np.zeros((m + 1, m))
    H[:m] = np.triu(g.standard_normal((m, m)), 1)
    H[np.arange(m), np.arange(m)] = 1.0 + np.arange(m)
    want = (1.0 + np.arange(m)).astype(complex)
    for i in range(start, m - 1, 3):
        a, b = H[i, i], 0.5 + 0.25 * (i % 4)
        H[i + 1, i + 1], H[i, i + 1], H[i + 1, i] = a, b, -b
        want[i], want[i + 1] = a + 1j * b, a - 1j * b
    got = _values(H, m, False)
    dist = np.abs(got[:, None] - want[None, :])
    assert max(dist.min(0).max(), dist.min(1).max()) <= 4 * 2.0 ** -53 * 1.25
