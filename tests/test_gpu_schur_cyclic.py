"""Cyclic shift matrices: every value of modulus 1, shifts that stand still until an exceptional one,
and trailing blocks whose discriminant is real and negative.  Values are the roots of unity; the
matrices are unitary, so that a backward error of a few m eps (m < 80) moves them by less than 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cx", [False, True])
@pytest.mark.parametrize("twist", [0.0, 0.7])
def test_roots_of_unity(cx, twist):
    from paper_2005_03070_gb300 import tg
    if twist and not cx:
        pytest.skip("a phase needs complex arithmetic")
    for m in range(2, 80):
        H = np.roll(np.eye(m + 1, m), 1, 0).astype(complex if cx else float)
        H[0, m - 1] = np.exp(1j * twist) if cx else 1.0
        H[m, m - 1] = 0.0
        th, _, _ = tg.harmonic_ritz(torch.from_numpy(np.ascontiguousarray(H.T)).cuda(), m, max(1, m // 2), complex_=cx)
        want = np.exp(1j * (twist + 2 * np.pi * np.arange(m)) / m)
        d = np.abs(th.cpu().numpy()[:, None] - want[None, :])
        assert max(d.min(0).max(), d.min(1).max()) <= 1e-12, m
