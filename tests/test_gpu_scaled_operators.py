"""The coarse phase and GMRES on operators of any size: with A scaled by a power of two every step
scales exactly (orthogonalisation, the small problems and their tests are relative), so the
solution comes out scaled by its inverse and the basis the same, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _op(N, e):
    from paper_2005_03070_gb300 import tg
    g = torch.Generator(device="cuda").manual_seed(N)
    kappa = torch.exp(0.3 * torch.randn((N + 2) ** 2, dtype=torch.float64, device="cuda", generator=g))
    A = tg.Operator("vark2d", N, (0.0,), kappa=kappa * 2.0 ** e)
    return A, torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g)


def _coarse(N, e, m, k, precision, cycles=4):
    A, b = _op(N, e)
    xc, d, st, _ = A.coarse_gmresdr(b, m, k, rtolev=1e-8, rtol=1e-12, max_cycles=cycles, precision=precision)
    return xc * 2.0 ** e, d.copy(0), st["coarse_mvps"], st["cycles"]


def _same(got, want):
    assert got[2:] == want[2:]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("N,m,k", [(31, 24, 8), (127, 30, 15), (255, 40, 12)])
@pytest.mark.parametrize("e", [-200, -60, 60, 200])
def test_coarse_f64(N, m, k, e):
    _same(_coarse(N, e, m, k, "f64"), _coarse(N, 0, m, k, "f64"))


@pytest.mark.parametrize("N,m,k", [(31, 24, 8), (33, 20, 7), (127, 30, 15), (255, 40, 12)])
@pytest.mark.parametrize("e", [-60, -30, 30, 60])
def test_coarse_f32(N, m, k, e):
    """The float32 basis: values of A, about 2^17 at most, stay within 2^-80 .. 2^80."""
    _same(_coarse(N, e, m, k, "f32_ir"), _coarse(N, 0, m, k, "f32_ir"))


@pytest.mark.parametrize("N,m", [(31, 24), (127, 30)])
@pytest.mark.parametrize("e", [-340, 340])
def test_coarse_far(N, m, e):
    """Norms whose cube leaves the float64 range.  Squares of squares do too, so that the small problems
    rescale by other numbers than powers of two: one cycle, whose solution is compared to 1e-9 as in
    the other one-cycle tests."""
    got, want = _coarse(N, e, m, 8, "f64", 1), _coarse(N, 0, m, 8, "f64", 1)
    assert got[2:] == want[2:]
    assert ((got[0] - want[0]).norm() / want[0].norm()).item() <= 1e-9


@pytest.mark.parametrize("N", [33, 127])
@pytest.mark.parametrize("e", [-200, 200])
def test_gmres(N, e):
    out = []
    for s in (e, 0):
        A, b = _op(N, s)
        x = torch.zeros_like(b)
        status, st = A.solve(b, x, None, method="gmres", rtol=1e-6, m3=30, max_mvps=300)
        out.append((x * 2.0 ** s, x, status, st[0]["mvps"]))
    assert out[0][2:] == out[1][2:]
    assert torch.equal(out[0][0], out[1][0])
