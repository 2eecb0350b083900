"""Blocks of a batch in proportion to its instances' points: one instance, instances smaller than
one block beside large ones, and equal ones.  Every column is solved to a relative residual of
1e-10, recomputed here with the instance's float64 operator, whose own rounding is below 1e-13."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns", [[15], [15, 255], [255, 15, 17, 15, 127], [31] * 9, [191, 15] * 3])
@pytest.mark.parametrize("ncyc,restart", [(10, 0), (0, 60)])
def test_uneven_instances(Ns, ncyc, restart):
    from paper_2005_03070_gb300 import tg
    betas = [0.5 + 0.25 * i for i in range(len(Ns))]
    batch = tg.Batch(Ns, betas)
    g = torch.Generator(device="cuda").manual_seed(len(Ns))
    rhs = torch.randn(batch.total, dtype=torch.float64, device="cuda", generator=g)
    batch.setup(rhs, m=20, k=8, rtolev=1e-2, threads=4)
    x = torch.zeros_like(rhs)
    status, stats = batch.solve(rhs, x, rtol=1e-10, ncyc=ncyc, restart_mvps=restart, threads=4)
    assert status == tg.TG_OK
    for i, N in enumerate(Ns):
        A = tg.Operator("cd2d", N, (betas[i],))
        o, n = batch.offsets[i], batch.sizes[i]
        B, X = rhs[o:o + 8 * n].view(n, 8), x[o:o + 8 * n].view(n, 8)
        for q in range(8):
            b = B[:, q].contiguous()
            r = b - A.apply(X[:, q].contiguous())
            assert (r.norm() / b.norm()).item() <= 1.001e-10, (N, q)
