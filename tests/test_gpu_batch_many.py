"""A batch of more instances than the partial sums have room for at 16 blocks each.  Every column is
solved to a relative residual of 1e-10, recomputed here with the instance's float64 operator, whose
own rounding is below 1e-13."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_many_instances():
    from paper_2005_03070_gb300 import tg
    count, N = 2100, 63
    n = N * N
    betas = [0.5 + 0.5 * (i % 4) for i in range(count)]
    batch = tg.Batch([N] * count, betas)
    g = torch.Generator(device="cuda").manual_seed(1)
    rhs = torch.randn(batch.total, dtype=torch.float64, device="cuda", generator=g)
    x = torch.zeros_like(rhs)
    status, _ = batch.solve(rhs, x, rtol=1e-10, ncyc=10, restart_mvps=0, threads=4)
    assert status == tg.TG_OK
    A = [tg.Operator("cd2d", N, (b,)) for b in betas[:4]]
    B, X = rhs.view(count, n, 8).permute(0, 2, 1).contiguous(), x.view(count, n, 8).permute(0, 2, 1).contiguous()
    R = torch.empty_like(B)
    for i in range(count):
        for q in range(8):
            R[i, q] = B[i, q] - A[i % 4].apply(X[i, q])
    assert (R.norm(dim=2) / B.norm(dim=2)).max().item() <= 1.001e-10
