"""A one-launch cycle whose barrier wait is given up: the launch ends by itself, the solve reports it,
and the operator solves as before afterwards."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(A, b, how):
    x = torch.zeros_like(b)
    if how.startswith("idr"):
        g = torch.Generator(device="cuda").manual_seed(2)
        P = torch.randn(4, A.n, dtype=torch.float64, device="cuda", generator=g)
        status, st = A.solve_idr(b, x, P, None, rtol=1e-10, ncyc=10,
                                 precision="f32_ir" if how == "idr_f32" else "f64")
    else:
        status, st = A.solve(b, x, None, precision=how, rtol=1e-10, ncyc=10, restart_mvps=0)
    return status, x, st[0]


@pytest.mark.parametrize("how", ["f64", "f32_ir", "idr", "idr_f32"])
def test_a_wait_that_runs_out_is_reported(how):
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd2d", 127, (2.0, 1.0))
    b = torch.randn(A.n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    status, x0, st0 = _solve(A, b, how)
    assert status == tg.TG_OK
    A.sync_limits(step=0)
    for _ in range(3):
        try:
            status = _solve(A, b, how)[0]
        except tg.TgError as e:
            status = e.status
        assert status == tg.TG_SYNC_TIMEOUT
    A.sync_limits()
    status, x, st = _solve(A, b, how)
    assert status == tg.TG_OK and st["mvps"] == st0["mvps"]
    assert torch.equal(x, x0)


def test_limits_are_checked():
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd2d", 15, (1.0,))
    for bad in ((-1, 1, 1), (1, -1, 1), (1, 1, -1)):
        with pytest.raises(tg.TgError) as e:
            A.sync_limits(*bad)
        assert e.value.status == tg.TG_BAD_ARG
