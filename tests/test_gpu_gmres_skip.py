"""GMRES cycles that meet their target between two looks of the host: the launches already queued do
no products.  The products of a cycle that ends after 18 to 24 of 64 steps are timed: 33 launches, of
which the reported number may take the time of a product and the others next to none.  At most one
and a half times the reported number of products' time is allowed; all 33 would take 1.4 times that at
least."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_no_products_after_the_target():
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd3d", 191, (2.0, 1.0, 0.5), mass=20000.0)
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g)
    x = torch.zeros_like(b)

    def apply_ms(f):
        tg.tg_profile_enable(True)
        try:
            p0 = tg.tg_profile_read().get("apply", {"launches": 0, "ms": 0.0})
            f()
            p1 = tg.tg_profile_read()["apply"]
        finally:
            tg.tg_profile_enable(False)
        return p1["launches"] - p0["launches"], p1["ms"] - p0["ms"]

    out = []

    def solve(rtol):
        x.zero_()
        out.append(A.solve(b, x, None, method="gmres", rtol=rtol, m3=64, max_mvps=64)[1][0])
    solve(1e-3)
    rtol = None
    for e in range(4, 40):
        solve(10.0 ** (-e / 3.0))
        if 18 <= out[-1]["mvps"] <= 24:
            rtol = 10.0 ** (-e / 3.0)
            break
    assert rtol is not None, [o["mvps"] for o in out]
    y = torch.empty_like(b)
    A.apply(b, y)
    n1, one = apply_ms(lambda: [A.apply(b, y) for _ in range(50)])
    assert n1 == 50
    launches, ms = apply_ms(lambda: solve(rtol))
    mvps = out[-1]["mvps"]
    assert launches >= 33 and 18 <= mvps <= 24
    assert ms <= min(1.5 * mvps, 0.85 * launches) * one / 50
