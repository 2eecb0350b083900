"""Small solves on several threads at once, an operator and a stream each: every solution meets its
tolerance, recomputed with the operator (rounding below 1e-13), every time."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [2, 6])
@pytest.mark.parametrize("how", ["f64", "f32_ir", "idr", "mixed"])
def test_solves_side_by_side(threads, how):
    from paper_2005_03070_gb300 import tg
    hows = ["f64", "f32_ir", "idr"]
    jobs = []
    for t in range(threads):
        kind, N = [("cd2d", 63), ("cd3d", 31), ("cd2d", 127)][t % 3]
        A = tg.Operator(kind, N, (2.0, 1.0, 0.5))
        g = torch.Generator(device="cuda").manual_seed(t)
        jobs.append((A, torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g),
                     torch.randn(3, A.n, dtype=torch.float64, device="cuda", generator=g),
                     torch.zeros(4, A.n, dtype=torch.float64, device="cuda"), torch.cuda.Stream(),
                     hows[t % 3] if how == "mixed" else how))
    torch.cuda.synchronize()
    status = []
    bar = threading.Barrier(threads)

    def work(A, b, P, X, s, h):
        bar.wait()
        for i in range(len(X)):
            if h == "idr":
                status.append(A.solve_idr(b, X[i], P, None, rtol=1e-10, ncyc=10, stream=s)[0])
            else:
                status.append(A.solve(b, X[i], None, precision=h, rtol=1e-10, ncyc=10, restart_mvps=0, stream=s)[0])
    pool = [threading.Thread(target=work, args=j) for j in jobs]
    for th in pool:
        th.start()
    for th in pool:
        th.join()
    torch.cuda.synchronize()
    assert status == [0] * (threads * 4)
    for A, b, _, X, _, _ in jobs:
        for x in X:
            assert ((b - A.apply(x)).norm() / b.norm()).item() <= 1.001e-10
