"""Solves whose one-launch cycles cannot start: because the blocks' first wait runs out, because
another stream's kernel holds SMs for longer than the solve takes, and because the caller's stream
owns fewer SMs than the launch has blocks.  Each then runs as a chain of launches and solves as
before.  A relative residual of 1e-10 is asked for and recomputed with the operator, whose rounding
is below 1e-13."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HOW = ["f64", "f32_ir", "idr", "idr_f32"]


def _problem(N=127, kind="cd2d"):
    from paper_2005_03070_gb300 import tg
    A = tg.Operator(kind, N, (2.0, 1.0, 0.5))
    g = torch.Generator(device="cuda").manual_seed(1)
    return A, torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g)


def _solve(A, b, how, defl=None, stream=None):
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    if how.startswith("idr"):
        P = torch.randn(4, A.n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
        torch.cuda.synchronize()
        status, st = A.solve_idr(b, x, P, defl, rtol=1e-10, ncyc=10, stream=stream,
                                 precision="f32_ir" if how == "idr_f32" else "f64")
    else:
        status, st = A.solve(b, x, defl, precision=how, rtol=1e-10, ncyc=10, restart_mvps=0, stream=stream)
    return status, x, st[0]


def _solved(A, b, status, x):
    torch.cuda.synchronize()
    assert status == 0
    assert ((b - A.apply(x)).norm() / b.norm()).item() <= 1.001e-10


@pytest.mark.parametrize("kind,N", [("cd2d", 127), ("cd3d", 31)])
@pytest.mark.parametrize("how", HOW)
@pytest.mark.parametrize("k", [0, 12])
def test_first_wait_runs_out(kind, N, how, k):
    A, b = _problem(N, kind)
    defl = None
    if k:
        g = torch.Generator(device="cuda").manual_seed(3)
        defl = A.defl_from_basis(torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g), k,
                                 precision="f32_ir" if "f32" in how else "f64")
    A.sync_limits(start=0)
    _solved(A, b, *_solve(A, b, how, defl)[:2])
    A.sync_limits()
    _solved(A, b, *_solve(A, b, how, defl)[:2])


def _classes(f):
    """Launches per class of the profile that f() adds."""
    from paper_2005_03070_gb300 import tg
    def read():
        return {k: v["launches"] for k, v in tg.tg_profile_read().items() if isinstance(v, dict)}
    tg.tg_profile_enable(True)
    try:
        before = read()
        f()
        after = read()
    finally:
        tg.tg_profile_enable(False)
    return {k: v - before.get(k, 0) for k, v in after.items()}


@pytest.mark.parametrize("method,precision", [("bicgstab", "f64"), ("bicgstab", "f32_ir"), ("idr", "f64"), ("idr", "f32_ir")])
@pytest.mark.parametrize("profiled", [False, True])
@pytest.mark.parametrize("k", [0, 8])
def test_a_later_launch_cannot_start(method, precision, profiled, k):
    """The indefinite Helmholtz problem whose cycle takes several launches: the chain takes it over
    after the first.  The residual is the solution's, and the cap on products holds."""
    from paper_2005_03070_gb300 import tg
    A = tg.Operator("cd2d", 63, (0.0,), mass=-2500.0)
    g = torch.Generator(device="cuda").manual_seed(4)
    b = torch.randn(A.n, dtype=torch.float64, device="cuda", generator=g)
    P = torch.randn(2, A.n, dtype=torch.float64, device="cuda", generator=g)
    defl = A.defl_from_basis(torch.randn(k, A.n, dtype=torch.float64, device="cuda", generator=g), k,
                             precision=precision) if k else None
    x = torch.zeros_like(b)
    cap = 5999
    A.sync_limits(again=0)
    out = []

    def run():
        if method == "idr":
            out.append(A.solve_idr(b, x, P, defl, rtol=1e-15, ncyc=0, restart_mvps=cap, max_mvps=cap, precision=precision))
        else:
            out.append(A.solve(b, x, defl, precision=precision, rtol=1e-15, ncyc=0, restart_mvps=cap, max_mvps=cap))
    if profiled:
        n = _classes(run)
        if precision == "f64":
            # the first launch and the one that gave up; the cycle went on and did not start again
            assert n["idr_cycle" if method == "idr" else "bicg_cycle"] == 2
            assert n.get("bicg_init", 0) == 0
            assert n["idr_apply" if method == "idr" else "bicg_x"] > 0
    else:
        run()
    status, st = out[0]
    assert status in (tg.TG_OK, tg.TG_NOT_CONVERGED, tg.TG_BREAKDOWN)
    rel = ((b - A.apply(x)).norm() / b.norm()).item()
    assert st[0]["mvps"] <= cap + 3
    assert abs(rel - st[0]["relres"]) <= 1e-12 * max(1.0, rel)


@pytest.mark.parametrize("kind,N", [("cd2d", 127), ("cd3d", 31)])
@pytest.mark.parametrize("precision", ["f64", "f32_ir"])
def test_idr_taken_over_converges(kind, N, precision):
    """A cycle of more than 64 rounds with one shadow column, taken over after its first launch."""
    A, b = _problem(N, kind)
    P = torch.randn(1, A.n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
    A.sync_limits(again=0)
    x = torch.zeros_like(b)
    status, st = A.solve_idr(b, x, P, None, rtol=1e-10, ncyc=1, precision=precision)
    assert st[0]["mvps"] > 2 * 64
    _solved(A, b, status, x)


@pytest.mark.parametrize("how", HOW)
def test_beside_a_long_kernel(how):
    """A kernel of about two seconds on another stream."""
    A, b = _problem()
    _solved(A, b, *_solve(A, b, how)[:2])
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    x = torch.zeros_like(b)
    P = torch.randn(4, A.n, dtype=torch.float64, device="cuda")
    mine = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(4_000_000_000)
    if how.startswith("idr"):
        status, _ = A.solve_idr(b, x, P, None, rtol=1e-10, ncyc=10, stream=mine,
                                precision="f32_ir" if how == "idr_f32" else "f64")
    else:
        status, _ = A.solve(b, x, None, precision=how, rtol=1e-10, ncyc=10, restart_mvps=0, stream=mine)
    _solved(A, b, status, x)


GREEN = r'''
#include <cuda.h>
static CUgreenCtx ctx;
extern "C" int green_stream(int sms, void **stream) {
    CUdevice dev;
    CUdevResource all, part, rest;
    CUdevResourceDesc desc;
    unsigned groups = 1;
    CUstream s;
    if (cuCtxGetDevice(&dev)) return 1;
    if (cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM)) return 2;
    if (cuDevSmResourceSplitByCount(&part, &groups, &all, &rest, 0, sms) || groups != 1) return 3;
    if (cuDevResourceGenerateDesc(&desc, &part, 1)) return 4;
    if (cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM)) return 5;
    if (cuGreenCtxStreamCreate(&s, ctx, CU_STREAM_NON_BLOCKING, 0)) return 6;
    *stream = s;
    return 0;
}
extern "C" void green_free(void *stream) {
    cuStreamDestroy((CUstream)stream);
    cuGreenCtxDestroy(ctx);
}
'''


@pytest.fixture(scope="module")
def green(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    torch.zeros(1, device="cuda")
    d = tmp_path_factory.mktemp("green")
    (d / "green.cu").write_text(GREEN)
    p = subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", str(d / "green.cu"), "-o", str(d / "green.so"), "-lcuda"],
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr
    lib = C.CDLL(str(d / "green.so"))
    handle = C.c_void_p()
    rc = lib.green_stream(16, C.byref(handle))
    if rc:
        pytest.skip(f"no stream on a part of the SMs here (step {rc})")
    yield torch.cuda.ExternalStream(handle.value)
    torch.cuda.synchronize()
    lib.green_free(handle)


@pytest.mark.parametrize("how", HOW)
def test_stream_with_few_sms(green, how):
    A, b = _problem()
    _solved(A, b, *_solve(A, b, how, stream=green)[:2])
