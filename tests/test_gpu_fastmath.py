"""The seeded square root, inverse square root and reciprocal (csrc/tg_fastmath.cuh) over the exponents
that they are used for, against exact values and against CUDA's functions.

With seeds good to s the cubic steps leave 5/2 s^3 (square roots) and s^3 (reciprocal); at
s = 2^-19 that is below 2^-55.  The last rounding adds half an ulp, the rounded product
in sqrt_fast half an ulp more: bounds of 0.75, 0.75 and 1.25 ulp here, of the result's own ulp.  CUDA's
rsqrt is within 1 ulp, its sqrt and division are correctly rounded: at most 2 ulp between them."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "tg_fastmath.cuh"
__global__ void k(const double *x, double *out, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double v = x[i];
        double *o = out + 9 * (size_t)i;
        o[0] = tg::rsqrt_fast(v); o[1] = tg::sqrt_fast(v); o[2] = tg::rcp_fast(v);
        o[3] = rsqrt(v); o[4] = sqrt(v); o[5] = 1.0 / v;
        o[6] = tg::rsqrt_seed(v); o[7] = tg::rcp_seed(v); o[8] = tg::mid_range(v) ? 1.0 : 0.0;
    }
}
extern "C" int run(const void *x, void *out, int n) {
    k<<<256, 256>>>((const double *)x, (double *)out, n);
    return (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fastmath")
    (d / "fm.cu").write_text(SRC)
    p = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                        "-fPIC", "-I" + os.path.join(ROOT, "paper_2005_03070_gb300", "csrc"), str(d / "fm.cu"), "-o",
                        str(d / "fm.so")], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr
    lib = C.CDLL(str(d / "fm.so"))

    def call(x):
        t = torch.from_numpy(x).cuda()
        out = torch.zeros(len(x), 9, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(C.c_void_p(t.data_ptr()), C.c_void_p(out.data_ptr()), C.c_int(len(x))) == 0
        return out.cpu().numpy()
    return call


def _values():
    """Every exponent of the range with random mantissas, and the neighbours of powers of two."""
    g = np.random.default_rng(3)
    e = np.arange(-900, 900)
    x = [np.ldexp(1.0 + g.random(len(e)), e) for _ in range(100)]
    p = np.ldexp(1.0, e)
    x += [p, np.nextafter(p, np.inf), np.nextafter(p[1:], 0.0), np.nextafter(2.0 * p, 0.0), 1.5 * p]
    return np.concatenate(x)


def test_within_their_bounds(run):
    x = _values()
    out = run(x)
    xl = x.astype(np.longdouble)
    exact = [1 / np.sqrt(xl), np.sqrt(xl), 1 / xl]
    for c, (want, bound) in enumerate(zip(exact, (0.75, 1.25, 0.75))):
        ulp = np.spacing(want.astype(np.float64)).astype(np.longdouble)
        assert np.max(np.abs(out[:, c].astype(np.longdouble) - want) / ulp) <= bound
        assert np.max(np.abs(out[:, c] - out[:, 3 + c]) / np.spacing(out[:, 3 + c])) <= 2.0
    for c, want in ((6, exact[0]), (7, exact[2])):
        assert np.max(np.abs(out[:, c].astype(np.longdouble) / want - 1)) <= 2.0 ** -19
    assert np.all(out[:, 8] == 1.0)


def test_range_edges(run):
    lo, hi = 2.0 ** -900, 2.0 ** 900
    inside = np.array([lo, np.nextafter(hi, 0.0), 1.0])
    outside = np.array([np.nextafter(lo, 0.0), hi, 0.0, 5e-324, 1e308, np.inf, np.nan, -1.0, -0.0, -np.inf])
    assert np.all(run(inside)[:, 8] == 1.0)
    assert np.all(run(outside)[:, 8] == 0.0)
