"""The block tables of a batch (csrc/tg_batch.cuh) on the host: for any number and mix of instances
the least candidate of the autotuner is taken, and no table of a candidate that is taken, nor that of
the refinement kernels, has more blocks than the partial sums have room for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include <random>
#include "tg_batch.cuh"
int main() {
    std::mt19937 rng(5);
    long checked = 0, bad = 0;
    auto table = [&](const std::vector<int64_t> &n, int64_t total) {
        const auto map = tg::batch_blocks(n, total);
        ++checked;
        bad += (int64_t)map.size() > tg::batch_room((int64_t)n.size());
        // every block in its instance's run, the runs one after the other
        size_t at = 0;
        for (size_t i = 0; i < n.size(); ++i) {
            const int nb = at < map.size() ? map[at].z : 0;
            bad += nb < 1 || nb > (n[i] + tg::kThreads - 1) / tg::kThreads;
            for (int k = 0; k < nb; ++k) {
                const int4 v = map[at + k];
                bad += v.x != (int)i || v.y != k || v.z != nb || v.w != (int)at;
            }
            at += nb;
        }
        bad += at != map.size();
    };
    for (int64_t count : {1, 2, 6, 9, 31, 128, 500, 1820, 2047, 2048, 2049, 2100, 4096, 16384, 20000}) {
        bad += !tg::batch_fits(8, count);
        for (int mix = 0; mix < 5; ++mix) {
            std::vector<int64_t> n(count);
            for (auto &v : n) {
                const int64_t N = mix == 0 ? 63 : mix == 1 ? 15 : mix == 2 ? 511 : mix == 3 ? 3 + 2 * (rng() % 255)
                                                                               : (rng() % 16 ? 3 : 1023);
                v = N * N;
            }
            for (int64_t gx : {8, 16, 32, 64, 128, 256, 512})
                if (tg::batch_fits(gx, count)) table(n, gx * count);
            table(n, 152 * 8);
        }
    }
    std::printf("%ld %ld\n", checked, bad);
    return bad != 0;
}
'''


def test_tables_fit_their_room(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "batch_blocks_check.cu"
    src.write_text(SRC)
    exe = tmp_path / "batch_blocks_check"
    inc = os.path.join(ROOT, "paper_2005_03070_gb300", "csrc")
    p = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-I" + inc,
                        "-I" + os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    checked, bad = (int(v) for v in r.stdout.split())
    assert r.returncode == 0 and bad == 0 and checked > 200, r.stdout
