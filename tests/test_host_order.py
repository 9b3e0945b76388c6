"""The spatial order of the points (csrc/order.cpp, host code run once per
point set), compiled with g++ and checked on the CPU: a permutation whose
aligned runs are compact boxes, on jittered and regular lattices (ties) of any
side, with one thread or several."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import mlpg_inputs as mi

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2008_02205_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

HARNESS = r'''
#include <cstdio>
#include "internal.h"
int main(int argc, char **argv) {
    FILE *f = fopen(argv[1], "rb");
    int64_t n, dim;
    if (fread(&n, 8, 1, f) != 1 || fread(&dim, 8, 1, f) != 1) return 1;
    std::vector<double> x(n * dim);
    if (fread(x.data(), 8, n * dim, f) != (size_t)(n * dim)) return 1;
    fclose(f);
    std::vector<int32_t> order(n);
    mlpg::spatial_order(n, (int)dim, x.data(), order.data());
    FILE *o = fopen(argv[2], "wb");
    fwrite(order.data(), 4, n, o);
    fclose(o);
    return 0;
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("order")
    src = d / "main.cpp"
    src.write_text(HARNESS)
    exe = d / "harness"
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), os.path.join(CSRC, "order.cpp"), "-o", str(exe)],
                   check=True, capture_output=True)
    return d, exe


# (points, or points per side and jitter); 101^2 and 25^3 run on several threads
@pytest.mark.parametrize("dim,side,jitter", [(2, 2, 0.2), (2, 13, 0.2), (2, 32, 0.0), (2, 75, 0.2), (2, 101, 0.2),
                                             (3, 7, 0.0), (3, 15, 0.2), (3, 25, 0.2)])
def test_order_is_a_compact_permutation(harness, dim, side, jitter):
    d, exe = harness
    x, h = mi.jittered_lattice(side, dim, 91 + side, jitter=jitter)
    n = len(x)
    with open(d / "in.bin", "wb") as f:
        np.array([n, dim], np.int64).tofile(f)
        x.tofile(f)
    subprocess.run([str(exe), str(d / "in.bin"), str(d / "out.bin")], check=True, timeout=120)
    order = np.fromfile(d / "out.bin", np.int32)
    assert np.array_equal(np.sort(order), np.arange(n))
    if n < 64:
        return
    y = x[order]
    # pairs: neighbours; runs of 16 and 64: boxes of about 16 and 64 cells (no run wider than twice a cube's side)
    dist = np.linalg.norm(y[0:n // 2 * 2:2] - y[1:n // 2 * 2:2], axis=1)
    assert dist.max() < 4.0 * h and np.mean(dist < 2.0 * h) > 0.9
    for run in (16, 64):
        r = y[:n // run * run].reshape(-1, run, dim)
        assert (r.max(1) - r.min(1)).max() < (2.0 * run ** (1.0 / dim) + 1.0) * h
