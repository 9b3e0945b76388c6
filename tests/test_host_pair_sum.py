"""The sums of FP32 products in pairs of floats (csrc/pair_sum.cuh), compiled with g++ without contraction:
chains of products and a tree of chains, as the Arnoldi step forms them, against exact sums (math.fsum) of the
rounded products.

Each addition's error goes into lo exactly and is rounded there to 24 bits of lo, which holds at most
2^-24 count of the magnitudes' sum: count^2 2^-48 of it bounds the error, against 2^-24 for a sum of floats.
Three floats carry the errors on once more: count^3 2^-72, below an FP64 sum's 2^-53 per addition."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_02205_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include "pair_sum.cuh"
int main() {
    float x[2 * 256];
    while (fread(x, sizeof(x), 1, stdin) == 1) {   // 32 lanes of 8 products, then the lanes by halves
        mlpg::Sum<float> s[32];
        for (int l = 0; l < 32; ++l) {
            s[l].clear();
            for (int k = 0; k < 8; ++k) s[l].add_product(x[2 * (8 * l + k)], x[2 * (8 * l + k) + 1]);
        }
        for (int o = 16; o > 0; o /= 2)
            for (int l = 0; l < o; ++l) s[l].add(s[l + o]);
        mlpg::TripleSum t;   // one chain over the same products
        for (int k = 0; k < 256; ++k) t.add(x[2 * k] * x[2 * k + 1]);
        const double v[2] = {s[0].value(), t.value()};
        fwrite(v, 8, 2, stdout);
    }
}
'''


def test_pair_sums_hold_more_than_forty_bits(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "main.cpp").write_text(HARNESS)
    exe = tmp_path / "sums"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-I{CSRC}", str(tmp_path / "main.cpp"), "-o", str(exe)],
                   check=True)
    rng = np.random.default_rng(2)
    x = rng.standard_normal((200, 256, 2))
    x[100:] *= np.exp(8.0 * rng.standard_normal((100, 256, 1)))      # magnitudes that differ
    x[50:100, 128:] = x[50:100, :128] * [-1.0, 1.0]                  # sums that cancel
    x = x.astype(np.float32)
    out = np.frombuffer(subprocess.run([str(exe)], input=x.tobytes(), capture_output=True, check=True).stdout, np.float64)
    for (v, t), row in zip(out.reshape(-1, 2), x):
        p = (row[:, 0] * row[:, 1]).astype(np.float64)
        exact, size = math.fsum(p), math.fsum(np.abs(p))
        assert abs(v - exact) <= 13**2 * 2.0**-48 * size
        # the two roundings of the final sum, and 256 additions' errors 2^-24 three times over
        assert abs(t - exact) <= 2.0**-52 * abs(exact) + 256**3 * 2.0**-72 * size
