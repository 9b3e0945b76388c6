"""The scattering source's division by 4 pi (csrc/four_pi.cuh), compiled with g++ and compared bit for bit with
the division: random mantissas at every exponent, zeros, subnormals, infinities, NaNs."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_02205_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include "four_pi.cuh"
int main() {
    double v;
    while (fread(&v, 8, 1, stdin) == 1) {
        const double o[2] = {mlpg::div_four_pi(v), (double)mlpg::div_four_pi_f(v)};
        fwrite(o, 8, 2, stdout);
    }
}
'''


def test_division_by_four_pi_rounds_as_the_division(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "main.cpp").write_text(HARNESS)
    exe = tmp_path / "div"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-I{CSRC}", str(tmp_path / "main.cpp"), "-o", str(exe)],
                   check=True)
    rng = np.random.default_rng(3)
    mant = rng.integers(0, 1 << 52, (2048, 200), dtype=np.uint64)
    mant[:, :3] = [0, 1, (1 << 52) - 1]
    bits = (np.arange(2048, dtype=np.uint64)[:, None] << np.uint64(52) | mant).ravel()
    v = np.concatenate([bits, bits | np.uint64(1 << 63)]).view(np.float64)
    v = np.concatenate([v, rng.standard_normal(500000)])
    out = np.frombuffer(subprocess.run([str(exe)], input=v.tobytes(), capture_output=True, check=True).stdout, np.float64)
    out, out32 = out[0::2], out[1::2]
    with np.errstate(invalid="ignore", over="ignore"):
        want = v / (4.0 * math.pi)
        want32 = want.astype(np.float32).astype(np.float64)
    nan = np.isnan(v)
    for got, w in ((out, want), (out32, want32)):
        assert np.array_equal(np.isnan(got), nan)
        same = got[~nan] == w[~nan]
        assert same.all()   # (the sign of a zero source does not matter)
