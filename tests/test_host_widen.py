"""The FP32 -> FP64 widening by integer moves (csrc/widen.cuh), compiled with g++ and compared bit for bit
with the conversion: zeros, subnormals, the edges of every exponent, infinities, NaNs and random bits."""
import shutil
import subprocess
import os

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_02205_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include "widen.cuh"
int main() {
    uint32_t b, w[2];
    while (fread(&b, 4, 1, stdin) == 1) {
        mlpg::widen_words(b, w[1], w[0]);
        fwrite(w, 4, 2, stdout);
    }
}
'''


def test_widening_equals_the_conversion(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "main.cpp").write_text(HARNESS)
    exe = tmp_path / "widen"
    subprocess.run(["g++", "-O2", "-std=c++17", f"-I{CSRC}", str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    mant = np.concatenate([[0, 1, 2, 0x400000, 0x7ffffe, 0x7fffff], 1 << np.arange(23)]).astype(np.uint32)
    bits = (np.arange(256, dtype=np.uint32)[:, None] << 23 | mant).ravel()
    bits = np.concatenate([bits, bits | np.uint32(1 << 31),
                           np.random.default_rng(1).integers(0, 1 << 32, 100000, dtype=np.uint32)])
    out = np.frombuffer(subprocess.run([str(exe)], input=bits.tobytes(), capture_output=True, check=True).stdout, np.float64)
    f = bits.view(np.float32)
    with np.errstate(invalid="ignore"):
        want = f.astype(np.float64)
    nan = np.isnan(f)
    assert np.array_equal(np.isnan(out), nan)
    assert np.array_equal(out[~nan].view(np.uint64), want[~nan].view(np.uint64))
