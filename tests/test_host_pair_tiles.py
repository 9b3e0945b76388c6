"""The row-pair tiles of the FP32 transport-operator apply (csrc/tiles.cpp,
host code run once per point set) on the spatial order (csrc/order.cpp), compiled with g++ and
checked on the CPU against the overlap pattern the oracle builds (Sec. 3.4).

Every pattern entry must sit in exactly one slot of its own pair and row, each slot
must lead back to its column, and a pair's slots must be the sorted union of
its two rows' columns."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import mlpg_inputs as mi
import oracle.mlpg_oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2008_02205_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

HARNESS = r'''
#include <cstdio>
#include <vector>
#include "internal.h"
template <class T> static void rd(FILE *f, T *p, size_t k) { if (fread(p, sizeof(T), k, f) != k) throw 1; }
template <class T> static void wr(FILE *f, const std::vector<T> &v) { fwrite(v.data(), sizeof(T), v.size(), f); }
int main(int argc, char **argv) {
    FILE *f = fopen(argv[1], "rb");
    int64_t n, nnz, dim, tr, halo;
    rd(f, &n, 1); rd(f, &nnz, 1); rd(f, &dim, 1); rd(f, &tr, 1); rd(f, &halo, 1);
    std::vector<double> x(n * dim);
    std::vector<int32_t> rowptr(n + 1), col(nnz), order(n);
    rd(f, x.data(), n * dim); rd(f, rowptr.data(), n + 1); rd(f, col.data(), nnz);
    fclose(f);
    mlpg::spatial_order(n, (int)dim, x.data(), order.data());
    mlpg::PairTileLayout t;
    int64_t nslot = mlpg::build_pair_tiles(n, rowptr.data(), col.data(), order.data(), (int)tr, 4, halo != 0, t);
    FILE *o = fopen(argv[2], "wb");
    std::vector<int64_t> head = {nslot, t.ntile, t.max_halo, (int64_t)t.hcol.size()};
    wr(o, head); wr(o, order); wr(o, t.base); wr(o, t.width); wr(o, t.row); wr(o, t.plen); wr(o, t.hptr);
    wr(o, t.hcol); wr(o, t.perm0); wr(o, t.perm1); wr(o, t.lcol);
    fclose(o);
    return 0;
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("pair_tiles")
    src = d / "main.cpp"
    src.write_text(HARNESS)
    exe = d / "harness"
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), os.path.join(CSRC, "tiles.cpp"), os.path.join(CSRC, "order.cpp"), "-o", str(exe)],
                   check=True, capture_output=True)
    return d, exe


# odd and even point counts, ragged last tiles, a regular lattice (ties), enough points for several threads
@pytest.mark.parametrize("dim,side,tr,halo,jitter", [
    (2, 13, 64, 1, 0.2), (2, 30, 16, 1, 0.2), (2, 17, 8, 0, 0.0), (3, 7, 4, 0, 0.2), (3, 6, 32, 1, 0.2),
    (2, 75, 32, 1, 0.2), (2, 2, 4, 1, 0.2)])
def test_pair_tiles_cover_the_pattern_once(harness, dim, side, tr, halo, jitter):
    d, exe = harness
    x, h = mi.jittered_lattice(side, dim, 91 + side, jitter=jitter)
    n = len(x)
    rowptr, col = O.neighbors(x, np.full(n, 2.0 * h))
    inp, out = d / "in.bin", d / "out.bin"
    with open(inp, "wb") as f:
        np.array([n, len(col), dim, tr, halo], np.int64).tofile(f)
        x.tofile(f)
        np.asarray(rowptr, np.int32).tofile(f)
        np.asarray(col, np.int32).tofile(f)
    subprocess.run([str(exe), str(inp), str(out)], check=True, timeout=120)
    b, pos = open(out, "rb").read(), 0

    def take(dtype, k):
        nonlocal pos
        a = np.frombuffer(b, dtype, k, pos)
        pos += a.nbytes
        return a
    nslot, ntile, max_halo, nh = (int(v) for v in take(np.int64, 4))
    tp = tr // 2
    order, base, width = take(np.int32, n), take(np.int64, ntile + 1), take(np.int32, ntile)
    rows, plen = take(np.int32, ntile * tr), take(np.int32, ntile * tp)
    hptr, hcol = take(np.int64, ntile + 1), take(np.int32, nh)
    perm = [take(np.int32, nslot), take(np.int32, nslot)]
    lcol = take(np.int32, nslot)
    assert pos == len(b) and ntile == -(-n // tr)
    assert np.array_equal(np.sort(order), np.arange(n))
    assert np.array_equal(rows[:n], order) and np.all(rows[n:] == -1)
    seen = np.zeros(len(col), np.int64)
    for t in range(ntile):
        w = width[t]
        assert base[t + 1] - base[t] == w * tp and w == -(-plen[t * tp:(t + 1) * tp].max() // 4) * 4
        sl = [p[base[t]:base[t + 1]].reshape(w, tp) for p in perm]
        lc = lcol[base[t]:base[t + 1]].reshape(w, tp)
        hc = hcol[hptr[t]:hptr[t + 1]]
        union = []
        for s in range(tp):
            pair = rows[t * tr + 2 * s:t * tr + 2 * s + 2]
            want = np.unique(np.concatenate([np.empty(0, np.int32)] + [col[rowptr[i]:rowptr[i + 1]] for i in pair if i >= 0]))
            k = plen[t * tp + s]
            assert k == len(want)
            got = hc[lc[:k, s]] if halo else lc[:k, s]
            assert np.array_equal(got, want) and np.all(lc[k:, s] == 0)
            union.append(want)
            for r in (0, 1):
                e = sl[r][:, s]
                assert np.all(e[k:] == -1)
                live = e[e >= 0]
                i = pair[r]
                assert np.array_equal(live, np.arange(rowptr[i], rowptr[i + 1]) if i >= 0 else [])
                assert np.array_equal(got[e[:k] >= 0], col[live])
                seen[live] += 1
        if halo:
            assert np.array_equal(hc, np.unique(np.concatenate(union)))
    assert np.all(seen == 1)
    assert max_halo == (max(hptr[1:] - hptr[:-1]) if halo else 0)
