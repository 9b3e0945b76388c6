"""Forms between functions that are small wherever they meet: two wide functions on a fine lattice whose supports
overlap in a thin lens, so that both are 1e-5 of the lattice's functions there, in every cell that they share.
The pair sums run in fixed point on each function's own scale, which keeps these entries to
2^-53 / (ratio of the values in the lens to the function's largest in the same cell)^2: the ratio is about 1e-3
here, 1e-10 of the entry.  (One scale for all functions of a cell would leave 1e-7 to 1e-6.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("dim,side,support,radius,gap", [(2, 20, 1.8, 0.2, 0.006), (3, 8, 1.8, 0.5, 0.02)])
def test_entries_of_barely_overlapping_functions(dim, side, support, radius, gap):
    prob = mi.make_problem("contrast", side, dim, 4, 11, 1.0, 0.3, 1.0, 0.01, 1, support=support, jitter=0.1)
    mid = 0.5 + 0.3 / side
    wide = np.full((2, dim), mid)
    wide[:, 0] = 0.5 - radius + gap / 2, 0.5 + radius - gap / 2
    prob.x = np.concatenate([prob.x, wide])
    prob.R = np.concatenate([prob.R, [radius, radius]])
    for k in ("sigma_t", "sigma_s", "q"):
        setattr(prob, k, np.full(len(prob.x), 0.7))
    with pkg.TransportProblem.from_problem(prob) as tp:
        tp.integrate().assemble()
        mats, _ = tp.forms()
        rowptr, col = tp.neighbors()
    disc = O.Discretization(prob.x, prob.R, prob.lo, prob.hi)
    assert np.array_equal(col, disc.col)
    F = disc.assemble_per_point(prob.sigma_t, prob.sigma_s, prob.q)
    a = prob.n - 2
    for i, j in ((a, a + 1), (a + 1, a)):
        p = rowptr[i] + int(np.searchsorted(col[rowptr[i]:rowptr[i + 1]], j))
        assert col[p] == j
        for got, ref in ((mats[0, p], F["M0"].reshape(-1)[p]), (mats[3 + 3 * dim, p], F["K"].reshape(dim * dim, -1)[0, p])):
            assert ref != 0.0 and abs(got - ref) <= 1e-9 * abs(ref)
