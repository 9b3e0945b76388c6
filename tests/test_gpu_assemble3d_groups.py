"""The 3D volume forms integrated by groups of tetrahedra (fixed-point pair sums,
upper entries mirrored) against the oracle's forms, where the group kernel can go
wrong: both RK orders, lattices whose groups fit its table and kernels so wide that
some or all groups are handed to the element kernel, materials and extents that
differ from point to point.

Tolerance: the oracle integrates in FP64 with another summation order; the library's
other 3D form tests hold 1e-11 of each form's largest entry, the fixed point adds
2^-55 of the largest function value per product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


# (points per side, support in spacings, RK order, spread of the extents)
@pytest.mark.parametrize("side,support,order,spread", [
    (4, 2.0, 1, 0.0), (5, 2.0, 1, 0.0), (5, 2.0, 0, 0.0), (6, 2.3, 1, 0.1), (6, 2.5, 1, 0.0), (5, 2.5, 0, 0.05)])
def test_group_forms_match_oracle(side, support, order, spread):
    rng = np.random.default_rng(40 + side)
    prob = mi.make_problem("groups", side, 3, 2, 700 + side, lambda x, r: r.uniform(0.1, 10.0, len(x)), 0.3, 1.0, 0.01, 1,
                           support=support)
    prob.R = prob.R * (1.0 + spread * rng.uniform(-1.0, 1.0, prob.n))
    prob.sigma_s = 0.4 * prob.sigma_t
    prob.q = rng.uniform(0.0, 1.0, prob.n)
    with pkg.TransportProblem.from_problem(prob, rk_order=order) as tp:
        tp.integrate().assemble()
        mats, vecs = tp.forms()
        rowptr, col = tp.neighbors()
    disc = O.Discretization(prob.x, prob.R, prob.lo, prob.hi, rk_order=order)
    assert np.array_equal(rowptr, disc.rowptr) and np.array_equal(col, disc.col)
    F = disc.assemble_per_point(prob.sigma_t, prob.sigma_s, prob.q)
    ref = np.concatenate([np.atleast_2d(np.asarray(F[k]).reshape(-1, len(col))) for k in ("M0", "Mt", "Ms", "G", "Gt", "Gs", "K", "S")])
    refv = np.concatenate([np.atleast_2d(np.asarray(F[k]).reshape(-1, prob.n)) for k in ("Q0", "Q", "B")])
    for got, want in ((mats, ref), (vecs, refv)):
        assert got.shape == want.shape
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= 1e-11 * max(np.abs(b).max(), 1e-300)
