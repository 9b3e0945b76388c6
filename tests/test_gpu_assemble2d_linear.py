"""The 2D forms with linear RK functions (fixed-point pair sums, upper entries
mirrored) against the oracle's forms where the kernel can go wrong: one to several
chunks of points per cell, corner cells with two faces, regular lattices (functions
exactly at their support's edge), extents that differ from point to point, function
counts up to the kernel's limit, materials that vary.

Tolerance: as the library's other form tests, 1e-11 of each form's largest entry; the
fixed point adds 2^-54 of the largest function value per product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


# (points per side, support in spacings, jitter, spread of the extents)
@pytest.mark.parametrize("side,support,jitter,spread", [
    (3, 2.0, 0.2, 0.0), (8, 2.0, 0.0, 0.0), (11, 2.0, 0.2, 0.0), (13, 1.8, 0.2, 0.1), (12, 2.2, 0.2, 0.05)])
def test_linear_forms_match_oracle(side, support, jitter, spread):
    rng = np.random.default_rng(60 + side)
    prob = mi.make_problem("linear", side, 2, 2, 800 + side, lambda x, r: r.uniform(0.1, 10.0, len(x)), 0.3, 1.0, 0.01, 1,
                           support=support, jitter=jitter)
    prob.R = prob.R * (1.0 + spread * rng.uniform(-1.0, 1.0, prob.n))
    prob.sigma_s = 0.4 * prob.sigma_t
    prob.q = rng.uniform(0.0, 1.0, prob.n)
    with pkg.TransportProblem.from_problem(prob) as tp:
        tp.integrate().assemble()
        mats, vecs = tp.forms()
        rowptr, col = tp.neighbors()
    disc = O.Discretization(prob.x, prob.R, prob.lo, prob.hi)
    assert np.array_equal(rowptr, disc.rowptr) and np.array_equal(col, disc.col)
    F = disc.assemble_per_point(prob.sigma_t, prob.sigma_s, prob.q)
    ref = np.concatenate([np.asarray(F[k]).reshape(-1, len(col)) for k in ("M0", "Mt", "Ms", "G", "Gt", "Gs", "K", "S")])
    refv = np.concatenate([np.asarray(F[k]).reshape(-1, prob.n) for k in ("Q0", "Q", "B")])
    for got, want in ((mats, ref), (vecs, refv)):
        assert got.shape == want.shape
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= 1e-11 * max(np.abs(b).max(), 1e-300)


def test_too_many_functions_are_refused():
    prob = mi.small_2d(12, sn=4)
    prob.R = prob.R * 1.5
    with pkg.TransportProblem.from_problem(prob) as tp:
        tp.integrate()
        with pytest.raises(pkg.MlpgError) as e:
            tp.assemble()
        assert e.value.status == pkg.MLPG_ERR_ARG
