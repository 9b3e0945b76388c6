"""The one-launch Arnoldi step (small problems) against the separate passes and the
oracle, at the sizes where it can go wrong: fewer rows than a cluster's CTAs hold
each, rows that do not divide evenly, one to four groups of basis vectors (restarts up
to the cap of 32; much shorter ones stagnate on these problems with either form), direction counts served by the two
cluster widths and those that keep the separate passes (no multiple of four), one
and two Gram-Schmidt passes.

The converged step does not depend on the Krylov basis: FP64 runs agree with the
oracle to the solves' tolerance (1e-9 of the flux), mixed ones to 1e-8, as in the
library's other solves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("side,sn,drop,restart,reorth", [
    (5, 4, 0, 20, 0), (9, 4, 0, 20, 1), (11, 6, 0, 24, 0), (13, 8, 0, 32, 1), (10, 4, 1, 20, 0), (17, 6, 0, 25, 1)])
def test_steps_match_oracle(side, sn, drop, restart, reorth):
    prob = mi.two_region_2d(n_per_dim=side, sn=sn, seed=2600 + side, steps=2)
    if drop:   # a direction set that is no multiple of four
        keep = prob.m - drop
        prob.omega, prob.w = prob.omega[:keep].copy(), prob.w[:keep].copy()
    ref = O.solve_problem(prob)
    with pkg.TransportProblem.from_problem(prob, inner_tol=1e-13, outer_tol=1e-13, inner_restart=max(restart, 20)) as tp:
        tp.integrate().assemble()
        assert _rel(tp.run(prob.dt, prob.steps), ref) < 1e-9
    with pkg.TransportProblem.from_problem(prob, precision=pkg.MLPG_MIXED, refine_tol=1e-12, mixed_restart=restart,
                                           mixed_reorth=reorth, max_refine=40) as tp:
        tp.integrate().assemble()
        assert _rel(tp.run(prob.dt, prob.steps), ref) < 1e-8


def test_batch_gives_each_problem_its_own_result():
    """In a batch the choice between the two forms also counts the problems: the same states."""
    probs = [mi.small_2d(n, sn=4, seed=1700 + n, steps=1) for n in (8, 40, 70)]
    single, batch = [], []
    for p in probs:
        with pkg.TransportProblem.from_problem(p, precision=pkg.MLPG_MIXED, refine_tol=1e-12) as tp:
            tp.integrate().assemble().step(p.dt)
            single.append(tp.state())
    tps = [pkg.TransportProblem.from_problem(p, precision=pkg.MLPG_MIXED, refine_tol=1e-12).integrate().assemble()
           for p in probs]
    pkg.TransportProblem.step_batch(tps, [p.dt for p in probs])
    for tp, s in zip(tps, single):
        assert _rel(tp.state(), s) < 1e-9
        tp.close()
