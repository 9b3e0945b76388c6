"""A batch takes the one-launch Arnoldi step or the separate passes by its points together, so that a problem
may take one form alone and the other in a batch: sizes where it does (16384 points in FP32, 4096 in FP64), one
and two Gram-Schmidt passes.  Both forms sum to the same accuracy, so the solves take the same iterations but for
a few that end one sooner or later: within 3 % in all, and as many refinements.  A lost pass or a wrong sum
costs orthogonality and with it iterations.  States agree to the refined or FP64 solves' tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("precision,reorth,sides", [
    (pkg.MLPG_MIXED, 0, (80, 78, 76)), (pkg.MLPG_MIXED, 1, (80, 78, 76)), (pkg.MLPG_FP64, 0, (40, 39, 38))])
def test_both_forms_take_the_same_iterations(precision, reorth, sides):
    limit = 16384 if precision == pkg.MLPG_MIXED else 4096
    assert all(k * k <= limit < len(sides) * k * k for k in sides)
    probs = [mi.two_region_2d(n_per_dim=k, sn=4, seed=9 + k, dt=1.28 / k) for k in sides]
    tps = [pkg.TransportProblem.from_problem(p, precision=precision, mixed_reorth=reorth).integrate().assemble()
           for p in probs]
    runs = []
    for batch in (False, True):
        for tp in tps:
            pkg.mlpg_set_initial(tp.ctx, None)
        if batch:
            pkg.TransportProblem.step_batch(tps, [p.dt for p in probs])
        else:
            for tp, p in zip(tps, probs):
                tp.step(p.dt)
        runs.append([(tp.stats(), tp.state()) for tp in tps])
    for (a, pa), (b, pb) in zip(*runs):
        assert a["last_refinements"] == b["last_refinements"]
        assert abs(a["last_inner_iters"] - b["last_inner_iters"]) <= 0.03 * a["last_inner_iters"]
        assert np.linalg.norm(pa - pb) <= 1e-9 * np.linalg.norm(pa)
    for tp in tps:
        tp.close()
