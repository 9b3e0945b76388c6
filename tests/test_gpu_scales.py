"""Units: the problem is linear in its source and homogeneous in its lengths, so that a solution or a form in
other units is the old one times a power, whatever the unit (FP64 holds its relative accuracy down to 1e-308,
the FP32 parts inside must not cut that short)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("scale", [1e-45, 1e-60, 1e-150, 1e60])
def test_fp64_step_scales_with_its_source(scale):
    """The block preconditioner holds FP32 inverses: their products with small FP64 vectors (the solution
    update is not normalised) must keep FP64's range.  Both solves end at a relative residual of 1e-12."""
    out = []
    for s in (1.0, scale):
        prob = mi.small_2d(12, sn=4, seed=3)
        prob.q = prob.q * s
        with pkg.TransportProblem.from_problem(prob, max_inner=400) as tp:
            tp.integrate().assemble().step(prob.dt)
            out.append(tp.state() / s)
    assert _rel(out[1], out[0]) < 1e-10
