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


@pytest.mark.parametrize("dim,side,scale", [(2, 10, 1e22), (2, 10, 1e-25), (3, 5, 1e22), (3, 5, 1e-25)])
def test_forms_scale_with_the_lengths(dim, side, scale):
    """Which functions reach a point is decided in FP32 where that is certain; lengths whose squares leave
    FP32's range are decided in FP64.  M0_ij = V_j int u_i u_j, K_ij = V_j int du_i du_j with u of order 1 / V:
    powers 0 and -2 of the unit."""
    forms = []
    for s in (1.0, scale):
        p = mi.small_2d(side, sn=4, seed=4) if dim == 2 else mi.lognormal_3d(side, sn=4, seed=4)
        with pkg.TransportProblem(p.x * s, p.R * s, p.omega, p.w, p.sigma_t, p.sigma_s, p.q, lo=[0.0] * dim,
                                  hi=[s] * dim) as tp:
            tp.integrate().assemble()
            forms.append((tp.neighbors()[1], tp.forms()[0]))
    (col, a), (col1, b) = forms
    assert np.array_equal(col, col1)
    for k, power in ((0, 0), (3 + 3 * dim, -2)):   # M0, K_xx
        assert np.abs(b[k] / scale**power - a[k]).max() < 1e-11 * np.abs(a[k]).max()
