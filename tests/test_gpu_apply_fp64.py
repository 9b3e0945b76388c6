"""The FP64 transport-operator apply with 1, 4, 8 and 16 lanes per (row, direction), at the sizes that each
serves, against the oracle's L_m.  The operators' forms agree to 1e-11 of their largest entry (the form tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("dim,side,sn,m", [
    (2, 64, 8, 40), (2, 60, 8, 13), (2, 13, 4, 12), (2, 13, 4, 1), (3, 6, 4, 24), (3, 8, 8, 27), (3, 8, 8, 1)])
def test_fp64_apply_matches_oracle(dim, side, sn, m):
    prob = mi.two_region_2d(n_per_dim=side, sn=sn, seed=2400 + side) if dim == 2 else \
        mi.lognormal_3d(side, sn=sn, seed=3400 + side)
    prob.omega, prob.w = prob.omega[:m].copy(), prob.w[:m].copy()
    X = np.random.default_rng(29).uniform(-1.0, 1.0, (prob.n, m))
    Xd = torch.tensor(X, device="cuda")
    Yd = torch.full_like(Xd, float("nan"))
    with pkg.TransportProblem.from_problem(prob) as tp:
        tp.integrate().assemble()
        torch.cuda.synchronize()
        pkg.mlpg_apply_L_dev(tp.ctx, prob.dt, pkg.MLPG_FP64, Xd.data_ptr(), Yd.data_ptr())
        torch.cuda.synchronize()
    Y = Yd.cpu().numpy()
    disc = O.Discretization(prob.x, prob.R, prob.lo, prob.hi)
    tr = O.Transport(disc, disc.assemble_per_point(prob.sigma_t, prob.sigma_s, prob.q), prob.omega, prob.w)
    assert np.isfinite(Y).all()
    for d in range(0, m, max(1, m // 5)):
        ref = tr.L_matrix(d, 1.0 / prob.dt) @ X[:, d]
        assert np.linalg.norm(Y[:, d] - ref) <= 1e-11 * np.linalg.norm(ref)
