"""The assembly's scratch counts in the problem's device_bytes and takes no room of its own: it lies where the
operators' arrays go, so that forming the operators adds that much less."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("dim,scratch", [(2, 6), (3, 9)])
def test_assembly_scratch_is_counted(dim, scratch):
    prob = mi.small_2d(20, sn=4, seed=2) if dim == 2 else mi.lognormal_3d(6, sn=4, seed=2)
    with pkg.TransportProblem.from_problem(prob) as tp:
        tp.integrate()
        before, nnz = tp.stats()["device_bytes"], tp.stats()["nnz"]
        tp.assemble()
        assert tp.stats()["device_bytes"] - before >= 8 * nnz * (pkg.mlpg_n_matrices(dim) + scratch)
        first = tp.forms()[0]
        X = torch.rand(prob.n, prob.m, device="cuda", dtype=torch.float64)
        Y = torch.empty_like(X)
        pkg.mlpg_apply_L_dev(tp.ctx, prob.dt, pkg.MLPG_FP64, X.data_ptr(), Y.data_ptr())
        torch.cuda.synchronize()
        assert torch.isfinite(Y).all() and (tp.forms()[0] == first).all()
