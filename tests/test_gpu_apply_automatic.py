"""The automatic FP32 transport-operator apply (apply_kernel 0), which takes forms that no explicit choice asks
for: direction counts that are no multiple of four (4-byte copies, a partial last quad), staged tiles of 8 and
16 rows, slots shared by several warp groups, a ragged last direction chunk, 3D sets with such counts, applies
back to back (each launched while the one before it drains), and vectors that hold infinities and NaNs.

Against the oracle's L_m in FP64 and the row teams: 3e-6 relative L2, as for the other FP32 applies."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import mlpg_inputs as mi  # noqa: E402
import oracle.mlpg_oracle as O  # noqa: E402
import paper_2008_02205_gb300 as pkg  # noqa: E402


def _problem(dim, side, sn, m):
    prob = mi.two_region_2d(n_per_dim=side, sn=sn, seed=2300 + side) if dim == 2 else \
        mi.lognormal_3d(side, sn=sn, seed=3300 + side)
    prob.omega, prob.w = prob.omega[:m].copy(), prob.w[:m].copy()   # a shard of the set
    return prob


def _open(prob, **opts):
    return pkg.TransportProblem.from_problem(prob, precision=pkg.MLPG_MIXED, **opts).integrate().assemble()


def _apply(tp, prob, X, Y):
    pkg.mlpg_apply_L_dev(tp.ctx, prob.dt, pkg.MLPG_MIXED, X.data_ptr(), Y.data_ptr())
    torch.cuda.synchronize()
    return Y


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# (dim, points per side, S_N, directions, rows per tile asked for, kernel that serves, several chunks)
CASES = [
    (2, 13, 4, 12, 0, 2, False),    # 8-row tiles, the last ragged
    (2, 13, 4, 11, 0, 2, False),
    (2, 17, 8, 14, 0, 2, False),
    (2, 70, 4, 12, 0, 2, False),    # 16-row tiles
    (2, 30, 12, 67, 64, 2, True),   # two chunks of 36 and 31 directions on 64-row tiles
    (2, 30, 12, 80, 64, 2, True),   # two equal chunks
    (3, 5, 8, 27, 0, 2, False),     # staged tiles in 3D
    (3, 6, 4, 23, 0, 2, False),
    (3, 6, 4, 24, 0, 4, False),     # gather mode, row pairs
    (3, 12, 4, 24, 0, 4, False),    # gather mode, single rows
    (3, 6, 4, 24, 32, 2, False),
    (3, 6, 4, 24, 64, 2, False),    # gather mode takes at most 32 rows: staged tiles
]


@pytest.mark.parametrize("dim,side,sn,m,rows,kernel,chunks", CASES)
def test_automatic_apply_matches_oracle_and_row_teams(dim, side, sn, m, rows, kernel, chunks):
    prob = _problem(dim, side, sn, m)
    X = np.random.default_rng(23).uniform(-1.0, 1.0, (prob.n, m))
    Xd = torch.tensor(X, dtype=torch.float32, device="cuda")
    got = {}
    for k in (0, 1):
        with _open(prob, apply_kernel=k, **({"tile_rows": rows} if k == 0 else {})) as tp:
            got[k] = _apply(tp, prob, Xd, torch.full_like(Xd, float("nan"))).double().cpu().numpy()
            st = tp.stats()
            assert st["apply_kernel"] == (1 if k else kernel)
            if k == 0:
                assert (st["tile_chunk"] < m) == chunks
    disc = O.Discretization(prob.x, prob.R, prob.lo, prob.hi)
    tr = O.Transport(disc, disc.assemble_per_point(prob.sigma_t, prob.sigma_s, prob.q), prob.omega, prob.w)
    ref = np.stack([tr.L_matrix(d, 1.0 / prob.dt) @ X[:, d] for d in range(m)], axis=1)
    assert _rel(got[0], ref) < 3e-6
    assert _rel(got[0], got[1]) < 3e-6


@pytest.mark.parametrize("dim,side,sn,m", [(2, 13, 4, 12), (2, 40, 8, 14), (3, 6, 4, 24)])
def test_applies_back_to_back_read_each_others_output(dim, side, sn, m):
    """A chain of applies over two buffers, each reading what the one before it wrote and overwriting what the
    one before that read: the same bits as with a synchronisation after each."""
    prob = _problem(dim, side, sn, m)
    with _open(prob) as tp:
        out = []
        for wait in (True, False):
            g = torch.Generator(device="cuda").manual_seed(3)
            buf = [torch.rand(prob.n, m, device="cuda", generator=g), torch.empty(prob.n, m, device="cuda")]
            torch.cuda.synchronize()
            for k in range(12):
                pkg.mlpg_apply_L_dev(tp.ctx, prob.dt, pkg.MLPG_MIXED, buf[k % 2].data_ptr(), buf[1 - k % 2].data_ptr())
                if wait:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            out.append([b.cpu() for b in buf])
        for a, b in zip(*out):
            assert torch.isfinite(a).all() and torch.equal(a, b)


@pytest.mark.parametrize("kernel", [0, 2, 4])
@pytest.mark.parametrize("dim,side,sn,m", [(2, 13, 4, 12), (2, 13, 4, 11), (2, 30, 8, 40), (3, 6, 4, 24), (3, 6, 4, 23), (3, 12, 4, 24)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_values_stay_in_their_rows(dim, side, sn, m, kernel, value):
    """A NaN or an infinity at one point and direction reaches the rows whose pattern holds the point, in that
    direction, and nothing else changes."""
    if kernel and m % 4:
        pytest.skip("the explicit tile kernels take multiples of four")
    prob = _problem(dim, side, sn, m)
    with _open(prob, apply_kernel=kernel) as tp:
        rowptr, col = tp.neighbors()
        X = torch.rand(prob.n, m, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
        clean = _apply(tp, prob, X, torch.empty_like(X)).cpu()
        for at, d in ((0, 0), (prob.n // 2, m - 1), (prob.n - 1, 3)):
            Xb = X.clone()
            Xb[at, d] = value
            got = _apply(tp, prob, Xb, torch.empty_like(X)).cpu()
            rows = [i for i in range(prob.n) if at in col[rowptr[i]:rowptr[i + 1]]]
            hit = torch.zeros(prob.n, m, dtype=torch.bool)
            hit[rows, d] = True
            assert not torch.isfinite(got[hit]).any()
            # a sum taken again adds in another order: one row's rounding
            assert torch.isfinite(got[~hit]).all()
            assert _rel(got[~hit].numpy(), clean[~hit].numpy()) < 1e-6


def test_a_refused_shape_stays_refused():
    prob = _problem(2, 13, 4, 12)
    with _open(prob, apply_kernel=2, tile_dpt=8) as tp:   # eight directions per thread do not divide twelve
        X = torch.rand(prob.n, 12, device="cuda")
        for _ in range(2):
            with pytest.raises(pkg.MlpgError) as e:
                _apply(tp, prob, X, torch.empty_like(X))
            assert e.value.status == pkg.MLPG_ERR_ARG
