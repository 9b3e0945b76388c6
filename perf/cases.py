"""Performance cases: the work that a user of the transport library has it do.

Each case goes through the public entry points of ``paper_2008_02205_gb300``:

* ``apply``: the batched transport operator ``mlpg_apply_L_dev`` for all
  directions at once, on resident operators (the call that a user's own Krylov
  or source-iteration driver makes, and that fills the library's own steps);
* ``setup``: a point set that has moved: create from device arrays, integrate,
  assemble, then the first operator apply, volumes and overlap pattern;
* ``step``: one backward-Euler step of an assembled problem from a zero state,
  in FP64 (the default precision) or mixed precision, and the state;
* ``solve``: a whole time-dependent solve, as the benchmark runs it: create to
  scalar flux;
* ``batch``: one step of several independent problems at once, as the serving
  loop runs them.

Point sets are the paper's jittered lattices (support radius of two spacings),
angular sets are level-symmetric S_N, the refined hierarchical set, or one
shard of an S_N set; materials and sizes are those of the repository's own
configurations (the uniform 2D problem, the two-region benchmark, the
lognormal 3D problem with inflow, the batched 2D problems).
"""
import math

import numpy as np
import torch

import mlpg_inputs as mi
import paper_2008_02205_gb300 as pkg

FP64, MIXED = pkg.MLPG_FP64, pkg.MLPG_MIXED


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one apply of the 32 x 32, S4 problem (12 directions); launch-bound
        {"name": "apply-2d-32-s4", "do": "apply", "dim": 2, "side": 32, "sn": 4, "shards": 1, "prec": "mixed"},
        # the benchmark's operator: 256 x 256 points, S8 (40 directions), FP32
        {"name": "apply-2d-256-s8", "do": "apply", "dim": 2, "side": 256, "sn": 8, "shards": 1, "prec": "mixed"},
        # one of three direction shards of S8 (14 of 40 directions: no multiple of four), an odd point count
        {"name": "apply-2d-181-s8-shard3", "do": "apply", "dim": 2, "side": 181, "sn": 8, "shards": 3, "prec": "mixed"},
        # 3D with the set refined within 15 degrees of +x (272 directions), FP32
        {"name": "apply-3d-24-refined", "do": "apply", "dim": 3, "side": 24, "sn": 0, "shards": 1, "prec": "mixed"},
        # a 2D point set that has moved: neighbours, cells, all forms, first FP64 apply
        {"name": "setup-2d-128-s4", "do": "setup", "dim": 2, "side": 128, "sn": 4, "prec": "fp64"},
        # the same in 3D, at an odd size
        {"name": "setup-3d-15-s4", "do": "setup", "dim": 3, "side": 15, "sn": 4, "prec": "fp64"},
        # one FP64 step of the smallest configuration: many short launches
        {"name": "step-2d-32-s4-fp64", "do": "step", "dim": 2, "side": 32, "sn": 4, "prec": "fp64"},
        # one FP64 step of a two-region problem of ordinary size
        {"name": "step-2d-96-s8-fp64", "do": "step", "dim": 2, "side": 96, "sn": 8, "prec": "fp64"},
        # one mixed-precision step of the benchmark problem
        {"name": "step-2d-256-s8-mixed", "do": "step", "dim": 2, "side": 256, "sn": 8, "prec": "mixed"},
        # one mixed-precision step in 3D (S8: 80 directions, inflow on one face)
        {"name": "step-3d-20-s8-mixed", "do": "step", "dim": 3, "side": 20, "sn": 8, "prec": "mixed"},
        # a whole mixed-precision solve of a small two-region problem at an odd size, 5 steps
        {"name": "solve-2d-75-s6-mixed", "do": "solve", "dim": 2, "side": 75, "sn": 6, "steps": 5, "prec": "mixed"},
        # eight independent 2D problems (about 1k to 16k points, S4 to S12) stepped at once
        {"name": "batch-2d-8-mixed", "do": "batch", "dim": 2, "count": 8, "nmax": 16384, "prec": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["apply", "apply", "setup", "step", "solve", "batch"])
    if do == "batch":
        return {"do": do, "dim": 2, "count": rng.randint(2, 8), "nmax": _log_int(rng, 2048, 16384), "prec": "mixed"}
    dim = rng.choice([2, 2, 3])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    sn = rng.choice([4, 6, 8, 10, 12] if dim == 2 else [4, 8, 12])
    if do == "apply":
        side = _log_int(rng, 20, 256) if dim == 2 else _log_int(rng, 8, 24)
        if dim == 3 and rng.random() < 0.25:
            sn = 0
        if dim == 2 and side > 180:
            sn = min(sn, 8)
        return {"do": do, "dim": dim, "side": side, "sn": sn, "shards": rng.choice([1, 1, 1, 2, 3]), "prec": prec}
    if do == "setup":
        side = _log_int(rng, 20, 128) if dim == 2 else _log_int(rng, 7, 15)
        return {"do": do, "dim": dim, "side": side, "sn": sn, "prec": prec}
    if do == "solve":
        side = _log_int(rng, 20, 96) if dim == 2 else _log_int(rng, 7, 12)
        return {"do": do, "dim": dim, "side": side, "sn": min(sn, 8), "steps": rng.randint(2, 5), "prec": "mixed"}
    if prec == "fp64":
        side, sn = (_log_int(rng, 20, 96), min(sn, 8)) if dim == 2 else (_log_int(rng, 7, 12), 4)
    else:
        side, sn = (_log_int(rng, 24, 200), min(sn, 8)) if dim == 2 else (_log_int(rng, 8, 20), min(sn, 8))
    return {"do": do, "dim": dim, "side": side, "sn": sn, "prec": prec}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
_refined = []


def _refined_set():
    if not _refined:
        _refined.append(mi.refined_quadrature(1, 5, mi.cone_hits((1.0, 0.0, 0.0), 15.0)))
    return _refined[0]


def _problem(case, seed):
    """The point set, angular set and materials of one case (an ``mlpg_inputs.Problem``)."""
    side, dim, sn = case["side"], case["dim"], case["sn"]
    if dim == 3:
        # the lognormal problem with inflow; a step moves about 0.4 spacings, as at its full size
        p = mi.lognormal_3d(side, sn=sn or 4, seed=seed, steps=1, dt=0.4 / side)
        if sn == 0:
            om, w = _refined_set()
            p.omega, p.w = om.copy(), w.copy()
    elif sn == 4:
        p = mi.small_2d(side, sn=4, seed=seed, dt=0.32 / side)   # uniform, vacuum
    else:
        p = mi.two_region_2d(side, sn=sn, seed=seed, dt=1.28 / side)
    shards = case.get("shards", 1)
    if shards > 1:   # the first of `shards` contiguous, balanced parts of the directions
        k = -(-p.m // shards)
        p.omega, p.w = np.ascontiguousarray(p.omega[:k]), np.ascontiguousarray(p.w[:k])
    return p


def _batch_sides(case):
    """Points per side and S_N of each problem: log-spaced sizes, the batched configuration's sets in turn."""
    c = case["count"]
    n = [1024.0 * (case["nmax"] / 1024.0) ** (b / max(c - 1, 1)) for b in range(c)]
    return [(int(round(math.sqrt(v))), (4, 6, 8, 10, 12)[b % 5]) for b, v in enumerate(n)]


def _batch_problems(case, seed):
    """Independent 2D problems with the batched configuration's materials, drawn from the seed."""
    rng = np.random.Generator(np.random.PCG64(4000 + seed))
    out = []
    for b, (k, sn) in enumerate(_batch_sides(case)):
        sig, ratio = float(rng.uniform(0.1, 10.0)), float(rng.uniform(0.0, 0.99))
        out.append(mi.make_problem(f"batch{b}", k, 2, sn, 4000 + 97 * seed + b, sig, ratio * sig, 1.0, 0.01, 1))
    return out


def _vectors(case, seed, n, m):
    """The vector X of an apply, from the seed alone, on the current device."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(1 + seed)
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    return torch.randn(n, m, device=dev, dtype=dt, generator=g)


def _options(case, prob, stream):
    prec = FP64 if case["prec"] == "fp64" else MIXED
    return dict(precision=prec, stream=stream.cuda_stream, lo=prob.lo, hi=prob.hi)


def _device_arrays(p):
    keys = ("x", "R", "omega", "w", "sigma_t", "sigma_s", "q")
    return {k: torch.from_numpy(np.ascontiguousarray(getattr(p, k), dtype=np.float64)).cuda() for k in keys}


def prepare(case, seed):
    do = case["do"]
    st = {"case": case, "do": do}
    if do == "batch":
        probs = _batch_problems(case, seed)
        st["dts"] = [p.dt for p in probs]
        st["tp"] = [pkg.TransportProblem.from_problem(p, precision=MIXED).integrate().assemble() for p in probs]
        return st
    p = _problem(case, seed)
    st["dt"], st["n"], st["m"] = p.dt, p.n, p.m
    st["stream"] = torch.cuda.Stream()
    if do in ("setup", "solve"):
        st["dev"] = _device_arrays(p)
        st["inflow"] = p.inflow
        st["opt"] = pkg.mlpg_default_options(dim=p.dim, **_options(case, p, st["stream"]))
        if do == "setup":
            st["X"] = _vectors(case, seed, p.n, p.m)
            st["Y"] = torch.empty_like(st["X"])
        else:
            st["phi"] = torch.empty(p.n, dtype=torch.float64, device="cuda")
            st["Phi"] = torch.empty(p.n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return st
    st["tp"] = pkg.TransportProblem.from_problem(p, **_options(case, p, st["stream"])).integrate().assemble()
    if do == "apply":
        st["X"] = _vectors(case, seed, p.n, p.m)
        st["Y"] = torch.empty_like(st["X"])
        torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _create(st):
    d = st["dev"]
    ctx = pkg.mlpg_create_dev(st["opt"], st["n"], st["m"], *(d[k].data_ptr() for k in
                                                             ("x", "R", "omega", "w", "sigma_t", "sigma_s", "q")))
    for f, v in st["inflow"].items():
        pkg.mlpg_set_inflow(ctx, int(f), float(v))
    return ctx


def run(st):
    do, case = st["do"], st["case"]
    prec = FP64 if case["prec"] == "fp64" else MIXED
    if do == "apply":
        pkg.mlpg_apply_L_dev(st["tp"].ctx, st["dt"], prec, st["X"].data_ptr(), st["Y"].data_ptr())
        return st["Y"]
    if do == "step":
        ctx = st["tp"].ctx
        pkg.mlpg_set_initial(ctx, None)
        pkg.mlpg_step(ctx, st["dt"])
        return {"psi": pkg.mlpg_get_state(ctx, st["n"], st["m"])}
    if do == "batch":
        for tp in st["tp"]:
            pkg.mlpg_set_initial(tp.ctx, None)
        pkg.mlpg_step_batch([tp.ctx for tp in st["tp"]], st["dts"])
        return [pkg.mlpg_get_state(tp.ctx, tp.n, tp.m) for tp in st["tp"]]
    ctx = _create(st)
    try:
        pkg.mlpg_integrate(ctx)
        pkg.mlpg_assemble(ctx)
        if do == "setup":
            pkg.mlpg_apply_L_dev(ctx, st["dt"], prec, st["X"].data_ptr(), st["Y"].data_ptr())
            # the pattern's column list is as long as the jitter makes it; the apply checks it
            rowptr, _ = pkg.mlpg_get_neighbors(ctx, st["n"], pkg.mlpg_get_stats(ctx)["nnz"])
            return {"y": st["Y"], "volume": pkg.mlpg_get_volumes(ctx, st["n"]), "rowptr": rowptr}
        for _ in range(case["steps"]):
            pkg.mlpg_step(ctx, st["dt"])
        pkg.mlpg_scalar_flux_dev(ctx, st["phi"].data_ptr(), 0)
        pkg.mlpg_scalar_flux_dev(ctx, st["Phi"].data_ptr(), 1)
        return {"phi": st["phi"], "coefficients": st["Phi"], "psi": pkg.mlpg_get_state(ctx, st["n"], st["m"])}
    finally:
        pkg.mlpg_destroy(ctx)


# --------------------------------------------------------------------------
# the work that a pass cannot do without
# --------------------------------------------------------------------------
def _directions(case):
    if case["sn"] == 0:
        m = 272
    else:
        m = case["sn"] * (case["sn"] + 2) // (2 if case["dim"] == 2 else 1)
    return -(-m // case.get("shards", 1))


def _entries(side, dim):
    """Overlap-pattern entries of a lattice: offsets closer than four spacings."""
    r = range(-4, 5)
    one = {o: max(0, side - abs(o)) for o in r}
    if dim == 2:
        return sum(one[a] * one[b] for a in r for b in r if a * a + b * b < 16)
    return sum(one[a] * one[b] * one[c] for a in r for b in r for c in r if a * a + b * b + c * c < 16)


def work(case):
    """apply: the CSR form of the operator (base arrays, columns, rows), X and Y
    once; one combination and one product per entry and direction.  setup: the
    inputs, the forms that are built and the apply; per quadrature point, the
    forms of each pair of functions that are non-zero there.  step, solve,
    batch: the operator once, the state in and out, one residual per step."""
    if case["do"] == "batch":
        size = [(k * k, sn * (sn + 2) // 2, _entries(k, 2)) for k, sn in _batch_sides(case)]
        return {"bytes": sum(28.0 * nnz + 2 * 8 * n * m for n, m, nnz in size),
                "flops": sum(2.0 * 6 * nnz * m for n, m, nnz in size)}
    side, dim = case["side"], case["dim"]
    n, m, nnz = side ** dim, _directions(case), _entries(side, dim)
    arrays = 6 if dim == 2 else 10
    size = 8 if case["prec"] == "fp64" else 4
    apply_bytes = nnz * (4 + size * arrays) + 4 * (n + 1) + 2 * n * m * size
    apply_flops = 2.0 * arrays * nnz * m
    # quadrature points per cell, functions at a point, products per pair of functions
    points, funcs, forms = (150, 12.6, 9) if dim == 2 else (632, 33.5, 16)
    setup_flops = 2.0 * n * points * (0.5 * funcs * (funcs + 1) * forms + 40 * funcs)
    mats, vecs = (17, 7) if dim == 2 else (27, 10)
    setup_bytes = 8.0 * (n * (dim + 4) + mats * nnz + vecs * n)
    if case["do"] == "apply":
        return {"bytes": apply_bytes, "flops": apply_flops}
    if case["do"] == "setup":
        return {"bytes": setup_bytes + apply_bytes, "flops": setup_flops + apply_flops}
    if case["do"] == "step":
        return {"bytes": apply_bytes + 2 * 8 * n * m, "flops": apply_flops}
    s = case["steps"]
    return {"bytes": setup_bytes + s * (apply_bytes + 2 * 8 * n * m), "flops": setup_flops + s * apply_flops}


# --------------------------------------------------------------------------
# the same quantities in 64 bits, in plain torch (2D)
#
# Everything lives on the lattice that the points were jittered from: point
# (ix, iy) and offsets to its lattice neighbours, with out-of-range ones masked.
# --------------------------------------------------------------------------
_OFF = 4            # overlap: closer than 4 spacings, jitter up to 0.2 each
_ROFF = 3           # functions that reach a cell: its radius + 2 spacings


class _Lattice2:
    def __init__(self, p, side, dev):
        self.k, self.n, self.dev = side, p.n, dev
        self.x = torch.as_tensor(p.x, device=dev)
        self.R = float(p.R[0])
        i = torch.arange(self.n, device=dev)
        self.ix, self.iy = i % side, i // side

    def near(self, rows, ox, oy):
        """(index, exists) of the points at lattice offset (ox, oy); any broadcastable shapes."""
        jx, jy = self.ix[rows] + ox, self.iy[rows] + oy
        ok = (jx >= 0) & (jx < self.k) & (jy >= 0) & (jy < self.k)
        return torch.where(ok, jy * self.k + jx, torch.zeros_like(jx)), ok


def _cells2(L, lo, hi):
    """Convex cells: the square x_i +- R in the box, cut by the bisectors with all
    overlapping points.  Vertices [n, P, 2] (counter-clockwise) and their counts."""
    n, dev, P = L.n, L.dev, 20
    a = torch.maximum(L.x - L.R, torch.as_tensor(lo[:2], device=dev, dtype=torch.float64))
    b = torch.minimum(L.x + L.R, torch.as_tensor(hi[:2], device=dev, dtype=torch.float64))
    v = torch.zeros(n, P, 2, device=dev, dtype=torch.float64)
    v[:, 0, 0], v[:, 0, 1], v[:, 1, 0], v[:, 1, 1] = a[:, 0], a[:, 1], b[:, 0], a[:, 1]
    v[:, 2, 0], v[:, 2, 1], v[:, 3, 0], v[:, 3, 1] = b[:, 0], b[:, 1], a[:, 0], b[:, 1]
    cnt = torch.full((n,), 4, device=dev)
    rows, slot = torch.arange(n, device=dev), torch.arange(P, device=dev)[None]
    offs = [(ox, oy) for ox in range(-_OFF, _OFF + 1) for oy in range(-_OFF, _OFF + 1) if (ox, oy) != (0, 0)]
    for ox, oy in sorted(offs, key=lambda o: o[0] ** 2 + o[1] ** 2):
        j, ok = L.near(rows, ox, oy)
        d = L.x[j] - L.x
        ok = ok & (d.norm(dim=1) < 2 * L.R)
        mid = 0.5 * (L.x[j] + L.x)
        f = ((v - mid[:, None]) * d[:, None]).sum(-1)              # > 0: cut off
        live = slot < cnt[:, None]
        cut = live & (f > 0) & ok[:, None]
        if not bool(cut.any()):
            continue
        nxt = torch.where(slot + 1 < cnt[:, None], slot + 1, torch.zeros_like(slot))
        fn = f.gather(1, nxt)
        vn = v.gather(1, nxt[..., None].expand(-1, -1, 2))
        inside, inside_n = f <= 0, fn <= 0
        keep, cross = live & (inside | ~ok[:, None]), live & (inside != inside_n) & ok[:, None]
        t = torch.where(cross, f / torch.where(cross, f - fn, torch.ones_like(f)), torch.zeros_like(f))
        pt = v + t[..., None] * (vn - v)
        num = keep.long() + cross.long()
        at = num.cumsum(1) - num
        new = torch.zeros(n, P + 1, 2, device=dev, dtype=torch.float64)
        for mask, val, shift in ((keep, v, 0), (cross, pt, keep.long())):
            pos = torch.where(mask, at + shift, torch.full_like(at, P))
            new.scatter_(1, pos[..., None].expand(-1, -1, 2), val)
        v, cnt = new[:, :P].contiguous(), num.sum(1)
    return v, cnt


def _rules2():
    """25-point conical product on the unit triangle, 5-point Gauss-Legendre on [0, 1]."""
    g, gw = np.polynomial.legendre.leggauss(5)
    # Gauss-Jacobi(1, 0): Golub-Welsch for the weight (1 - t) on [-1, 1]
    k = np.arange(5, dtype=np.float64)
    diag = -1.0 / ((2 * k + 1) * (2 * k + 3))
    j = np.arange(1, 5, dtype=np.float64)
    off = np.sqrt(j * (j + 1) / (2 * j + 1) ** 2)
    ev, vec = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    u, uw = 0.5 * (1 + ev), 0.25 * 2.0 * vec[0] ** 2
    t, tw = 0.5 * (1 + g), 0.5 * gw
    xi = np.array([(a, b * (1 - a)) for a in u for b in t])
    w = np.array([p * q for p in uw for q in tw])
    return xi, w, t, tw


def _rk2(L, rows, pts):
    """U, dU/dx, dU/dy [cells, points, functions] of the linear RK functions near each cell."""
    r = torch.arange(-_ROFF, _ROFF + 1, device=L.dev)
    oy, ox = [o.reshape(-1) for o in torch.meshgrid(r, r, indexing="ij")]
    j, ok = L.near(rows[:, None], ox[None], oy[None])
    h = 0.5 * L.R
    d = pts[:, :, None] - L.x[j][:, None]                           # [c, q, a, 2]
    dist = d.norm(dim=-1)
    chi = dist / h
    one = torch.where(chi < 1, 1 - 1.5 * chi ** 2 + 0.75 * chi ** 3, 0.25 * (2 - chi).clamp(min=0) ** 3)
    der = torch.where(chi < 1, chi * (2.25 * chi - 3), -0.75 * (2 - chi).clamp(min=0) ** 2)
    live = ok[:, None].to(pts.dtype)
    W = one * live
    g = der * live / torch.where(dist > 0, dist * h, torch.ones_like(dist))
    V = L.V[j][:, None]
    P = torch.cat([torch.ones_like(d[..., :1]), d / h], -1)         # [c, q, a, 3]
    C0 = torch.linalg.inv(torch.einsum("cqa,cqai,cqaj->cqij", V * W, P, P))
    C = C0[..., 0]
    U, grads = W * torch.einsum("cqai,cqi->cqa", P, C), []
    for ax in range(2):
        dP = torch.zeros_like(P)
        dP[..., 1 + ax] = 1.0 / h
        gw = g * d[..., ax]
        T = torch.einsum("cqa,cqai,cqaj->cqij", V * W, dP, P)
        D = T + T.transpose(-1, -2) + torch.einsum("cqa,cqai,cqaj->cqij", V * gw, P, P)
        dC = -torch.einsum("cqij,cqjk,cqk->cqi", C0, D, C)
        grads.append(W * (torch.einsum("cqai,cqi->cqa", dP, C) + torch.einsum("cqai,cqi->cqa", P, dC))
                     + gw * torch.einsum("cqai,cqi->cqa", P, C))
    return U, grads[0], grads[1], j, ok, ox, oy


def _forms2(p, side, dev):
    """Lattice, and the forms of the weak transport equation as [form][n, 9 * 9] over the
    offsets within +-4: M0 Mt Ms G(2) Gt(2) Gs(2) K(xx xy yx yy) S(4), and Q0, Q(2)."""
    L = _Lattice2(p, side, dev)
    n = L.n
    v, cnt = _cells2(L, p.lo, p.hi)
    c = L.x[:, None]
    P = int(cnt.max())
    slot = torch.arange(P, device=dev)[None]
    nxt = torch.where(slot + 1 < cnt[:, None], slot + 1, torch.zeros_like(slot))
    v0 = v[:, :P]
    v1 = v.gather(1, nxt[..., None].expand(-1, -1, 2))
    live = (slot < cnt[:, None]).double()
    e0, e1 = (v0 - c) * live[..., None], (v1 - c) * live[..., None]     # unused slots: the generator
    det = (e0[..., 0] * e1[..., 1] - e0[..., 1] * e1[..., 0]).abs()
    L.V = 0.5 * det.sum(1)
    xi, wt, t, tw = (torch.as_tensor(a, device=dev) for a in _rules2())
    nf, nw, na = 17, 2 * _OFF + 1, (2 * _ROFF + 1) ** 2
    F = torch.zeros(nf, n * nw * nw, device=dev, dtype=torch.float64)
    Q = torch.zeros(3, n, device=dev, dtype=torch.float64)
    st, ss, q = (torch.as_tensor(a, device=dev) for a in (p.sigma_t, p.sigma_s, p.q))
    step = max(1, (1 << 27) // (P * 25 * na * 4))
    for a0 in range(0, n, step):
        rows = torch.arange(a0, min(n, a0 + step), device=dev)
        m = len(rows)
        E0, E1 = e0[rows], e1[rows]
        pts = (c[rows][:, :, None] + E0[:, :, None] * xi[None, None, :, :1] + E1[:, :, None] * xi[None, None, :, 1:])
        w = (det[rows][:, :, None] * wt).reshape(m, -1)
        U, Ux, Uy, j, ok, ox, oy = _rk2(L, rows, pts.reshape(m, -1, 2))
        dx, dy = ox[None, :] - ox[:, None], oy[None, :] - oy[:, None]        # trial minus test
        use = (dx.abs() <= _OFF) & (dy.abs() <= _OFF)
        pos = (j[:, :, None] * nw * nw + ((dy + _OFF) * nw + dx + _OFF)[None]).reshape(m, -1)
        mask = (ok[:, :, None] & ok[:, None, :] & use[None]).reshape(m, -1)
        pos = torch.where(mask, pos, torch.zeros_like(pos)).reshape(-1)
        Vb = L.V[j][:, None, :]

        def add(f, test, trial, weight, scale=None):
            val = torch.einsum("cqa,cqb->cab", weight[..., None] * test, trial) * Vb
            val = torch.where(mask, val.reshape(m, -1), torch.zeros((), device=dev, dtype=torch.float64))
            for k, s in ((f, None),) if scale is None else scale:
                F[k].index_add_(0, pos, (val if s is None else val * s[:, None]).reshape(-1))
        sig = lambda k: ((k[0], None), (k[1], st[rows]), (k[2], ss[rows]))  # noqa: E731
        add(0, U, U, w, sig((0, 1, 2)))
        add(3, Ux, U, w, sig((3, 5, 7)))
        add(4, Uy, U, w, sig((4, 6, 8)))
        for k, (A, B) in enumerate(((Ux, Ux), (Ux, Uy), (Uy, Ux), (Uy, Uy))):
            add(9 + k, A, B, w)
        for k, A in enumerate((U, Ux, Uy)):
            val = torch.where(ok, (w[..., None] * A).sum(1) * q[rows][:, None], torch.zeros((), device=dev, dtype=torch.float64))
            Q[k].index_add_(0, torch.where(ok, j, torch.zeros_like(j)).reshape(-1), val.reshape(-1))
    # box faces: edges whose two ends lie on a face
    for f in range(4):
        ax, at = f // 2, (p.lo if f % 2 == 0 else p.hi)[f // 2]
        on = ((v0[..., ax] - at).abs() < 1e-13) & ((v1[..., ax] - at).abs() < 1e-13) & (live > 0)
        rows, e = on.nonzero(as_tuple=True)
        if len(rows) == 0:
            continue
        A, B = v0[rows, e], v1[rows, e]
        pts = A[:, None] + (B - A)[:, None] * t[None, :, None]
        w = (B - A).norm(dim=1)[:, None] * tw[None]
        U, _, _, j, ok, ox, oy = _rk2(L, rows, pts)
        dx, dy = ox[None, :] - ox[:, None], oy[None, :] - oy[:, None]
        use = ok[:, :, None] & ok[:, None, :] & ((dx.abs() <= _OFF) & (dy.abs() <= _OFF))[None]
        pos = j[:, :, None] * nw * nw + ((dy + _OFF) * nw + dx + _OFF)[None]
        val = torch.einsum("cqa,cqb->cab", w[..., None] * U, U) * L.V[j][:, None, :]
        F[13 + f].index_add_(0, torch.where(use, pos, torch.zeros_like(pos)).reshape(-1),
                             torch.where(use, val, torch.zeros_like(val)).reshape(-1))
    return L, F.view(nf, n, nw * nw), Q


def _offsets():
    return [(k, k % (2 * _OFF + 1) - _OFF, k // (2 * _OFF + 1) - _OFF) for k in range((2 * _OFF + 1) ** 2)]


def _values2(F, p, kappa, tau):
    """Per-direction values of L_m: a function of the offset's forms and Omega."""
    o = torch.as_tensor(p.omega, device=F.device)
    ox, oy = o[:, 0], o[:, 1]
    face = [(-ox).clamp(min=0), ox.clamp(min=0), (-oy).clamp(min=0), oy.clamp(min=0)]

    def at(k):
        g = F[:, :, k, None]
        v = kappa * g[0] + g[1] + ox * ((kappa * tau - 1) * g[3] + tau * g[5]) + oy * ((kappa * tau - 1) * g[4] + tau * g[6])
        v = v + tau * (ox * ox * g[9] + ox * oy * (g[10] + g[11]) + oy * oy * g[12])
        for f in range(4):
            v = v + face[f] * g[13 + f]
        return v
    return at


def _apply2(L, F, p, X):
    X = X.double()
    Y = torch.zeros_like(X)
    at = _values2(F, p, 1.0 / p.dt, 0.5 * L.R)
    rows = torch.arange(L.n, device=L.dev)
    for k, ox, oy in _offsets():
        j, ok = L.near(rows, ox, oy)
        Y += torch.where(ok[:, None], at(k) * X[j], torch.zeros((), device=L.dev, dtype=torch.float64))
    return Y


def _step2(L, F, Q, p):
    """One backward-Euler step from a zero state, by dense elimination."""
    n, tau = L.n, 0.5 * L.R
    at = _values2(F, p, 1.0 / p.dt, tau)
    om, w = torch.as_tensor(p.omega, device=L.dev), torch.as_tensor(p.w, device=L.dev)
    rows = torch.arange(n, device=L.dev)
    near = [(k, *L.near(rows, ox, oy)) for k, ox, oy in _offsets()]
    vals = {k: at(k) for k, _, _ in near}
    total, rhs, keep = torch.eye(n, device=L.dev, dtype=torch.float64), 0.0, []
    for m in range(p.m):
        A = torch.zeros(n, n, device=L.dev, dtype=torch.float64)
        S = torch.zeros_like(A)
        for k, j, ok in near:
            r = rows[ok]
            A[r, j[ok]] = vals[k][r, m]
            S[r, j[ok]] = (F[2, r, k] + tau * (om[m, 0] * F[7, r, k] + om[m, 1] * F[8, r, k])) / (4 * math.pi)
        f = Q[0] + tau * (om[m, 0] * Q[1] + om[m, 1] * Q[2])
        sol = torch.linalg.solve(A, torch.cat([S, f[:, None]], 1))
        keep.append(sol)
        total -= w[m] * sol[:, :n]
        rhs = rhs + w[m] * sol[:, n]
    phi = torch.linalg.solve(total, rhs)
    return torch.stack([s[:, :n] @ phi + s[:, n] for s in keep], 1)


def exact(case, seed):
    """2D: the apply, the set-up's apply and volumes, and a step of up to about a thousand
    points.  3D cells (polyhedra cut by some 250 planes each) and larger or repeated
    steps take plain torch too long."""
    do = case["do"]
    if case["dim"] != 2 or do not in ("apply", "setup", "step") or (do == "step" and case["side"] > 33):
        return None
    p = _problem(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    L, F, Q = _forms2(p, case["side"], dev)
    if do == "step":
        return {"psi": _step2(L, F, Q, p)}
    Y = _apply2(L, F, p, _vectors(case, seed, p.n, p.m))
    if do == "apply":
        return Y
    return {"y": Y, "volume": L.V, "rowptr": None}
