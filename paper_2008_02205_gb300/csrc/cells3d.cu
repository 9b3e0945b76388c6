// 3D integration cells on the device (Sec. 3.1): one warp per point starts
// from the kernel-extent cube cut to the domain box and clips it by the
// bisector half-space of every overlap neighbour, then splits the polyhedron
// into tetrahedra (x_i, c_f, v_k, v_k+1) per face edge and boundary triangles
// (c_f, v_k, v_k+1) per edge of a face on the box (c_f: the face's vertex
// average).  A cut keeps the inside part of every face and closes the
// polyhedron with a new face: the convex hull, in the cutting plane, of the
// vertices on the plane and the points where face edges cross it (monotone
// chain).  Distances within 1e-12 R |x_j - x_i| of a plane count as on it.
//
// The same steps, in the same order and the same arithmetic, as the host
// builder (geometry.cpp); this file is compiled without floating-point
// contraction, so both give the same cells.  Two passes around a scan: the
// first counts each cell's tetrahedra and boundary triangles and records its
// volume, the second writes the elements at the cell's offsets, in cell
// order.  With the cells on the device the whole integration stage of a 3D
// point set runs on the GPU and can be repeated when the points move.
//
// A warp per cell, the polyhedron in shared memory: the vertex tests, the cut of
// every face (positions by warp scans), the merging of points on the plane and their
// sort run over the lanes; sums whose order matters (volume, face centres) and the
// hull's chain keep the host's order.  One thread per cell, its polyhedron in
// global memory, was a chain of dependent loads and took 38 ms a pass whatever the
// number of points (15^3 to 20^3); this one takes 3.2 ms a pass at 15^3, bound by the
// FP64 units (1.6 operations per clock and SM) and the serial parts.
#include "internal.h"

namespace mlpg {
namespace {

constexpr int kMaxF = 64;    // faces of a cell during clipping
constexpr int kMaxV = 384;   // vertices over all faces
constexpr int kMaxOn = 96;   // points on a cutting plane

struct P3 {
    double x, y, z;
};
__device__ __forceinline__ P3 sub(const P3 &a, const P3 &b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double dotp(const P3 &a, const P3 &b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ P3 crossp(const P3 &a, const P3 &b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// faces as vertex runs: face f has vertices v[f0[f] .. f0[f] + nv[f]) and label lab[f]; runs are
// contiguous and in face order; fid: face of each vertex
struct Poly {
    int nf, nvt;
    int f0[kMaxF], nv[kMaxF];
    int32_t lab[kMaxF];
    P3 v[kMaxV];
    uint8_t fid[kMaxV];
};
struct Q2 {
    double u, v;
    int k;
};
// shared memory of one warp
struct CellWork {
    Poly poly[2];
    P3 on[kMaxOn];              // points on the cutting plane, in the order they are met
    Q2 q[kMaxOn], qs[kMaxOn];   // their plane coordinates, then sorted
    int h[2 * kMaxOn];          // hull chains, indices into qs
    uint16_t pos[kMaxV + 1];    // vertices emitted before each vertex of the old polyhedron
    int toff[kMaxF], tface[kMaxF];
};

constexpr unsigned kFull = 0xffffffffu;
__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// convex hull of the np points W.on (merged within dist_tol) in the plane of unit normal nh,
// counter-clockwise about nh, appended to T as a face labelled j; nothing for fewer than three points.
// False on overflow.
__device__ bool plane_hull(CellWork &W, Poly &T, int np, const P3 &nh, double dist_tol, double area_tol, int32_t j,
                           int lane) {
    P3 *pts = W.on;
    int nu = 0;
    for (int k = 0; k < np; ++k) {
        const P3 pk = pts[k];
        bool dup = false;
        for (int u = lane; u < nu; u += 32) {
            const P3 e = sub(pk, pts[u]);
            dup |= sqrt(dotp(e, e)) <= dist_tol;
        }
        dup = __any_sync(kFull, dup);
        if (!dup) {
            if (lane == 0) pts[nu] = pk;   // nu <= k: a point that every lane has read
            ++nu;
        }
        __syncwarp();
    }
    if (nu < 3) return true;
    const P3 t = fabs(nh.x) < 0.6 ? P3{1, 0, 0} : P3{0, 1, 0};
    P3 e1 = sub(t, {nh.x * dotp(t, nh), nh.y * dotp(t, nh), nh.z * dotp(t, nh)});
    const double l = sqrt(dotp(e1, e1));
    e1 = {e1.x / l, e1.y / l, e1.z / l};
    const P3 e2 = crossp(nh, e1);
    for (int k = lane; k < nu; k += 32) W.q[k] = {dotp(pts[k], e1), dotp(pts[k], e2), k};
    __syncwarp();
    for (int k = lane; k < nu; k += 32) {   // stable sort by (u, v): each point's rank
        const Q2 a = W.q[k];
        int r = 0;
        for (int m = 0; m < nu; ++m) {
            const Q2 b = W.q[m];
            const bool less = b.u < a.u || (b.u == a.u && b.v < a.v), eq = b.u == a.u && b.v == a.v;
            r += less || (eq && m < k);
        }
        W.qs[r] = a;
    }
    __syncwarp();
    int m = 0;
    if (lane == 0) {   // monotone chain
        const Q2 *q = W.qs;
        int *h = W.h;
        auto turn = [q](int o, int a, int b) {
            return (q[a].u - q[o].u) * (q[b].v - q[o].v) - (q[a].v - q[o].v) * (q[b].u - q[o].u);
        };
        for (int k = 0; k < nu; ++k) {   // lower chain
            while (m >= 2 && turn(h[m - 2], h[m - 1], k) <= area_tol) --m;
            h[m++] = k;
        }
        for (int k = nu - 1, lo = m + 1; k-- > 0;) {   // upper chain
            while (m >= lo && turn(h[m - 2], h[m - 1], k) <= area_tol) --m;
            h[m++] = k;
        }
    }
    m = __shfl_sync(kFull, m, 0);
    __syncwarp();
    if (m < 4) return true;
    const int n = m - 1, at = T.nvt, f = T.nf;
    if (f >= kMaxF || at + n > kMaxV) return false;
    for (int k = lane; k < n; k += 32) {
        T.v[at + k] = pts[W.qs[W.h[k]].k];
        T.fid[at + k] = (uint8_t)f;
    }
    __syncwarp();
    if (lane == 0) {
        T.f0[f] = at;
        T.nv[f] = n;
        T.lab[f] = j;
        T.nf = f + 1;
        T.nvt = at + n;
    }
    __syncwarp();
    return true;
}

// keep {p : nrm . p <= c}; the new face gets label j.  *cut: the result is in
// T (F is unchanged otherwise).  False on overflow.
__device__ bool clip3(CellWork &W, const Poly &F, Poly &T, bool *cut, const P3 &nrm, double c, double eps,
                      double dist_tol, double area_tol, int32_t j, int lane) {
    const int nvt = F.nvt, nf = F.nf;
    bool any_out = false;
    for (int k = lane; k < nvt; k += 32) any_out |= dotp(nrm, F.v[k]) - c > eps;
    *cut = __any_sync(kFull, any_out);
    if (!*cut) return true;
    // what every vertex k emits: itself when inside, then the crossing of its edge
    auto edge = [&](int k, P3 *p, P3 *r, bool *keep, bool *on, bool *cross) {
        const int f = F.fid[k], kn = k + 1 - F.f0[f] == F.nv[f] ? F.f0[f] : k + 1;
        *p = F.v[k];
        const P3 qq = F.v[kn];
        const double sp = dotp(nrm, *p) - c, sq = dotp(nrm, qq) - c;
        *keep = sp <= eps;
        *on = *keep && sp >= -eps;
        *cross = (sp < -eps && sq > eps) || (sp > eps && sq < -eps);
        if (*cross) {
            const double t = sp / (sp - sq);
            *r = {p->x + t * (qq.x - p->x), p->y + t * (qq.y - p->y), p->z + t * (qq.z - p->z)};
        }
    };
    int carry = 0, ocarry = 0;
    for (int k0 = 0; k0 < nvt; k0 += 32) {
        const int k = k0 + lane;
        P3 p{0, 0, 0}, r{0, 0, 0};
        bool keep = false, on = false, cross = false;
        if (k < nvt) edge(k, &p, &r, &keep, &on, &cross);
        const int e = keep + cross, w = on + cross;
        const int es = warp_incl_scan(e, lane), ws = warp_incl_scan(w, lane);
        if (k < nvt) W.pos[k] = (uint16_t)(carry + es - e);
        int at = ocarry + ws - w;
        if (on && at < kMaxOn) W.on[at] = p;
        at += on;
        if (cross && at < kMaxOn) W.on[at] = r;
        carry += __shfl_sync(kFull, es, 31);
        ocarry += __shfl_sync(kFull, ws, 31);
    }
    if (lane == 0) W.pos[nvt] = (uint16_t)carry;
    __syncwarp();
    if (ocarry > kMaxOn) return false;
    // faces that keep at least three vertices, at their new places
    int vcarry = 0, fcarry = 0;
    bool over = false;
    for (int f0 = 0; f0 < nf; f0 += 32) {
        const int f = f0 + lane;
        const int tot = f < nf ? W.pos[F.f0[f] + F.nv[f]] - W.pos[F.f0[f]] : 0;
        const bool kept = tot >= 3;
        const int vs = warp_incl_scan(kept ? tot : 0, lane), fs = warp_incl_scan(kept, lane);
        const int to = vcarry + vs - (kept ? tot : 0), nfi = fcarry + fs - kept;
        over |= to + tot > kMaxV;
        if (f < nf) {
            W.toff[f] = kept ? to : -1;
            W.tface[f] = nfi;
            if (kept && nfi < kMaxF) {
                T.f0[nfi] = to;
                T.nv[nfi] = tot;
                T.lab[nfi] = F.lab[f];
            }
        }
        vcarry += __shfl_sync(kFull, vs, 31);
        fcarry += __shfl_sync(kFull, fs, 31);
    }
    if (__any_sync(kFull, over) || fcarry > kMaxF) return false;
    if (lane == 0) {
        T.nf = fcarry;
        T.nvt = vcarry;
    }
    __syncwarp();
    for (int k = lane; k < nvt; k += 32) {
        const int f = F.fid[k];
        if (W.toff[f] < 0) continue;
        P3 p, r;
        bool keep, on, cross;
        edge(k, &p, &r, &keep, &on, &cross);
        int at = W.toff[f] + W.pos[k] - W.pos[F.f0[f]];
        const uint8_t id = (uint8_t)W.tface[f];
        if (keep) {
            T.v[at] = p;
            T.fid[at++] = id;
        }
        if (cross) {
            T.v[at] = r;
            T.fid[at] = id;
        }
    }
    __syncwarp();
    const double ln = sqrt(dotp(nrm, nrm));
    return plane_hull(W, T, ocarry, {nrm.x / ln, nrm.y / ln, nrm.z / ln}, dist_tol, area_tol, j, lane);
}

// largest squared distance of a vertex from g
__device__ double reach2(const Poly &F, const P3 &g, int lane) {
    double r2 = 0.0;
    for (int k = lane; k < F.nvt; k += 32) {
        const P3 e = sub(F.v[k], g);
        r2 = fmax(r2, dotp(e, e));
    }
    for (int o = 16; o > 0; o >>= 1) r2 = fmax(r2, __shfl_xor_sync(kFull, r2, o));
    return r2;
}

struct Cell3Args {
    int64_t n;
    const double *x, *R;
    const int32_t *rowptr, *col;
    double lo[3], hi[3];
    int32_t *ntet, *ntri;          // [n] counts (first pass)
    double *vol;                   // [n]
    const int32_t *tptr, *bptr;    // [n + 1] offsets (second pass)
    int32_t *tet_owner, *tri_owner, *tri_face;
    double *tet_v, *tri_v;
    int *flag;                     // bit 128: a cell overflowed its buffers or is empty
    int32_t *bad;                  // smallest failing point
};

template <bool WRITE>
__global__ void __launch_bounds__(32) k_cells_3d(Cell3Args A) {
    extern __shared__ __align__(16) unsigned char cell_smem[];
    CellWork &W = *reinterpret_cast<CellWork *>(cell_smem);
    const int lane = threadIdx.x;
    const int64_t i = blockIdx.x;
    // the current polyhedron and the next, swapped after every cut
    Poly *pf = &W.poly[0], *pt = &W.poly[1];
    Poly &F0 = *pf;   // the starting polyhedron
    const P3 g{A.x[3 * i], A.x[3 * i + 1], A.x[3 * i + 2]};
    const double r = A.R[i];
    double b0[3] = {g.x - r, g.y - r, g.z - r}, b1[3] = {g.x + r, g.y + r, g.z + r};
    bool dlo[3], dhi[3];
    for (int a = 0; a < 3; ++a) {
        dlo[a] = b0[a] <= A.lo[a];
        dhi[a] = b1[a] >= A.hi[a];
        if (dlo[a]) b0[a] = A.lo[a];
        if (dhi[a]) b1[a] = A.hi[a];
    }
    // the six faces of the box, counter-clockwise about their outward normals
    if (lane == 0) {
        const int quad[6][4] = {{0, 4, 6, 2}, {1, 3, 7, 5}, {0, 1, 5, 4}, {2, 6, 7, 3}, {0, 2, 3, 1}, {4, 5, 7, 6}};
        F0.nf = 6;
        F0.nvt = 24;
        for (int f = 0; f < 6; ++f) {
            const bool dom = (f & 1) ? dhi[f / 2] : dlo[f / 2];
            F0.f0[f] = 4 * f;
            F0.nv[f] = 4;
            F0.lab[f] = dom ? -(f + 1) : kLabelExtent;
            for (int k = 0; k < 4; ++k) {
                const int c = quad[f][k];
                F0.v[4 * f + k] = {(c & 1) ? b1[0] : b0[0], (c & 2) ? b1[1] : b0[1], (c & 4) ? b1[2] : b0[2]};
                F0.fid[4 * f + k] = (uint8_t)f;
            }
        }
    }
    __syncwarp();
    bool okc = true;
    // A bisector at distance |d| / 2 from g cuts nothing while every vertex lies closer to g:
    // then d . v - c <= |d| (|v - g| - |d| / 2) < 0, so the vertex scan of clip3 would find no
    // vertex beyond the plane.  Such planes are skipped on the polyhedron's reach (its largest
    // vertex distance from g), with a relative margin of 1e-9 far above the rounding of either
    // test: the cells stay those of the scan, bit for bit.
    // Two rounds over the neighbours, each in column order: those closer than the kernel
    // extent first (they carve the cell to about its final size), then the rest, most of
    // which the reach test skips.  The host builder takes the same order.
    double r2 = reach2(*pf, g, lane);
    bool empty = false;
    for (int round = 0; round < 2 && okc && !empty; ++round) {
        const int32_t p1 = A.rowptr[i + 1];
        // 32 neighbours at a time: the round's own that the reach may let through, in order
        for (int32_t pb = A.rowptr[i]; pb < p1 && okc && !empty; pb += 32) {
            P3 xl{0, 0, 0};
            int32_t jl = (int32_t)i;
            double d2l = 0.0;
            bool mine = false;
            if (pb + lane < p1) {
                jl = A.col[pb + lane];
                xl = {A.x[3 * (int64_t)jl], A.x[3 * (int64_t)jl + 1], A.x[3 * (int64_t)jl + 2]};
                const P3 d = sub(xl, g);
                d2l = dotp(d, d);
                mine = jl != i && (d2l < r * r) == (round == 0);
            }
            for (unsigned todo = __ballot_sync(kFull, mine); todo && okc && !empty; todo &= todo - 1) {
                const int src = __ffs((int)todo) - 1;
                const int32_t j = __shfl_sync(kFull, jl, src);
                const double d2 = __shfl_sync(kFull, d2l, src);
                if (r2 < 0.25 * d2 * (1.0 - 1e-9)) continue;
                const P3 xj{__shfl_sync(kFull, xl.x, src), __shfl_sync(kFull, xl.y, src), __shfl_sync(kFull, xl.z, src)};
                const P3 d = sub(xj, g);
                const P3 mid{0.5 * (xj.x + g.x), 0.5 * (xj.y + g.y), 0.5 * (xj.z + g.z)};
                const double dl = sqrt(d2);
                bool cut = false;
                okc = clip3(W, *pf, *pt, &cut, d, dotp(d, mid), 1e-12 * r * dl, 1e-12 * r, 1e-13 * r * r, j, lane);
                if (cut && okc) {
                    Poly *tmp = pf;
                    pf = pt;
                    pt = tmp;
                    r2 = reach2(*pf, g, lane);
                    empty = pf->nf == 0;
                }
            }
        }
    }
    // tetrahedra (g, c_f, v_k, v_k+1): face centres into the other polyhedron's vertices, terms of the
    // volume into its labels' place after them; both sums in the host's order
    const Poly &F = *pf;
    const int nvt = okc ? F.nvt : 0, nf = okc ? F.nf : 0;
    P3 *cfs = pt->v;
    double *term = reinterpret_cast<double *>(pt->v + kMaxF);   // kMaxV doubles in 3 (kMaxV - kMaxF)
    static_assert(3 * (kMaxV - kMaxF) >= kMaxV, "the volume's terms fit behind the face centres");
    for (int f = lane; f < nf; f += 32) {
        const int nv = F.nv[f];
        const P3 *fv = F.v + F.f0[f];
        P3 cf{0, 0, 0};
        for (int k = 0; k < nv; ++k) cf = {cf.x + fv[k].x, cf.y + fv[k].y, cf.z + fv[k].z};
        cfs[f] = {cf.x / nv, cf.y / nv, cf.z / nv};
    }
    __syncwarp();
    const int32_t to = WRITE ? A.tptr[i] : 0, bo = WRITE ? A.bptr[i] : 0;
    int nb = 0;
    for (int k0 = 0; k0 < nvt; k0 += 32) {
        const int k = k0 + lane;
        bool bnd = false;
        if (k < nvt) {
            const int f = F.fid[k], kn = k + 1 - F.f0[f] == F.nv[f] ? F.f0[f] : k + 1;
            const P3 cf = cfs[f], a = F.v[k], b = F.v[kn];
            bnd = F.lab[f] < 0 && F.lab[f] != kLabelExtent;
            if (!WRITE) {
                term[k] = fabs(dotp(sub(cf, g), crossp(sub(a, g), sub(b, g)))) / 6.0;
            } else {
                const P3 pts[3] = {cf, a, b};
                const int64_t e = (int64_t)to + k;
                A.tet_owner[e] = (int32_t)i;
                for (int c = 0; c < 3; ++c) {
                    A.tet_v[9 * e + 3 * c] = pts[c].x;
                    A.tet_v[9 * e + 3 * c + 1] = pts[c].y;
                    A.tet_v[9 * e + 3 * c + 2] = pts[c].z;
                }
            }
        }
        const unsigned bb = __ballot_sync(kFull, bnd);
        if (WRITE && bnd) {
            const int f = F.fid[k], kn = k + 1 - F.f0[f] == F.nv[f] ? F.f0[f] : k + 1;
            const P3 pts[3] = {cfs[f], F.v[k], F.v[kn]};
            const int64_t eb = (int64_t)bo + nb + __popc(bb & ((1u << lane) - 1u));
            A.tri_owner[eb] = (int32_t)i;
            A.tri_face[eb] = -F.lab[f] - 1;
            for (int c = 0; c < 3; ++c) {
                A.tri_v[9 * eb + 3 * c] = pts[c].x;
                A.tri_v[9 * eb + 3 * c + 1] = pts[c].y;
                A.tri_v[9 * eb + 3 * c + 2] = pts[c].z;
            }
        }
        nb += __popc(bb);
    }
    __syncwarp();
    if (!WRITE && lane == 0) {
        double vol = 0.0;
        for (int k = 0; k < nvt; ++k) vol += term[k];
        const bool bad = !okc || !(vol > 0.0);
        if (bad) {
            atomicOr(A.flag, 128);
            atomicMin(A.bad, (int32_t)i);
        }
        A.ntet[i] = bad ? 0 : nvt;
        A.ntri[i] = bad ? 0 : nb;
        A.vol[i] = vol;
    }
}

// exclusive scans of two count arrays into out[n + 1], out2[n + 1] (one block)
__global__ void k_scan_two(int64_t n, const int32_t *__restrict__ c1, const int32_t *__restrict__ c2,
                           int32_t *__restrict__ o1, int32_t *__restrict__ o2) {
    __shared__ long long p1[1024], p2[1024];
    const int t = threadIdx.x, T = blockDim.x;
    const int64_t chunk = (n + T - 1) / T, a = t * chunk, b = min(n, a + chunk);
    long long s1 = 0, s2 = 0;
    for (int64_t k = a; k < b; ++k) {
        s1 += c1[k];
        s2 += c2[k];
    }
    p1[t] = s1;
    p2[t] = s2;
    __syncthreads();
    for (int off = 1; off < T; off <<= 1) {
        const long long v1 = t >= off ? p1[t - off] : 0, v2 = t >= off ? p2[t - off] : 0;
        __syncthreads();
        p1[t] += v1;
        p2[t] += v2;
        __syncthreads();
    }
    long long r1 = p1[t] - s1, r2 = p2[t] - s2;
    for (int64_t k = a; k < b; ++k) {
        o1[k] = (int32_t)r1;
        o2[k] = (int32_t)r2;
        r1 += c1[k];
        r2 += c2[k];
    }
    if (t == T - 1) {
        o1[n] = (int32_t)p1[T - 1];
        o2[n] = (int32_t)p2[T - 1];
    }
}

}  // namespace

// The cells of all points, the tetrahedra and boundary triangles into the
// context's element arrays (tet_owner, tet_v, tri_owner, tri_face, tri_v), the
// volumes into V.
mlpg_status run_cells_3d(mlpg_ctx *ctx) {
    const int64_t n = ctx->n;
    cudaStream_t s = ctx->stream;
    int32_t *ntet, *ntri, *bad, *tptr, *bptr;
    MLPG_TRY(dalloc(ctx, &ntet, n));
    MLPG_TRY(dalloc(ctx, &ntri, n));
    MLPG_TRY(dalloc(ctx, &tptr, n + 1));
    MLPG_TRY(dalloc(ctx, &bptr, n + 1));
    MLPG_TRY(dalloc(ctx, &bad, 1));
    if (!ctx->d_flag) MLPG_TRY(dalloc(ctx, &ctx->d_flag, 1));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), s));
    const int32_t big = 0x7fffffff;
    CU(ctx, cudaMemcpyAsync(bad, &big, sizeof(int32_t), cudaMemcpyHostToDevice, s));
    Cell3Args a{};
    a.x = ctx->x; a.R = ctx->R; a.rowptr = ctx->rowptr; a.col = ctx->col;
    for (int d = 0; d < 3; ++d) { a.lo[d] = ctx->opt.lo[d]; a.hi[d] = ctx->opt.hi[d]; }
    a.ntet = ntet; a.ntri = ntri; a.vol = ctx->V; a.tptr = tptr; a.bptr = bptr;
    a.flag = ctx->d_flag; a.bad = bad;
    auto pass = [&](bool write) -> mlpg_status {
        a.tet_owner = ctx->tet_owner; a.tri_owner = ctx->tri_owner; a.tri_face = ctx->tri_face;
        a.tet_v = ctx->tet_v; a.tri_v = ctx->tri_v;
        a.n = n;
        if (write) {
            CU(ctx, cudaFuncSetAttribute(k_cells_3d<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CellWork)));
            k_cells_3d<true><<<(unsigned)n, 32, sizeof(CellWork), s>>>(a);
        } else {
            CU(ctx, cudaFuncSetAttribute(k_cells_3d<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CellWork)));
            k_cells_3d<false><<<(unsigned)n, 32, sizeof(CellWork), s>>>(a);
        }
        CU_LAUNCH(ctx);
        return MLPG_OK;
    };
    MLPG_TRY(pass(false));
    k_scan_two<<<1, 1024, 0, s>>>(n, ntet, ntri, tptr, bptr);
    CU_LAUNCH(ctx);
    int32_t tot[2] = {0, 0}, badi = big;
    int flag = 0;
    CU(ctx, cudaMemcpyAsync(&tot[0], tptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaMemcpyAsync(&tot[1], bptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaMemcpyAsync(&flag, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaMemcpyAsync(&badi, bad, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaStreamSynchronize(s));
    if (flag & 128) return set_err(ctx, MLPG_ERR_GEOMETRY, "empty or oversized cell at point " + std::to_string(badi));
    ctx->ntet = tot[0];
    ctx->nbtri = tot[1];
    ctx->nvq = 8 * ctx->ntet;
    ctx->nbq = 4 * ctx->nbtri;
    MLPG_TRY(dalloc(ctx, &ctx->tet_owner, ctx->ntet));
    MLPG_TRY(dalloc(ctx, &ctx->tet_v, 9 * ctx->ntet));
    MLPG_TRY(dalloc(ctx, &ctx->tri_owner, ctx->nbtri + 1));
    MLPG_TRY(dalloc(ctx, &ctx->tri_face, ctx->nbtri + 1));
    MLPG_TRY(dalloc(ctx, &ctx->tri_v, 9 * ctx->nbtri + 9));
    MLPG_TRY(pass(true));
    return MLPG_OK;
}

}  // namespace mlpg
