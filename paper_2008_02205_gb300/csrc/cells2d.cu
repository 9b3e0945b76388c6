// 2D integration cells on the device (Sec. 3.1): one warp per point clips
// the kernel-extent square, cut to the domain box, by the perpendicular
// bisector of every overlap neighbour.  Two passes over the cells: the first
// counts vertices and boundary edges and records the area, the second (after a
// scan of the counts) writes every cell's vertices and edge labels at its
// offset.  The cells depend only on the points and extents, so the whole
// integration stage can rerun on the device when the points move.
//
// Lane k of the warp holds vertex k: a bisector is tested against all vertices at
// once, and a cut moves the kept vertices and the two new ones to their places by
// ballots.  One thread per cell kept its polygon in local memory and walked it vertex
// by vertex, and computed every neighbour's bisector: the FP64 units take 20 clocks per
// warp instruction and SM, however few lanes are active (0.97 ms a pass at 128^2
// points).  Here a lane computes the bisector of its own neighbour, 32 at once, and
// those beyond the polygon's reach are dropped by one ballot: 0.72 ms.
#include "internal.h"

namespace mlpg {
namespace {

constexpr int kMaxPoly = 32;   // polygon vertices during clipping

struct CellArgs {
    int64_t n;
    const double *x, *R;
    const int32_t *rowptr, *col;
    double lo0, lo1, hi0, hi1;
    int32_t *nvert;        // [n]
    int32_t *nbedge;       // [n]
    double *vol;           // [n]
    const int32_t *cptr;   // [n + 1] (second pass)
    double *verts;         // [2 * total] (second pass)
    int32_t *labels;       // [total] (second pass)
    int *flag;             // bit 64: a cell needs more than kMaxPoly vertices or is empty
    int32_t *bad;          // smallest failing point
};

constexpr int kCellWarps = 4;   // cells per CTA

template <bool WRITE>
__global__ void __launch_bounds__(32 * kCellWarps) k_cells_2d(CellArgs A) {
    static_assert(kMaxPoly == 32, "one vertex per lane");
    __shared__ double sx[kCellWarps][kMaxPoly], sy[kCellWarps][kMaxPoly];
    __shared__ int32_t sl[kCellWarps][kMaxPoly];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)kCellWarps + warp;
    if (i >= A.n) return;
    constexpr unsigned full = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const double xi = A.x[2 * i], yi = A.x[2 * i + 1], r = A.R[i];
    double x0 = xi - r, x1 = xi + r, y0 = yi - r, y1 = yi + r;
    const bool bx0 = x0 <= A.lo0, bx1 = x1 >= A.hi0, by0 = y0 <= A.lo1, by1 = y1 >= A.hi1;
    x0 = bx0 ? A.lo0 : x0;
    x1 = bx1 ? A.hi0 : x1;
    y0 = by0 ? A.lo1 : y0;
    y1 = by1 ? A.hi1 : y1;
    // counter-clockwise from the lower-left corner; the label is that of the edge starting there
    double px = lane == 1 || lane == 2 ? x1 : x0, py = lane >= 2 ? y1 : y0;
    int32_t lab = lane == 0 ? (by0 ? -3 : kLabelExtent)            // face 2 (-y)
                  : lane == 1 ? (bx1 ? -2 : kLabelExtent)          // face 1 (+x)
                  : lane == 2 ? (by1 ? -4 : kLabelExtent)          // face 3 (+y)
                              : (bx0 ? -1 : kLabelExtent);         // face 0 (-x)
    int nv = 4;
    bool overflow = false;
    // the polygon's reach: its largest squared vertex distance, rounded up to FP32 (the maximum of the floats'
    // bits).  A bisector at distance |d| / 2 cuts nothing while every vertex lies closer than that; the margin
    // of 1e-9 in hl is far above the rounding of either test.
    auto reach2 = [&]() {
        const double dx = px - xi, dy = py - yi;
        const unsigned u = lane < nv ? __float_as_uint(__double2float_ru(dx * dx + dy * dy)) : 0u;
        return (double)__uint_as_float(__reduce_max_sync(full, u));
    };
    double r2 = reach2();
    const int32_t p1 = A.rowptr[i + 1];
    for (int32_t pb = A.rowptr[i]; pb < p1 && nv > 0; pb += 32) {   // 32 neighbours' data at a time
        // each lane its neighbour's bisector; one that lies farther than the polygon's reach cuts nothing
        int32_t jl = (int32_t)i;
        double al = 0.0, bl = 0.0, cl = 0.0, hl = 0.0;
        if (pb + lane < p1) {
            jl = A.col[pb + lane];
            const double xj = A.x[2 * (int64_t)jl], yj = A.x[2 * (int64_t)jl + 1];
            al = xj - xi;
            bl = yj - yi;
            cl = al * 0.5 * (xj + xi) + bl * 0.5 * (yj + yi);
            hl = 0.25 * (al * al + bl * bl) * (1.0 - 1e-9);
        }
        unsigned todo = __ballot_sync(full, jl != i && hl <= r2);
        while (todo && nv > 0) {
            const int q = __ffs((int)todo) - 1;
            const int32_t j = __shfl_sync(full, jl, q);
            const double a = __shfl_sync(full, al, q), b = __shfl_sync(full, bl, q), c = __shfl_sync(full, cl, q);
            todo &= todo - 1;
            // keep {p : a p.x + b p.y <= c}; edges created by the cut get label j
            const double s = a * px + b * py - c;
            if (!__any_sync(full, lane < nv && s > 0.0)) continue;
            const int k1 = lane + 1 >= nv ? 0 : lane + 1;
            const double sq = __shfl_sync(full, s, k1), qx = __shfl_sync(full, px, k1), qy = __shfl_sync(full, py, k1);
            const bool pin = s <= 0.0, keep = lane < nv && pin, cross = lane < nv && pin != (sq <= 0.0);
            const unsigned mk = __ballot_sync(full, keep), mc = __ballot_sync(full, cross);
            const int total = __popc(mk) + __popc(mc);
            if (total > kMaxPoly) {   // (warp-uniform)
                overflow = true;
                nv = 0;
                break;
            }
            int at = __popc(mk & below) + __popc(mc & below);
            if (keep) {
                sx[warp][at] = px;
                sy[warp][at] = py;
                sl[warp][at++] = lab;
            }
            if (cross) {
                const double t = s / (s - sq);
                sx[warp][at] = px + t * (qx - px);
                sy[warp][at] = py + t * (qy - py);
                sl[warp][at] = pin ? j : lab;
            }
            nv = total;
            __syncwarp();
            if (lane < nv) {
                px = sx[warp][lane];
                py = sy[warp][lane];
                lab = sl[warp][lane];
            }
            __syncwarp();
            r2 = reach2();
            todo &= __ballot_sync(full, hl <= r2);
        }
    }
    const int k1 = lane + 1 >= nv ? 0 : lane + 1;
    const double term = px * __shfl_sync(full, py, k1) - __shfl_sync(full, px, k1) * py;
    double area2 = 0.0;
    for (int k = 0; k < nv; ++k) area2 += __shfl_sync(full, term, k);
    const int nb = __popc(__ballot_sync(full, lane < nv && lab < 0 && lab != kLabelExtent));
    if (!WRITE) {
        if (lane != 0) return;
        const bool bad = overflow || nv < 3 || !(area2 > 0.0);
        if (bad) {
            atomicOr(A.flag, 64);
            atomicMin(A.bad, (int32_t)i);
        }
        A.nvert[i] = bad ? 0 : nv;
        A.nbedge[i] = bad ? 0 : nb;
        A.vol[i] = 0.5 * area2;
        return;
    }
    const int32_t o = A.cptr[i];
    if (A.cptr[i + 1] - o != nv) return;   // unchanged between passes (same arithmetic)
    if (lane < nv) {
        A.verts[2 * (o + lane)] = px;
        A.verts[2 * (o + lane) + 1] = py;
        A.labels[o + lane] = lab;
    }
}

// exclusive scan of n counts into out[n + 1] and the two totals (one block)
__global__ void k_scan_counts(int64_t n, const int32_t *__restrict__ cnt, const int32_t *__restrict__ cnt2,
                              int32_t *__restrict__ out, long long *__restrict__ totals) {
    __shared__ long long part[1024];
    __shared__ long long part2[1024];
    const int t = threadIdx.x, T = blockDim.x;
    const int64_t chunk = (n + T - 1) / T, a = t * chunk, b = min(n, a + chunk);
    long long s = 0, s2 = 0;
    for (int64_t k = a; k < b; ++k) {
        s += cnt[k];
        s2 += cnt2[k];
    }
    part[t] = s;
    part2[t] = s2;
    __syncthreads();
    for (int off = 1; off < T; off <<= 1) {
        long long v = t >= off ? part[t - off] : 0, v2 = t >= off ? part2[t - off] : 0;
        __syncthreads();
        part[t] += v;
        part2[t] += v2;
        __syncthreads();
    }
    long long run = part[t] - s;
    for (int64_t k = a; k < b; ++k) {
        out[k] = (int32_t)run;
        run += cnt[k];
    }
    if (t == T - 1) {
        out[n] = (int32_t)part[T - 1];
        totals[0] = part[T - 1];
        totals[1] = part2[T - 1];
    }
}

}  // namespace

mlpg_status run_cells_2d(mlpg_ctx *ctx, int tri_points, int line_points) {
    const int64_t n = ctx->n;
    cudaStream_t s = ctx->stream;
    int32_t *nvert, *nbedge, *bad;
    long long *totals;
    MLPG_TRY(dalloc(ctx, &nvert, n));
    MLPG_TRY(dalloc(ctx, &nbedge, n));
    MLPG_TRY(dalloc(ctx, &bad, 1));
    MLPG_TRY(dalloc(ctx, &totals, 2));
    MLPG_TRY(dalloc(ctx, &ctx->cptr, n + 1));
    if (!ctx->d_flag) MLPG_TRY(dalloc(ctx, &ctx->d_flag, 1));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), s));
    const int32_t big = 0x7fffffff;
    CU(ctx, cudaMemcpyAsync(bad, &big, sizeof(int32_t), cudaMemcpyHostToDevice, s));
    CellArgs a{};
    a.n = n; a.x = ctx->x; a.R = ctx->R; a.rowptr = ctx->rowptr; a.col = ctx->col;
    a.lo0 = ctx->opt.lo[0]; a.lo1 = ctx->opt.lo[1]; a.hi0 = ctx->opt.hi[0]; a.hi1 = ctx->opt.hi[1];
    a.nvert = nvert; a.nbedge = nbedge; a.vol = ctx->V; a.cptr = ctx->cptr; a.flag = ctx->d_flag; a.bad = bad;
    k_cells_2d<false><<<(unsigned)((n + kCellWarps - 1) / kCellWarps), 32 * kCellWarps, 0, s>>>(a);
    CU_LAUNCH(ctx);
    k_scan_counts<<<1, 1024, 0, s>>>(n, nvert, nbedge, ctx->cptr, totals);
    CU_LAUNCH(ctx);
    long long tot[2] = {0, 0};
    int flag = 0;
    int32_t badi = big;
    CU(ctx, cudaMemcpyAsync(tot, totals, sizeof(tot), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaMemcpyAsync(&flag, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaMemcpyAsync(&badi, bad, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaStreamSynchronize(s));
    if (flag & 64) return set_err(ctx, MLPG_ERR_GEOMETRY, "empty or oversized cell at point " + std::to_string(badi));
    ctx->nverts = tot[0];
    ctx->nvq = tot[0] * tri_points;
    ctx->nbq = tot[1] * line_points;
    MLPG_TRY(dalloc(ctx, &ctx->verts, 2 * ctx->nverts));
    MLPG_TRY(dalloc(ctx, &ctx->labels, ctx->nverts));
    a.verts = ctx->verts;
    a.labels = ctx->labels;
    k_cells_2d<true><<<(unsigned)((n + kCellWarps - 1) / kCellWarps), 32 * kCellWarps, 0, s>>>(a);
    CU_LAUNCH(ctx);
    return MLPG_OK;
}

}  // namespace mlpg
