// Reproducing-kernel functions at quadrature points and the quadrature-
// outermost integration of the SUPG transport forms (Sec. 2.2, Sec. 3.2,
// Alg. 1, Eq. weak-transport), 2D.
//
// The linear functions (the default) have a kernel of their own, k_assemble_2d_lin.
// Orders 0 and 2: one CTA integrates one cell i.  The functions that can reach the cell (at
// most MLPG_MAX_CELL_FUNCS, drawn from the overlap row of i) are staged in
// shared memory.  Quadrature points are generated in the kernel from the cell
// polygon: fan triangles (x_i, v_k, v_{k+1}) with the conical-product rule
// mapped by x = p0 + (p1 - p0) xi1 + (p2 - p0) xi2 (App. A), and Gauss-Legendre
// points on edges that lie on the domain boundary.  Chunks of points are
// evaluated one point per thread (RK moment matrix, Cholesky, corrections and
// derivatives, FP64), their values written to a shared table, and every thread
// then accumulates its own unordered function pairs a <= b over the chunk (the
// sums of both entries (a, b) and (b, a): the mass, diagonal stiffness and
// face forms are symmetric, the mixed stiffness forms are each other's
// transposes, and both gradient forms use the same point values).  The
// per-cell sums are added into the CSR pattern at the end.
// Materials are constant over the cell, so sigma-weighted forms are the cell
// sums times sigma_t(i), sigma_s(i).
#include <algorithm>
#include <cmath>

#include "fixed_sum.cuh"
#include "internal.h"

namespace mlpg {

namespace {

constexpr int kMaxS = MLPG_MAX_CELL_FUNCS;
constexpr int kThreads = 512;
constexpr int kMaxTri = 64;   // reference triangle rule size cap
constexpr int kMaxLine = 16;

__constant__ double c_tri_xi[2 * kMaxTri];
__constant__ double c_tri_w[kMaxTri];
__constant__ double c_line_t[kMaxLine];
__constant__ double c_line_w[kMaxLine];

__device__ __forceinline__ double spline_w(double chi) {
    if (chi < 1.0) return 1.0 - chi * chi * (1.5 - 0.75 * chi);
    if (chi < 2.0) { double t = 2.0 - chi; return 0.25 * t * t * t; }
    return 0.0;
}
__device__ __forceinline__ double spline_dw(double chi) {
    if (chi < 1.0) return chi * (2.25 * chi - 3.0);
    if (chi < 2.0) { double t = 2.0 - chi; return -0.75 * t * t; }
    return 0.0;
}

// RK functions at (px, py) for the S staged functions; basis P = [1, d/s].
// Writes U, Ux, Uy (zero outside the support); returns false when the moment
// matrix is not positive definite.
__device__ bool rk_point(double px, double py, double s, int S, const double *fx, const double *fy,
                         const double *fR, const double *fV, double *U, double *Ux, double *Uy,
                         int stride) {
    double M[3][3] = {{0}}, Dx[3][3] = {{0}}, Dy[3][3] = {{0}};
    const double is = 1.0 / s;
    for (int a = 0; a < S; ++a) {
        double dx = px - fx[a], dy = py - fy[a];
        double r = sqrt(dx * dx + dy * dy);
        if (!(r < fR[a])) continue;
        double h = 0.5 * fR[a], chi = r / h;
        double W = spline_w(chi);
        double g = r > 0.0 ? spline_dw(chi) / (r * h) : 0.0;
        double Wx = g * dx, Wy = g * dy, v = fV[a];
        double P[3] = {1.0, dx * is, dy * is};
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                double pp = P[i] * P[j];
                M[i][j] += v * W * pp;
                double ex = ((i == 1) * P[j] + (j == 1) * P[i]) * is;
                double ey = ((i == 2) * P[j] + (j == 2) * P[i]) * is;
                Dx[i][j] += v * (ex * W + pp * Wx);
                Dy[i][j] += v * (ey * W + pp * Wy);
            }
    }
    // Cholesky M = L L^T
    double L00 = M[0][0];
    if (!(L00 > 0.0)) return false;
    L00 = sqrt(L00);
    double L10 = M[1][0] / L00, L20 = M[2][0] / L00;
    double d1 = M[1][1] - L10 * L10;
    if (!(d1 > 1e-14 * M[1][1])) return false;
    double L11 = sqrt(d1);
    double L21 = (M[2][1] - L20 * L10) / L11;
    double d2 = M[2][2] - L20 * L20 - L21 * L21;
    if (!(d2 > 1e-14 * M[2][2])) return false;
    double L22 = sqrt(d2);
    auto solve = [&](double b0, double b1, double b2, double *o) {
        double y0 = b0 / L00, y1 = (b1 - L10 * y0) / L11, y2 = (b2 - L20 * y0 - L21 * y1) / L22;
        o[2] = y2 / L22;
        o[1] = (y1 - L21 * o[2]) / L11;
        o[0] = (y0 - L10 * o[1] - L20 * o[2]) / L00;
    };
    double C[3], Cx[3], Cy[3];
    solve(1.0, 0.0, 0.0, C);
    solve(-(Dx[0][0] * C[0] + Dx[0][1] * C[1] + Dx[0][2] * C[2]),
          -(Dx[1][0] * C[0] + Dx[1][1] * C[1] + Dx[1][2] * C[2]),
          -(Dx[2][0] * C[0] + Dx[2][1] * C[1] + Dx[2][2] * C[2]), Cx);
    solve(-(Dy[0][0] * C[0] + Dy[0][1] * C[1] + Dy[0][2] * C[2]),
          -(Dy[1][0] * C[0] + Dy[1][1] * C[1] + Dy[1][2] * C[2]),
          -(Dy[2][0] * C[0] + Dy[2][1] * C[1] + Dy[2][2] * C[2]), Cy);
    for (int a = 0; a < S; ++a) {
        double dx = px - fx[a], dy = py - fy[a];
        double r = sqrt(dx * dx + dy * dy);
        double u = 0.0, ux = 0.0, uy = 0.0;
        if (r < fR[a]) {
            double h = 0.5 * fR[a], chi = r / h;
            double W = spline_w(chi);
            double g = r > 0.0 ? spline_dw(chi) / (r * h) : 0.0;
            double P1 = dx * is, P2 = dy * is;
            double PC = C[0] + P1 * C[1] + P2 * C[2];
            u = W * PC;
            ux = W * (C[1] * is + Cx[0] + P1 * Cx[1] + P2 * Cx[2]) + PC * g * dx;
            uy = W * (C[2] * is + Cy[0] + P1 * Cy[1] + P2 * Cy[2]) + PC * g * dy;
        }
        U[a * stride] = u;
        Ux[a * stride] = ux;
        Uy[a * stride] = uy;
    }
    return true;
}

// RK functions of order ORD (0 or 2; the linear ones are in k_assemble_2d_lin) at
// (px, py), into the shared table (U, Ux, Uy at [a * stride]): the basis is every
// monomial of xi = (p - x_j)/s up to degree ORD, ordered 1, xi_x, xi_y, xi_x^2,
// xi_x xi_y, xi_y^2.  The first pass stores W and its gradient in the table slots so
// that the second does not repeat the square roots; support tests compare squared
// distances.  Returns the support mask (bit a set when function a is supported), or 0
// when the moment matrix is not positive definite.
template <int ORD>
__device__ uint64_t rk_point_gen(double px, double py, double s, int S, const double *fx, const double *fy,
                                 const double *fR2, const double *finvh, const double *fV, double *U, double *Ux,
                                 double *Uy, int stride) {
    static_assert(ORD == 0 || ORD == 2, "the linear functions have kernels of their own");
    constexpr int NP = ORD == 0 ? 1 : 6;
    double M[NP][NP], Dx[NP][NP], Dy[NP][NP];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int j = 0; j < NP; ++j) M[i][j] = Dx[i][j] = Dy[i][j] = 0.0;
    const double is = 1.0 / s;
    // basis and its x, y derivatives at offset (dx, dy)
    auto basis = [&](double dx, double dy, double *P, double *Px, double *Py) {
        const double ex = dx * is, ey = dy * is;
        P[0] = 1.0; Px[0] = 0.0; Py[0] = 0.0;
        if constexpr (ORD == 2) {
            P[1] = ex; Px[1] = is; Py[1] = 0.0;
            P[2] = ey; Px[2] = 0.0; Py[2] = is;
            P[3] = ex * ex; Px[3] = 2.0 * ex * is; Py[3] = 0.0;
            P[4] = ex * ey; Px[4] = ey * is; Py[4] = ex * is;
            P[5] = ey * ey; Px[5] = 0.0; Py[5] = 2.0 * ey * is;
        }
    };
    uint64_t mask = 0;
    for (int a = 0; a < S; ++a) {
        const double dx = px - fx[a], dy = py - fy[a];
        const double r2 = dx * dx + dy * dy;
        if (!(r2 < fR2[a])) {
            U[a * stride] = 0.0;
            Ux[a * stride] = 0.0;
            Uy[a * stride] = 0.0;
            continue;
        }
        mask |= uint64_t(1) << a;
        const double ir = r2 > 0.0 ? rsqrt(r2) : 0.0;
        const double chi = r2 * ir * finvh[a];
        const double W = spline_w(chi), g = spline_dw(chi) * finvh[a] * ir;
        const double Wx = g * dx, Wy = g * dy, v = fV[a];
        U[a * stride] = W;
        Ux[a * stride] = Wx;
        Uy[a * stride] = Wy;
        double P[NP], Px[NP], Py[NP];
        basis(dx, dy, P, Px, Py);
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const double pp = P[i] * P[j];
                M[i][j] += v * W * pp;
                Dx[i][j] += v * ((Px[i] * P[j] + P[i] * Px[j]) * W + pp * Wx);
                Dy[i][j] += v * ((Py[i] * P[j] + P[i] * Py[j]) * W + pp * Wy);
            }
    }
    // Cholesky M = L L^T
    double L[NP][NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        double d = M[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
        if (!(d > 1e-14 * M[j][j])) return 0;
        L[j][j] = sqrt(d);
#pragma unroll
        for (int i = j + 1; i < NP; ++i) {
            double t = M[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[i][k] * L[j][k];
            L[i][j] = t / L[j][j];
        }
    }
    auto solve = [&](double *b) {   // in place: b <- M^{-1} b
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            double t = b[i];
#pragma unroll
            for (int k = 0; k < i; ++k) t -= L[i][k] * b[k];
            b[i] = t / L[i][i];
        }
#pragma unroll
        for (int i = NP - 1; i >= 0; --i) {
            double t = b[i];
#pragma unroll
            for (int k = i + 1; k < NP; ++k) t -= L[k][i] * b[k];
            b[i] = t / L[i][i];
        }
    };
    double C[NP], Cx[NP], Cy[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) C[i] = i == 0 ? 1.0 : 0.0;
    solve(C);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        double tx = 0.0, ty = 0.0;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            tx += Dx[i][j] * C[j];
            ty += Dy[i][j] * C[j];
        }
        Cx[i] = -tx;
        Cy[i] = -ty;
    }
    solve(Cx);
    solve(Cy);
    for (uint64_t bits = mask; bits; bits &= bits - 1) {
        const int a = __ffsll((long long)bits) - 1;
        const double W = U[a * stride], Wx = Ux[a * stride], Wy = Uy[a * stride];
        double P[NP], Px[NP], Py[NP];
        basis(px - fx[a], py - fy[a], P, Px, Py);
        double PC = 0.0, dxC = 0.0, dyC = 0.0, PCx = 0.0, PCy = 0.0;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            PC += P[i] * C[i];
            dxC += Px[i] * C[i];
            dyC += Py[i] * C[i];
            PCx += P[i] * Cx[i];
            PCy += P[i] * Cy[i];
        }
        U[a * stride] = W * PC;
        Ux[a * stride] = W * (dxC + PCx) + PC * Wx;
        Uy[a * stride] = W * (dyC + PCy) + PC * Wy;
    }
    return mask;
}

__device__ int find_col(const int32_t *__restrict__ col, int32_t lo, int32_t hi, int32_t key) {
    hi -= 1;
    while (lo <= hi) {
        int32_t mid = (lo + hi) >> 1;
        int32_t c = col[mid];
        if (c == key) return mid;
        if (c < key) lo = mid + 1; else hi = mid - 1;
    }
    return -1;
}

struct AsmArgs {
    int64_t n, nnz;
    const double *x, *R, *V, *sig_t, *sig_s, *q;
    const int32_t *rowptr, *col, *cptr, *labels;
    const double *verts;
    int ntri, nline;
    double *mats, *vecs;
    int *flag;
};

// mats layout: 0 M0, 1 Mt, 2 Ms, 3-4 G, 5-6 Gt, 7-8 Gs, 9-12 K (xx, xy, yx, yy), 13-16 S_f
// ORD: RK order (0 or 2); MAXS: functions reaching one cell (<= 64, one mask word);
// CHUNK: quadrature points per RK pass.
template <int ORD, int MAXS, int CHUNK>
__global__ void __launch_bounds__(kThreads, 1) k_assemble_2d(AsmArgs A) {
    // unordered pairs a <= b of the staged functions: M0, K^xx, K^yy and the face forms are
    // symmetric, K^yx(a, b) = K^xy(b, a), and both G(a, b) and G(b, a) come from the same
    // point values, so one pass over a <= b fills both entries (a, b) and (b, a)
    constexpr int kMaxS = MAXS, kChunk = CHUNK, kPairs = MAXS * (MAXS + 1) / 2;
    constexpr int kPPT = (kPairs + kThreads - 1) / kThreads;
    constexpr int kAcc = 11;   // running sums per unordered pair
    static_assert(MAXS <= 64 && CHUNK <= kThreads, "one 64-bit support mask per point");
    const int64_t i = blockIdx.x;
    __shared__ double fx[kMaxS], fy[kMaxS], fR[kMaxS], fV[kMaxS], fR2[kMaxS], finvh[kMaxS];
    __shared__ uint64_t tMask[kChunk];
    __shared__ int32_t fidx[kMaxS];
    __shared__ uint8_t pairA[kPairs], pairB[kPairs];
    __shared__ int S;
    __shared__ int face_slot[2];
    extern __shared__ double tab[];  // [6][kChunk][kMaxS] + [kChunk] weights + [kChunk] face
    double *tU = tab, *tUx = tU + kChunk * kMaxS, *tUy = tUx + kChunk * kMaxS;
    double *tW = tUy + kChunk * kMaxS;                 // weight per point
    int *tF = (int *)(tW + kChunk);                    // face slot (-1 volume)

    const int tid = threadIdx.x;
    const double xi = A.x[2 * i], yi = A.x[2 * i + 1];
    const int32_t c0 = A.cptr[i], nv = A.cptr[i + 1] - c0;
    if (tid == 0) {
        // radius of the cell around its generator and the boundary faces it touches
        double rc = 0.0;
        int nf = 0;
        face_slot[0] = face_slot[1] = -1;
        for (int k = 0; k < nv; ++k) {
            double dx = A.verts[2 * (c0 + k)] - xi, dy = A.verts[2 * (c0 + k) + 1] - yi;
            rc = fmax(rc, sqrt(dx * dx + dy * dy));
            int32_t L = A.labels[c0 + k];
            if (L < 0 && L != kLabelExtent) {
                int f = -L - 1;
                if (face_slot[0] != f && face_slot[1] != f) {
                    if (nf < 2) face_slot[nf] = f;
                    ++nf;
                }
            }
        }
        if (nf > 2) atomicOr(A.flag, 4);
        int s = 0;
        for (int32_t p = A.rowptr[i]; p < A.rowptr[i + 1]; ++p) {
            int32_t j = A.col[p];
            double dx = A.x[2 * j] - xi, dy = A.x[2 * j + 1] - yi;
            if (sqrt(dx * dx + dy * dy) < A.R[j] + rc * (1.0 + 1e-12)) {
                if (s < kMaxS) {
                    fidx[s] = j;
                    fx[s] = A.x[2 * j];
                    fy[s] = A.x[2 * j + 1];
                    fR[s] = A.R[j];
                    fR2[s] = A.R[j] * A.R[j];
                    finvh[s] = 2.0 / A.R[j];
                    fV[s] = A.V[j];
                }
                ++s;
            }
        }
        if (s > kMaxS) atomicOr(A.flag, 2);
        S = s > kMaxS ? kMaxS : s;
    }
    __syncthreads();
    const int nS = S, nP = nS * (nS + 1) / 2;
    const double scale = 0.5 * A.R[i];
    // unordered pair p = (a, b), a <= b, row by row of the upper triangle
    if (tid < nS) {
        const int a = tid, p0 = a * nS - a * (a - 1) / 2;
        for (int b = a; b < nS; ++b) {
            pairA[p0 + b - a] = (uint8_t)a;
            pairB[p0 + b - a] = (uint8_t)b;
        }
    }
    // pairs owned by this thread: p = tid + k * kThreads.  Their running sums live in
    // shared memory, sacc[f][p] (one owner per p):
    //   0 M0, 1-2 G(a, b), 3-4 G(b, a), 5 K^xx, 6 K^xy(a, b), 7 K^yx(a, b), 8 K^yy, 9-10 faces
    double *sacc = tab + 3 * kChunk * kMaxS + kChunk + kChunk / 2 + 1;
    for (int p = tid; p < kPairs; p += kThreads)
#pragma unroll
        for (int f = 0; f < kAcc; ++f) sacc[f * kPairs + p] = 0.0;
    double vq0 = 0.0, vqx = 0.0, vqy = 0.0, vb0 = 0.0, vb1 = 0.0;  // vectors for a = tid

    // count boundary points of this cell
    int nbe = 0;
    for (int k = 0; k < nv; ++k) {
        int32_t L = A.labels[c0 + k];
        nbe += (L < 0 && L != kLabelExtent);
    }
    const int nvol = nv * A.ntri, ntot = nvol + nbe * A.nline;
    for (int base = 0; base < ntot; base += kChunk) {
        const int cnt = min(kChunk, ntot - base);
        if (tid < cnt) {
            int k = base + tid;
            double px, py, wq;
            int fslot = -1;
            if (k < nvol) {
                int e = k / A.ntri, r = k - e * A.ntri;
                int e1 = (e + 1 == nv) ? 0 : e + 1;
                double ax = A.verts[2 * (c0 + e)] - xi, ay = A.verts[2 * (c0 + e) + 1] - yi;
                double bx = A.verts[2 * (c0 + e1)] - xi, by = A.verts[2 * (c0 + e1) + 1] - yi;
                double det = fabs(ax * by - ay * bx);
                px = xi + ax * c_tri_xi[2 * r] + bx * c_tri_xi[2 * r + 1];
                py = yi + ay * c_tri_xi[2 * r] + by * c_tri_xi[2 * r + 1];
                wq = c_tri_w[r] * det;
            } else {
                int kb = k - nvol, eb = kb / A.nline, r = kb - eb * A.nline;
                // eb-th boundary edge of the cell
                int e = -1, c = -1;
                for (int t = 0; t < nv; ++t) {
                    int32_t L = A.labels[c0 + t];
                    if (L < 0 && L != kLabelExtent && ++c == eb) { e = t; break; }
                }
                int e1 = (e + 1 == nv) ? 0 : e + 1;
                double p0x = A.verts[2 * (c0 + e)], p0y = A.verts[2 * (c0 + e) + 1];
                double dx = A.verts[2 * (c0 + e1)] - p0x, dy = A.verts[2 * (c0 + e1) + 1] - p0y;
                double s01 = 0.5 * (c_line_t[r] + 1.0);
                px = p0x + dx * s01;
                py = p0y + dy * s01;
                wq = c_line_w[r] * 0.5 * sqrt(dx * dx + dy * dy);
                int f = -A.labels[c0 + e] - 1;
                fslot = (f == face_slot[0]) ? 0 : 1;
            }
            const uint64_t mk = rk_point_gen<ORD>(px, py, scale, nS, fx, fy, fR2, finvh, fV, tU + tid, tUx + tid,
                                                  tUy + tid, kChunk);
            if (!mk) atomicOr(A.flag, 1);
            tMask[tid] = mk;
            tW[tid] = wq;
            tF[tid] = fslot;
        }
        __syncthreads();
        for (int qk = 0; qk < cnt; ++qk) {
            const double wq = tW[qk];
            const int fs = tF[qk];
            const uint64_t mk = tMask[qk];
#pragma unroll
            for (int k = 0; k < kPPT; ++k) {
                int p = tid + k * kThreads;
                if (p >= nP) break;
                const int a = pairA[p], b = pairB[p];
                if (!((mk >> a) & (mk >> b) & 1)) continue;   // both functions must be supported here
                double ua = tU[a * kChunk + qk];
                double uax = tUx[a * kChunk + qk], uay = tUy[a * kChunk + qk];
                double ub = tU[b * kChunk + qk];
                double ubx = tUx[b * kChunk + qk], uby = tUy[b * kChunk + qk];
                if (fs < 0) {
                    double wa = wq * ua, wax = wq * uax, way = wq * uay;
                    sacc[0 * kPairs + p] += wa * ub;
                    sacc[1 * kPairs + p] += wax * ub;
                    sacc[2 * kPairs + p] += way * ub;
                    sacc[3 * kPairs + p] += wa * ubx;
                    sacc[4 * kPairs + p] += wa * uby;
                    sacc[5 * kPairs + p] += wax * ubx;
                    sacc[6 * kPairs + p] += wax * uby;
                    sacc[7 * kPairs + p] += way * ubx;
                    sacc[8 * kPairs + p] += way * uby;
                } else {
                    sacc[(9 + fs) * kPairs + p] += wq * ua * ub;
                }
            }
            if (tid < nS) {
                double ua = tU[tid * kChunk + qk];
                if (fs < 0) {
                    vq0 += wq * ua;
                    vqx += wq * tUx[tid * kChunk + qk];
                    vqy += wq * tUy[tid * kChunk + qk];
                } else if (fs == 0) {
                    vb0 += wq * ua;
                } else {
                    vb1 += wq * ua;
                }
            }
        }
        __syncthreads();
    }
    // scatter into the pattern: entry (a, b) and, for a != b, entry (b, a)
    const double st = A.sig_t[i], ss = A.sig_s[i], qi = A.q[i];
    const int64_t nnz = A.nnz, n = A.n;
    auto put = [&](int32_t ra, int32_t cb, double v, double m0, double gx, double gy, double kxx, double kxy,
                   double kyx, double kyy, double f0, double f1) {
        int pos = find_col(A.col, A.rowptr[ra], A.rowptr[ra + 1], cb);
        if (pos < 0) {
            atomicOr(A.flag, 8);
            return;
        }
        m0 *= v;
        atomicAdd(&A.mats[0 * nnz + pos], m0);
        atomicAdd(&A.mats[1 * nnz + pos], st * m0);
        atomicAdd(&A.mats[2 * nnz + pos], ss * m0);
        gx *= v;
        gy *= v;
        atomicAdd(&A.mats[3 * nnz + pos], gx);
        atomicAdd(&A.mats[4 * nnz + pos], gy);
        atomicAdd(&A.mats[5 * nnz + pos], st * gx);
        atomicAdd(&A.mats[6 * nnz + pos], st * gy);
        atomicAdd(&A.mats[7 * nnz + pos], ss * gx);
        atomicAdd(&A.mats[8 * nnz + pos], ss * gy);
        atomicAdd(&A.mats[9 * nnz + pos], kxx * v);
        atomicAdd(&A.mats[10 * nnz + pos], kxy * v);
        atomicAdd(&A.mats[11 * nnz + pos], kyx * v);
        atomicAdd(&A.mats[12 * nnz + pos], kyy * v);
        if (face_slot[0] >= 0 && f0 != 0.0) atomicAdd(&A.mats[(13 + face_slot[0]) * nnz + pos], f0 * v);
        if (face_slot[1] >= 0 && f1 != 0.0) atomicAdd(&A.mats[(13 + face_slot[1]) * nnz + pos], f1 * v);
    };
#pragma unroll
    for (int k = 0; k < kPPT; ++k) {
        int p = tid + k * kThreads;
        if (p >= nP) break;
        const int a = pairA[p], b = pairB[p];
        double acc[kAcc];
        bool any = false;
#pragma unroll
        for (int f = 0; f < kAcc; ++f) {
            acc[f] = sacc[f * kPairs + p];
            any |= acc[f] != 0.0;
        }
        if (!any) continue;
        // (a, b): trial function b carries V_b; (b, a): G from the (b, a) sums, K^xy and K^yx swap
        put(fidx[a], fidx[b], fV[b], acc[0], acc[1], acc[2], acc[5], acc[6], acc[7], acc[8], acc[9], acc[10]);
        if (a != b)
            put(fidx[b], fidx[a], fV[a], acc[0], acc[3], acc[4], acc[5], acc[7], acc[6], acc[8], acc[9], acc[10]);
    }
    if (tid < nS) {
        int32_t a = fidx[tid];
        if (vq0 != 0.0) atomicAdd(&A.vecs[a], qi * vq0);
        if (vqx != 0.0) atomicAdd(&A.vecs[n + a], qi * vqx);
        if (vqy != 0.0) atomicAdd(&A.vecs[2 * n + a], qi * vqy);
        if (face_slot[0] >= 0 && vb0 != 0.0) atomicAdd(&A.vecs[(3 + face_slot[0]) * n + a], vb0);
        if (face_slot[1] >= 0 && vb1 != 0.0) atomicAdd(&A.vecs[(3 + face_slot[1]) * n + a], vb1);
    }
}

// ---------------------------------------------------------------------------
// Volume and surface forms with the linear RK functions (the default): one CTA per
// cell, its points in chunks of at most 64 (one mask word per function).  Per chunk:
//   1. each function's point mask and each point's function list (distances in
//      FP32 from the generator, FP64 where that could decide wrongly);
//   2. RK functions, two lanes per point over the point's own list (about 13 of the
//      35 functions that reach the cell); the derivative moments are the third-order
//      moments of the kernel's radial derivative (9 sums instead of 12);
//   3. the table sqrt(w) (U, U_x, U_y) in fixed point, 54 bits below each function's
//      largest U and largest derivative in the chunk;
//   4. every unordered pair a <= b sums the nine products over the points both
//      support, in 64-bit integers (fixed_sum.cuh), and adds them to the pattern's
//      upper entry; G(b, a) goes to six buffers of its own, and k_mirror_2d fills the lower
//      entries (M0, K and S are each other's transposes) and applies the volumes V_b.
// Points on box edges follow in chunks of their own, in FP64 (S_f and B_f only).
//
// What bounds it: the FP64 units (1.6 operations per clock and SM), in the RK
// functions; before, every warp of a cell ran twelve FP64 operations for each point
// at which any of its 32 pairs was supported, and the RK functions one point per thread
// on 64 of 512 threads.  128^2 points: 40.4 -> 9.9 ms (FP64 pipe 78 % busy).
// ---------------------------------------------------------------------------
constexpr int kLinThreads = 128, kLinPts = 64;
constexpr int kLinEntries = 2048;   // table entries (points x functions) of 24 bytes: four CTAs per SM

__global__ void __launch_bounds__(kLinThreads, 4) k_assemble_2d_lin(AsmArgs A, double *__restrict__ gt) {
    __shared__ double fx[kMaxS], fy[kMaxS], fR2[kMaxS], finvh[kMaxS], fV[kMaxS];
    __shared__ float ffx[kMaxS], ffy[kMaxS], ffR2[kMaxS], fslack[kMaxS], qfx[kLinPts], qfy[kLinPts];
    __shared__ double qx[kLinPts], qy[kLinPts], qsw[kLinPts];
    __shared__ int qfs[kLinPts], pcnt[kLinPts];
    __shared__ int32_t fidx[kMaxS];
    __shared__ uint64_t fmask[kMaxS];
    __shared__ uint8_t plist[kLinPts][kMaxS];
    __shared__ int wcnt[kLinThreads / 32];
    __shared__ int S_sh;
    __shared__ int16_t xu[kMaxS], xd[kMaxS];   // exponents of each function's largest values in the chunk
    extern __shared__ __align__(16) double lin_tab[];
    const int64_t i = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double xi = A.x[2 * i], yi = A.x[2 * i + 1];
    const int32_t c0 = A.cptr[i], nv = A.cptr[i + 1] - c0;
    const double *vt = A.verts + 2 * (int64_t)c0;
    // radius of the cell around its generator, the boundary edges and the faces it touches (every thread)
    double rc2 = 0.0;
    int nbe = 0, nf = 0, face_slot[2] = {-1, -1};
    for (int k = 0; k < nv; ++k) {
        const int32_t L = A.labels[c0 + k];
        if (L < 0 && L != kLabelExtent) {
            const int f = -L - 1;
            ++nbe;
            if (face_slot[0] != f && face_slot[1] != f) {
                if (nf == 0) face_slot[0] = f;
                else if (nf == 1) face_slot[1] = f;
                ++nf;
            }
        }
    }
    for (int k = lane; k < nv; k += 32) {
        const double dx = vt[2 * k] - xi, dy = vt[2 * k + 1] - yi;
        rc2 = fmax(rc2, dx * dx + dy * dy);
    }
    for (int o = 16; o > 0; o >>= 1) rc2 = fmax(rc2, __shfl_xor_sync(0xffffffffu, rc2, o));
    const double rc = sqrt(rc2);
    if (tid == 0) {
        S_sh = 0;
        if (nf > 2) atomicOr(A.flag, 4);
    }
    __syncthreads();
    // the functions that can reach the cell, in overlap-row order (ascending)
    const int32_t r0 = A.rowptr[i], rl = A.rowptr[i + 1] - r0;
    for (int base = 0; base < rl; base += kLinThreads) {
        const int c = base + tid;
        bool in = false;
        int32_t j = 0;
        double xj = 0.0, yj = 0.0, Rj = 0.0;
        if (c < rl) {
            j = A.col[r0 + c];
            xj = A.x[2 * (int64_t)j];
            yj = A.x[2 * (int64_t)j + 1];
            Rj = A.R[j];
            const double dx = xj - xi, dy = yj - yi;
            in = sqrt(dx * dx + dy * dy) < Rj + rc * (1.0 + 1e-12);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        if (lane == 0) wcnt[warp] = __popc(bal);
        __syncthreads();
        int off = S_sh;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        const int slot = off + __popc(bal & ((1u << lane) - 1u));
        if (in && slot < kMaxS) {
            fidx[slot] = j;
            fx[slot] = xj;
            fy[slot] = yj;
            fR2[slot] = Rj * Rj;
            finvh[slot] = 2.0 / Rj;
            fV[slot] = A.V[j];
            const float dx = (float)(xj - xi), dy = (float)(yj - yi), r2 = (float)Rj * (float)Rj;
            ffx[slot] = dx;
            ffy[slot] = dy;
            ffR2[slot] = r2;
            // coordinates rounded to 2^-24 of at most a few R: 1e-4 is far outside
            fslack[slot] = 1e-4f * (dx * dx + dy * dy + r2);
        }
        __syncthreads();
        if (tid == 0)
            for (int w = 0; w < kLinThreads / 32; ++w) S_sh += wcnt[w];
        __syncthreads();
    }
    const int S = S_sh;
    if (S > kMaxS) {   // (block-uniform) too many functions reach the cell
        if (tid == 0) atomicOr(A.flag, 2);
        return;
    }
    const double s = 0.5 * A.R[i], is = 1.0 / s;
    const int nP = S * (S + 1) / 2;
    const int nvol = nv * A.ntri, ntot = nvol + nbe * A.nline;
    const int cap = min(kLinPts, kLinEntries / S);
    const int nvc = (nvol + cap - 1) / cap, vstep = (nvol + nvc - 1) / nvc;   // even volume chunks
    double vq0 = 0.0, vqx = 0.0, vqy = 0.0, vb0 = 0.0, vb1 = 0.0;   // vectors of function tid
    const double st = A.sig_t[i], ss = A.sig_s[i];
    const int64_t nnz = A.nnz, n = A.n;
    for (int base = 0; base < ntot;) {
        const bool vol = base < nvol;
        const int P = vol ? min(vstep, nvol - base) : min(cap, ntot - base);
        double *tabu = lin_tab;                                            // [P][S] u
        double2 *tabd = reinterpret_cast<double2 *>(lin_tab + ((P * S + 1) & ~1));   // [P][S] (u_x, u_y)
        if (tid < P) {
            const int k = base + tid;
            double dx, dy, wq;   // relative to the generator
            int fs = -1;
            if (vol) {
                const int e = k / A.ntri, r = k - e * A.ntri, e1 = e + 1 == nv ? 0 : e + 1;
                const double ax = vt[2 * e] - xi, ay = vt[2 * e + 1] - yi, bx = vt[2 * e1] - xi, by = vt[2 * e1 + 1] - yi;
                dx = ax * c_tri_xi[2 * r] + bx * c_tri_xi[2 * r + 1];
                dy = ay * c_tri_xi[2 * r] + by * c_tri_xi[2 * r + 1];
                wq = c_tri_w[r] * fabs(ax * by - ay * bx);
                qx[tid] = xi + dx;
                qy[tid] = yi + dy;
            } else {
                const int kb = k - nvol, eb = kb / A.nline, r = kb - eb * A.nline;
                int e = -1, c = -1;   // eb-th boundary edge of the cell
                for (int t = 0; t < nv; ++t) {
                    const int32_t L = A.labels[c0 + t];
                    if (L < 0 && L != kLabelExtent && ++c == eb) { e = t; break; }
                }
                const int e1 = e + 1 == nv ? 0 : e + 1;
                const double p0x = vt[2 * e], p0y = vt[2 * e + 1], ex = vt[2 * e1] - p0x, ey = vt[2 * e1 + 1] - p0y;
                const double s01 = 0.5 * (c_line_t[r] + 1.0);
                qx[tid] = p0x + ex * s01;
                qy[tid] = p0y + ey * s01;
                wq = c_line_w[r] * 0.5 * sqrt(ex * ex + ey * ey);
                dx = qx[tid] - xi;
                dy = qy[tid] - yi;
                fs = -A.labels[c0 + e] - 1 == face_slot[0] ? 0 : 1;
            }
            qfx[tid] = (float)dx;
            qfy[tid] = (float)dy;
            qsw[tid] = sqrt(wq);
            qfs[tid] = fs;
        }
        for (int k = tid; k < P * S; k += kLinThreads) {
            tabu[k] = 0.0;
            tabd[k] = make_double2(0.0, 0.0);
        }
        __syncthreads();
        // 1. masks: four lanes per function
        for (int f0 = 0; f0 < S; f0 += kLinThreads / 4) {
            const int a = f0 + (tid >> 2);
            unsigned lo = 0, hi = 0;
            if (a < S) {
                const float ax = ffx[a], ay = ffy[a], R2 = ffR2[a], slack = fslack[a];
                for (int p = tid & 3; p < P; p += 4) {
                    const float dx = qfx[p] - ax, dy = qfy[p] - ay, r2 = dx * dx + dy * dy;
                    bool sup = r2 < R2;
                    if (!(fabsf(r2 - R2) > slack)) {   // close, or beyond FP32's range
                        const double ex = qx[p] - fx[a], ey = qy[p] - fy[a];
                        sup = ex * ex + ey * ey < fR2[a];
                    }
                    if (p < 32) lo |= (unsigned)sup << p;
                    else hi |= (unsigned)sup << (p - 32);
                }
            }
            lo |= __shfl_xor_sync(0xffffffffu, lo, 1);
            hi |= __shfl_xor_sync(0xffffffffu, hi, 1);
            lo |= __shfl_xor_sync(0xffffffffu, lo, 2);
            hi |= __shfl_xor_sync(0xffffffffu, hi, 2);
            if (a < S && (tid & 3) == 0) fmask[a] = (uint64_t)hi << 32 | lo;
        }
        __syncthreads();
        if (tid < P) {
            int c = 0;
            for (int a = 0; a < S; ++a)
                if ((fmask[a] >> tid) & 1) plist[tid][c++] = (uint8_t)a;
            pcnt[tid] = c;
        }
        __syncthreads();
        // 2. RK functions: two lanes per point, 16 points per warp
        for (int p0 = warp * 16; p0 < P; p0 += kLinThreads / 2) {
            const int p = min(p0 + (lane >> 1), P - 1), l2 = lane & 1;   // spare lanes repeat the last point
            const bool mine = p0 + (lane >> 1) < P;
            const int cnt = pcnt[p];
            const double px = qx[p], py = qy[p];
            double m[6], t[9];
#pragma unroll
            for (int k = 0; k < 6; ++k) m[k] = 0.0;
#pragma unroll
            for (int k = 0; k < 9; ++k) t[k] = 0.0;
            for (int k = l2; k < cnt; k += 2) {
                const int a = plist[p][k];
                const double dx = px - fx[a], dy = py - fy[a], r2 = dx * dx + dy * dy;
                const double ir = r2 > 0.0 ? rsqrt(r2) : 0.0, ih = finvh[a], chi = r2 * ir * ih;
                const double W = spline_w(chi), g = spline_dw(chi) * ih * ir, v = fV[a];
                if (mine) tabd[p * S + a] = make_double2(W, g);
                const double aw = v * W, bw = v * g * s, X = dx * is, Y = dy * is;
                const double ax = aw * X, ay = aw * Y;
                m[0] += aw; m[1] += ax; m[2] += ay;
                m[3] += ax * X; m[4] += ax * Y; m[5] += ay * Y;
                const double bx = bw * X, by = bw * Y, bxx = bx * X, bxy = bx * Y, byy = by * Y;
                t[0] += bx; t[1] += by; t[2] += bxx; t[3] += bxy; t[4] += byy;
                t[5] += bxx * X; t[6] += bxx * Y; t[7] += bxy * Y; t[8] += byy * Y;
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) m[k] += __shfl_xor_sync(0xffffffffu, m[k], 1);
#pragma unroll
            for (int k = 0; k < 9; ++k) t[k] += __shfl_xor_sync(0xffffffffu, t[k], 1);
            // M = L L^T with reciprocal pivots
            bool ok = m[0] > 0.0;
            const double i0 = rsqrt(m[0]), L10 = m[1] * i0, L20 = m[2] * i0;
            const double d1 = m[3] - L10 * L10;
            ok = ok && d1 > 1e-14 * m[3];
            const double i1 = rsqrt(d1), L21 = (m[4] - L20 * L10) * i1;
            const double d2 = m[5] - L20 * L20 - L21 * L21;
            ok = ok && d2 > 1e-14 * m[5];
            const double i2 = rsqrt(d2);
            auto solve = [&](double b0, double b1, double b2, double *r) {
                const double y0 = b0 * i0, y1 = (b1 - L10 * y0) * i1, y2 = (b2 - L20 * y0 - L21 * y1) * i2;
                r[2] = y2 * i2;
                r[1] = (y1 - L21 * r[2]) * i1;
                r[0] = (y0 - L10 * r[1] - L20 * r[2]) * i0;
            };
            double C[3], Cx[3], Cy[3];
            solve(1.0, 0.0, 0.0, C);
            // C_c = -M^-1 D_c C, D_c C [i] = ((i == c) + m_i C_c) / s + sum_j T_c[i][j] C_j (M C = e_1 takes the
            // first term's sum); T_c[i][j] the third-order moments
            solve(-(m[0] * C[1] * is + t[0] * C[0] + t[2] * C[1] + t[3] * C[2]),
                  -((1.0 + m[1] * C[1]) * is + t[2] * C[0] + t[5] * C[1] + t[6] * C[2]),
                  -(m[2] * C[1] * is + t[3] * C[0] + t[6] * C[1] + t[7] * C[2]), Cx);
            solve(-(m[0] * C[2] * is + t[1] * C[0] + t[3] * C[1] + t[4] * C[2]),
                  -(m[1] * C[2] * is + t[3] * C[0] + t[6] * C[1] + t[7] * C[2]),
                  -((1.0 + m[2] * C[2]) * is + t[4] * C[0] + t[7] * C[1] + t[8] * C[2]), Cy);
            if (!ok && mine && l2 == 0) atomicOr(A.flag, 1);
            const double sw = qsw[p], gx = C[1] * is + Cx[0], gy = C[2] * is + Cy[0];
            for (int k = l2; k < cnt && mine; k += 2) {
                const int a = plist[p][k];
                const double dx = px - fx[a], dy = py - fy[a], X = dx * is, Y = dy * is;
                const double2 wg = tabd[p * S + a];
                const double W = wg.x * sw, PC = C[0] + X * C[1] + Y * C[2], h = PC * (wg.y * sw);
                const double u = W * PC;
                const double ux = W * (gx + X * Cx[1] + Y * Cx[2]) + h * dx, uy = W * (gy + X * Cy[1] + Y * Cy[2]) + h * dy;
                tabu[p * S + a] = ok ? u : 0.0;
                tabd[p * S + a] = ok ? make_double2(ux, uy) : make_double2(0.0, 0.0);
            }
        }
        __syncthreads();
        if (tid < S) {   // vectors and scales, before the table changes to fixed point
            unsigned mx0 = 0, mx1 = 0;   // high words of the largest |sqrt(w) u|, |sqrt(w) du|
            for (uint64_t bits = fmask[tid]; bits; bits &= bits - 1) {
                const int p = __ffsll((long long)bits) - 1;
                const double sw = qsw[p], u = sw * tabu[p * S + tid];
                if (vol) {
                    const double2 d = tabd[p * S + tid];
                    vq0 += u;
                    vqx += sw * d.x;
                    vqy += sw * d.y;
                    mx0 = max(mx0, abs_hiword(tabu[p * S + tid]));
                    mx1 = max(mx1, max(abs_hiword(d.x), abs_hiword(d.y)));
                } else if (qfs[p] == 0) {
                    vb0 += u;
                } else {
                    vb1 += u;
                }
            }
            xu[tid] = (int16_t)top_exp(mx0);
            xd[tid] = (int16_t)top_exp(mx1);
        }
        // 3. fixed point, in place
        int2 *iu = reinterpret_cast<int2 *>(tabu);
        int4 *id = reinterpret_cast<int4 *>(tabd);
        if (vol) {
            __syncthreads();
            for (int k = tid; k < P * S; k += kLinThreads) {
                const int p = k / S, a = k - p * S;
                if (!((fmask[a] >> p) & 1)) continue;   // zero already
                const double u = tabu[k];
                const double2 d = tabd[k];
                const double sc0 = pow2(54 - xu[a]), sc1 = pow2(54 - xd[a]);   // 64 products of 2^108 fit 64 bits
                iu[k] = fixed_parts(u, sc0);
                const int2 ix = fixed_parts(d.x, sc1), iy = fixed_parts(d.y, sc1);
                id[k] = make_int4(ix.x, ix.y, iy.x, iy.y);
            }
            __syncthreads();
        }
        // 4. pairs.  value = 2^(e_a + e_b) 2^-108 (A 2^56 + B 2^28) = 2^(e_a + e_b - 56) (16 A + B / 2^24)
        for (int pb = warp * 32; pb < nP; pb += kLinThreads) {   // whole warps: the reductions name every lane
            const int pr = pb + lane;
            int a = 0, b = 0;
            uint64_t mask = 0;
            if (pr < nP) {   // row a of the upper triangle: a S - a (a - 1) / 2 <= pr
                a = (int)(((float)(2 * S + 1) - sqrtf((float)((2 * S + 1) * (2 * S + 1) - 8 * pr))) * 0.5f);
                a = max(0, min(a, S - 1));
                while (a > 0 && a * S - a * (a - 1) / 2 > pr) --a;
                while ((a + 1) * S - (a + 1) * a / 2 <= pr) ++a;
                b = a + pr - (a * S - a * (a - 1) / 2);
                mask = fmask[a] & fmask[b];
            }
            const uint64_t any = (uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)mask) |
                                 ((uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)(mask >> 32)) << 32);
            if (!any) continue;
            int pos = -1;
            if (mask) {
                pos = find_col(A.col, A.rowptr[fidx[a]], A.rowptr[fidx[a] + 1], fidx[b]);
                if (pos < 0) atomicOr(A.flag, 8);
            }
            if (!vol) {
                double f[2] = {0.0, 0.0};
                for (uint64_t bits = mask; bits; bits &= bits - 1) {
                    const int p = __ffsll((long long)bits) - 1;
                    const double w = tabu[p * S + a] * tabu[p * S + b];
                    if (qfs[p] == 0) f[0] += w;
                    else f[1] += w;
                }
                if (pos < 0) continue;
                if (f[0] != 0.0) atomicAdd(&A.mats[(13 + face_slot[0]) * nnz + pos], f[0]);
                if (f[1] != 0.0) atomicAdd(&A.mats[(13 + face_slot[1]) * nnz + pos], f[1]);
                continue;
            }
            long long hh[9], hl[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) hh[k] = hl[k] = 0;
            for (uint64_t bits = any; bits; bits &= bits - 1) {
                const int p = __ffsll((long long)bits) - 1;
                const int2 ua = iu[p * S + a], ub = iu[p * S + b];
                const int4 da = id[p * S + a], db = id[p * S + b];
                const int ah[3] = {ua.x, da.x, da.z}, al[3] = {ua.y, da.y, da.w};
                const int bh[3] = {ub.x, db.x, db.z}, bl[3] = {ub.y, db.y, db.w};
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        hh[3 * q + r] = mad_wide(ah[q], bh[r], hh[3 * q + r]);
                        hl[3 * q + r] = mad_wide(ah[q], bl[r], hl[3 * q + r]);
                        hl[3 * q + r] = mad_wide(al[q], bh[r], hl[3 * q + r]);
                    }
            }
            if (pos < 0) continue;
            double v[9];
            const double f00 = pow2(xu[a] + xu[b] - 56), f01 = pow2(xu[a] + xd[b] - 56), f10 = pow2(xd[a] + xu[b] - 56),
                         f11 = pow2(xd[a] + xd[b] - 56);
#pragma unroll
            for (int k = 0; k < 9; ++k)
                v[k] = (double)(hh[k] * 16 + ((hl[k] + (1 << 23)) >> 24)) *
                       (k == 0 ? f00 : (k < 3 ? f01 : (k % 3 == 0 ? f10 : f11)));
            atomicAdd(&A.mats[pos], v[0]);
            atomicAdd(&A.mats[nnz + pos], st * v[0]);
            atomicAdd(&A.mats[2 * nnz + pos], ss * v[0]);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const double gab = v[3 * (1 + c)], gba = v[1 + c];   // d_c u_a u_b, u_a d_c u_b
                atomicAdd(&A.mats[(3 + c) * nnz + pos], gab);
                atomicAdd(&A.mats[(5 + c) * nnz + pos], st * gab);
                atomicAdd(&A.mats[(7 + c) * nnz + pos], ss * gab);
                atomicAdd(&gt[c * nnz + pos], gba);
                atomicAdd(&gt[(2 + c) * nnz + pos], st * gba);
                atomicAdd(&gt[(4 + c) * nnz + pos], ss * gba);
#pragma unroll
                for (int d = 0; d < 2; ++d) atomicAdd(&A.mats[(9 + 2 * c + d) * nnz + pos], v[3 * (1 + c) + 1 + d]);
            }
        }
        __syncthreads();
        base += P;
    }
    if (tid < S) {
        const int32_t a = fidx[tid];
        const double qi = A.q[i];
        if (vq0 != 0.0) atomicAdd(&A.vecs[a], qi * vq0);
        if (vqx != 0.0) atomicAdd(&A.vecs[n + a], qi * vqx);
        if (vqy != 0.0) atomicAdd(&A.vecs[2 * n + a], qi * vqy);
        if (face_slot[0] >= 0 && vb0 != 0.0) atomicAdd(&A.vecs[(3 + face_slot[0]) * n + a], vb0);
        if (face_slot[1] >= 0 && vb1 != 0.0) atomicAdd(&A.vecs[(3 + face_slot[1]) * n + a], vb1);
    }
}

// Lower entries from the upper ones of k_assemble_2d_lin, and the trial volumes: entry (i, j), i < j, holds the
// sums without V_j; gt holds G(j, i).  Eight lanes per row.
__global__ void k_mirror_2d(int64_t n, int64_t nnz, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                            const double *__restrict__ V, const double *__restrict__ gt, double *__restrict__ mats,
                            int *__restrict__ flag) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    if (i >= n) return;
    const double vi = V[i];
    for (int32_t p = rowptr[i] + (threadIdx.x & 7); p < rowptr[i + 1]; p += 8) {
        const int32_t j = col[p];
        if (j < i) continue;
        const double vj = V[j];
        int q = p;
        if (j != i) {
            q = find_col(col, rowptr[j], rowptr[j + 1], (int32_t)i);
            if (q < 0) { atomicOr(flag, 8); continue; }
        }
        auto both = [&](int f, double up, double low) {
            mats[f * nnz + p] = up * vj;
            if (q != p) mats[f * nnz + q] = low * vi;
        };
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const double v = mats[f * nnz + p];
            both(f, v, v);
        }
#pragma unroll
        for (int f = 0; f < 6; ++f) both(3 + f, mats[(3 + f) * nnz + p], gt[f * nnz + p]);
        double k[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) k[f] = mats[(9 + f) * nnz + p];
#pragma unroll
        for (int f = 0; f < 4; ++f) both(9 + f, k[f], k[2 * (f % 2) + f / 2]);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const double v = mats[(13 + f) * nnz + p];
            if (v != 0.0) both(13 + f, v, v);
        }
    }
}

// RK point interpolation at the centres: interp[pos(i, j)] = V_j U_j(x_i).
template <int ORD>
__global__ void k_interp_2d(int64_t n, const double *__restrict__ x, const double *__restrict__ R,
                            const double *__restrict__ V, const int32_t *__restrict__ rowptr,
                            const int32_t *__restrict__ col, double *__restrict__ interp,
                            int *__restrict__ flag) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t s0 = rowptr[i], len = rowptr[i + 1] - s0;
    double fx[kMaxS * 2], fy[kMaxS * 2], fR[kMaxS * 2], fV[kMaxS * 2];
    int32_t fp[kMaxS * 2];
    const double px = x[2 * i], py = x[2 * i + 1];
    int S = 0;
    for (int32_t p = 0; p < len; ++p) {
        int32_t j = col[s0 + p];
        double dx = px - x[2 * j], dy = py - x[2 * j + 1];
        if (sqrt(dx * dx + dy * dy) < R[j]) {
            if (S < 2 * kMaxS) {
                fx[S] = x[2 * j]; fy[S] = x[2 * j + 1]; fR[S] = R[j]; fV[S] = V[j]; fp[S] = s0 + p;
            }
            ++S;
        }
    }
    if (S > 2 * kMaxS) { atomicOr(flag, 2); return; }
    double U[kMaxS * 2], Ux[kMaxS * 2], Uy[kMaxS * 2];
    bool ok;
    if constexpr (ORD == 1) {
        ok = rk_point(px, py, 0.5 * R[i], S, fx, fy, fR, fV, U, Ux, Uy, 1);
    } else {
        double fR2[kMaxS * 2], finvh[kMaxS * 2];
        for (int a = 0; a < S; ++a) {
            fR2[a] = fR[a] * fR[a];
            finvh[a] = 2.0 / fR[a];
        }
        ok = S <= 64 && rk_point_gen<ORD>(px, py, 0.5 * R[i], S, fx, fy, fR2, finvh, fV, U, Ux, Uy, 1) != 0;
    }
    if (!ok) {
        atomicOr(flag, 1);
        return;
    }
    for (int a = 0; a < S; ++a) interp[fp[a]] = fV[a] * U[a];
}

}  // namespace

static mlpg_status upload_rules(mlpg_ctx *ctx, int ntri1d, int nline) {
    double xi[2 * kMaxTri], w[kMaxTri], t[kMaxLine], lw[kMaxLine];
    triangle_rule(ntri1d, xi, w);
    line_rule(nline, t, lw);
    CU(ctx, cudaMemcpyToSymbolAsync(c_tri_xi, xi, sizeof(double) * 2 * ntri1d * ntri1d, 0,
                                    cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, cudaMemcpyToSymbolAsync(c_tri_w, w, sizeof(double) * ntri1d * ntri1d, 0,
                                    cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, cudaMemcpyToSymbolAsync(c_line_t, t, sizeof(double) * nline, 0, cudaMemcpyHostToDevice,
                                    ctx->stream));
    CU(ctx, cudaMemcpyToSymbolAsync(c_line_w, lw, sizeof(double) * nline, 0, cudaMemcpyHostToDevice,
                                    ctx->stream));
    return MLPG_OK;
}

static mlpg_status check_flag(mlpg_ctx *ctx, const char *stage) {
    int flag = 0;
    CU(ctx, cudaMemcpyAsync(&flag, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    CU(ctx, cudaStreamSynchronize(ctx->stream));
    if (flag & 1) return set_err(ctx, MLPG_ERR_RK_SINGULAR, std::string(stage) + ": RK moment matrix singular");
    if (flag & 2) return set_err(ctx, MLPG_ERR_ARG, std::string(stage) + ": too many functions reach one cell");
    if (flag & 4) return set_err(ctx, MLPG_ERR_GEOMETRY, std::string(stage) + ": a cell touches more than two faces");
    if (flag & 8) return set_err(ctx, MLPG_ERR_GEOMETRY, std::string(stage) + ": support pair outside the overlap pattern");
    return MLPG_OK;
}

mlpg_status run_interp(mlpg_ctx *ctx) {
    MLPG_TRY(dalloc(ctx, &ctx->interp, ctx->nnz));
    if (!ctx->d_flag) MLPG_TRY(dalloc(ctx, &ctx->d_flag, 1));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->interp, 0, ctx->nnz * sizeof(double), ctx->stream));
    int B = 128;
    const int ord = ctx->opt.rk_order;
    auto launch = [&](auto kern) {
        kern<<<(ctx->n + B - 1) / B, B, 0, ctx->stream>>>(ctx->n, ctx->x, ctx->R, ctx->V, ctx->rowptr, ctx->col,
                                                          ctx->interp, ctx->d_flag);
    };
    if (ord == 0) launch(k_interp_2d<0>);
    else if (ord == 2) launch(k_interp_2d<2>);
    else launch(k_interp_2d<1>);
    CU_LAUNCH(ctx);
    return check_flag(ctx, "interpolation");
}

mlpg_status run_assemble(mlpg_ctx *ctx) {
    const int tri1d = 5, nline = 5;
    MLPG_TRY(upload_rules(ctx, tri1d, nline));
    ctx->nmats = mlpg_n_matrices(2);
    ctx->nvecs = mlpg_n_vectors(2);
    if (!ctx->mats) MLPG_TRY(dalloc(ctx, &ctx->mats, (size_t)ctx->nmats * ctx->nnz));
    if (!ctx->vecs) MLPG_TRY(dalloc(ctx, &ctx->vecs, (size_t)ctx->nvecs * ctx->n));
    CU(ctx, cudaMemsetAsync(ctx->mats, 0, sizeof(double) * ctx->nmats * ctx->nnz, ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->vecs, 0, sizeof(double) * ctx->nvecs * ctx->n, ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
    AsmArgs a;
    a.n = ctx->n; a.nnz = ctx->nnz;
    a.x = ctx->x; a.R = ctx->R; a.V = ctx->V; a.sig_t = ctx->sig_t; a.sig_s = ctx->sig_s; a.q = ctx->q;
    a.rowptr = ctx->rowptr; a.col = ctx->col; a.cptr = ctx->cptr; a.labels = ctx->labels;
    a.verts = ctx->verts;
    a.ntri = tri1d * tri1d; a.nline = nline;
    a.mats = ctx->mats; a.vecs = ctx->vecs; a.flag = ctx->d_flag;
    // shared table + weights + faces + pair sums for <ORD, MAXS, CHUNK>
    auto run = [&](auto kern, int maxs, int chunk) -> mlpg_status {
        size_t smem = sizeof(double) * (3 * (size_t)chunk * maxs + chunk + chunk / 2 + 1 +
                                        11 * (size_t)maxs * (maxs + 1) / 2);
        CU(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<ctx->n, kThreads, smem, ctx->stream>>>(a);
        CU_LAUNCH(ctx);
        return MLPG_OK;
    };
    if (ctx->opt.rk_order == 0) {
        MLPG_TRY(run(k_assemble_2d<0, 48, 32>, 48, 32));
    } else if (ctx->opt.rk_order == 2) {
        MLPG_TRY(run(k_assemble_2d<2, 48, 32>, 48, 32));
    } else {
        double *gt = nullptr;   // G of the lower entries
        MLPG_TRY(assembly_scratch(ctx, &gt));
        CU(ctx, cudaMemsetAsync(gt, 0, sizeof(double) * 6 * ctx->nnz, ctx->stream));
        // u and (u_x, u_y) of kLinEntries entries, the first rounded to a 16-byte boundary
        const size_t smem = sizeof(double) * (3 * (size_t)kLinEntries + 2);
        CU(ctx, cudaFuncSetAttribute(k_assemble_2d_lin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_assemble_2d_lin<<<(unsigned)ctx->n, kLinThreads, smem, ctx->stream>>>(a, gt);
        CU_LAUNCH(ctx);
        k_mirror_2d<<<(unsigned)((ctx->n * 8 + 255) / 256), 256, 0, ctx->stream>>>(ctx->n, ctx->nnz, ctx->rowptr, ctx->col,
                                                                                   ctx->V, gt, ctx->mats, ctx->d_flag);
        CU_LAUNCH(ctx);
        return check_flag(ctx, "assembly");
    }
    return check_flag(ctx, "assembly");
}

}  // namespace mlpg
