// 3D integration (Sec. 3.2, Alg. 1) over the elements of the polyhedral cells:
// one CTA per tetrahedron (volume forms) or per boundary triangle (surface
// forms).  Each element's quadrature points are mapped from the reference rule
// (App. A); the functions supported at any of its points are taken from the
// overlap row of the cell's generator; the RK functions and gradients are
// evaluated warp-cooperatively per point (Sec. 2.2, basis P = [1, (x - x_j)/s]
// for the linear correction or P = [1] for order 0, s = h of the generator);
// every pair's forms are summed over the element's
// points in registers and added to the shared pattern with FP64 atomics.
//
// mats layout in 3D: 0 M0, 1 Mt, 2 Ms, 3-5 G, 6-8 Gt, 9-11 Gs, 12-20 K (a-major),
// 21-26 S_f; vecs: 0 Q0, 1-3 Q, 4-9 B_f.
#include <algorithm>
#include <cmath>

#include "fixed_sum.cuh"
#include "internal.h"

namespace mlpg {

namespace {
constexpr int kMaxS3 = 96;        // functions supported on one element
constexpr int kMaxQ3 = 27;        // points per element (tetrahedron rule up to 3x3x3)
constexpr int kThreads3 = 256;
constexpr int kMaxCand = 1024;    // overlap row length

__constant__ double c3_tet_xi[3 * kMaxQ3];
__constant__ double c3_tet_w[kMaxQ3];
__constant__ double c3_tri_xi[2 * kMaxQ3];
__constant__ double c3_tri_w[kMaxQ3];

__device__ __forceinline__ double w3(double chi) {   // cubic spline, support chi < 2
    if (chi < 1.0) return 1.0 - chi * chi * (1.5 - 0.75 * chi);
    if (chi < 2.0) { double t = 2.0 - chi; return 0.25 * t * t * t; }
    return 0.0;
}
__device__ __forceinline__ double dw3(double chi) {
    if (chi < 1.0) return chi * (2.25 * chi - 3.0);
    if (chi < 2.0) { double t = 2.0 - chi; return -0.75 * t * t; }
    return 0.0;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// index of the symmetric NP x NP entry (i, j) in a packed array of NP (NP + 1) / 2
template <int NP>
__device__ __forceinline__ int symn(int i, int j) {
    return i <= j ? i * NP - i * (i - 1) / 2 + (j - i) : j * NP - j * (j - 1) / 2 + (i - j);
}

// RK functions of the S staged functions at p (one warp; lane owns a = lane +
// 32 k), basis P_j = [1] (order 0, NP = 1) or [1, (p - x_j)/s] (order 1,
// NP = 4).  Writes U, dU (3 components) at tab[c * cs + a], c = 0..3, and the
// support mask bits into mk[2].  Returns false when the moment matrix is not
// positive definite.
template <int NP>
__device__ bool rk3_warp(const double p[3], double s, int S, const double *fx, const double *fR2,
                         const double *finvh, const double *fV, double *tab, int cs, uint64_t *mk) {
    static_assert(NP == 1 || NP == 4, "order 0 or 1");
    constexpr int NE = NP * (NP + 1) / 2;
    const int lane = threadIdx.x & 31;
    const double is = 1.0 / s;
    double M[NE], D[3][NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) { M[e] = 0.0; D[0][e] = D[1][e] = D[2][e] = 0.0; }
    double Wl[3], Gl[3][3];
    bool on[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a = lane + 32 * k;
        on[k] = false;
        Wl[k] = 0.0;
        Gl[k][0] = Gl[k][1] = Gl[k][2] = 0.0;
        if (a >= S) continue;
        const double d0 = p[0] - fx[3 * a], d1 = p[1] - fx[3 * a + 1], d2 = p[2] - fx[3 * a + 2];
        const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
        if (!(r2 < fR2[a])) continue;
        on[k] = true;
        const double ir = r2 > 0.0 ? rsqrt(r2) : 0.0;
        const double chi = r2 * ir * finvh[a];
        const double W = w3(chi), g = dw3(chi) * finvh[a] * ir;
        const double Wg[3] = {g * d0, g * d1, g * d2}, v = fV[a];
        Wl[k] = W;
        Gl[k][0] = Wg[0]; Gl[k][1] = Wg[1]; Gl[k][2] = Wg[2];
        const double Pall[4] = {1.0, d0 * is, d1 * is, d2 * is};
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int j = i; j < NP; ++j) {
                const int e = symn<NP>(i, j);
                const double pp = Pall[i] * Pall[j];
                M[e] += v * W * pp;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double dp = ((i == c + 1) * Pall[j] + (j == c + 1) * Pall[i]) * is;
                    D[c][e] += v * (dp * W + pp * Wg[c]);
                }
            }
    }
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        M[e] = warp_sum(M[e]);
        D[0][e] = warp_sum(D[0][e]);
        D[1][e] = warp_sum(D[1][e]);
        D[2][e] = warp_sum(D[2][e]);
    }
    // support mask of this point
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        unsigned b = __ballot_sync(0xffffffffu, on[k]);
        if (lane == 0) {
            if (k == 0) mk[0] = b;
            else if (k == 1) mk[0] |= uint64_t(b) << 32;
            else mk[1] = b;
        }
    }
    // Cholesky of M (every lane, same values)
    double L[NP][NP];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int j = 0; j < NP; ++j) L[i][j] = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        double dsum = M[symn<NP>(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) dsum -= L[j][k] * L[j][k];
        if (!(dsum > 1e-14 * M[symn<NP>(j, j)])) return false;
        L[j][j] = sqrt(dsum);
#pragma unroll
        for (int i = j + 1; i < NP; ++i) {
            double t = M[symn<NP>(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[i][k] * L[j][k];
            L[i][j] = t / L[j][j];
        }
    }
    auto solve = [&](const double b[NP], double o[NP]) {
        double y[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            double t = b[i];
#pragma unroll
            for (int k = 0; k < i; ++k) t -= L[i][k] * y[k];
            y[i] = t / L[i][i];
        }
#pragma unroll
        for (int i = NP - 1; i >= 0; --i) {
            double t = y[i];
#pragma unroll
            for (int k = i + 1; k < NP; ++k) t -= L[k][i] * o[k];
            o[i] = t / L[i][i];
        }
    };
    // C = M^-1 e1, and its derivatives Cd[c] = -M^-1 (dM/dx_c) C
    double C[NP], Cd[3][NP];
    double e1[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) e1[i] = i == 0 ? 1.0 : 0.0;
    solve(e1, C);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double b[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            double t = 0.0;
#pragma unroll
            for (int j = 0; j < NP; ++j) t += D[c][symn<NP>(i, j)] * C[j];
            b[i] = -t;
        }
        solve(b, Cd[c]);
    }
    // U_a = W_a P_a . C;  d_c U_a = W_a (dP_a/dx_c . C + P_a . Cd[c]) + (P_a . C) dW_a/dx_c
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a = lane + 32 * k;
        if (a >= S) continue;
        double u = 0.0, ud[3] = {0.0, 0.0, 0.0};
        if (on[k]) {
            const double Pall[4] = {1.0, (p[0] - fx[3 * a]) * is, (p[1] - fx[3 * a + 1]) * is,
                                    (p[2] - fx[3 * a + 2]) * is};
            double PC = 0.0;
#pragma unroll
            for (int i = 0; i < NP; ++i) PC += Pall[i] * C[i];
            const double W = Wl[k];
            u = W * PC;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double t = NP > 1 ? C[NP > 1 ? c + 1 : 0] * is : 0.0;
#pragma unroll
                for (int i = 0; i < NP; ++i) t += Pall[i] * Cd[c][i];
                ud[c] = W * t + PC * Gl[k][c];
            }
        }
        tab[a] = u;
        tab[cs + a] = ud[0];
        tab[2 * cs + a] = ud[1];
        tab[3 * cs + a] = ud[2];
    }
    return true;
}

__device__ int find_col3(const int32_t *__restrict__ col, int32_t lo, int32_t hi, int32_t key) {
    hi -= 1;
    while (lo <= hi) {
        int32_t mid = (lo + hi) >> 1;
        int32_t c = col[mid];
        if (c == key) return mid;
        if (c < key) lo = mid + 1; else hi = mid - 1;
    }
    return -1;
}

struct Asm3Args {
    int64_t n, nnz, nelem;
    const double *x, *R, *V, *sig_t, *sig_s, *q;
    const int32_t *rowptr, *col;
    const int32_t *owner, *face;   // face: boundary triangles only
    const double *ev;              // 9 per element: three vertices
    int nq;
    double *mats, *vecs;
    int *flag;
    const int32_t *list;           // elements to integrate (null: all, in order)
};

// BND = false: tetrahedra (generator, v0, v1, v2) -> M0, Mt, Ms, G, Gt, Gs, K, Q0, Q.
// BND = true: boundary triangles (v0, v1, v2) on face f -> S_f, B_f.
template <bool BND, int NP>
__global__ void __launch_bounds__(kThreads3) k_assemble_3d(Asm3Args A) {
    __shared__ double fx[3 * kMaxS3], fR2[kMaxS3], finvh[kMaxS3], fV[kMaxS3];
    __shared__ int32_t fidx[kMaxS3];
    __shared__ double qx[3 * kMaxQ3], qw[kMaxQ3];
    __shared__ uint64_t qmk[kMaxQ3][2];
    __shared__ int wcnt[kThreads3 / 32];
    __shared__ int S_sh, bad;
    extern __shared__ double tab[];   // [nq][4][kMaxS3]
    const int64_t e = A.list ? A.list[blockIdx.x] : blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t o = A.owner[e];
    const int nq = A.nq;
    if (tid == 0) { S_sh = 0; bad = 0; }
    // quadrature points of the element (App. A maps)
    if (tid < nq) {
        const double *v = A.ev + 9 * e;
        double p0[3], e1[3], e2[3], e3[3], wq;
        if (!BND) {
            const double *g = A.x + 3 * (int64_t)o;
            for (int c = 0; c < 3; ++c) {
                p0[c] = g[c];
                e1[c] = v[c] - g[c];
                e2[c] = v[3 + c] - g[c];
                e3[c] = v[6 + c] - g[c];
            }
            const double det = e1[0] * (e2[1] * e3[2] - e2[2] * e3[1]) - e1[1] * (e2[0] * e3[2] - e2[2] * e3[0]) +
                               e1[2] * (e2[0] * e3[1] - e2[1] * e3[0]);
            const double a = c3_tet_xi[3 * tid], b = c3_tet_xi[3 * tid + 1], c = c3_tet_xi[3 * tid + 2];
            for (int k = 0; k < 3; ++k) qx[3 * tid + k] = p0[k] + e1[k] * a + e2[k] * b + e3[k] * c;
            wq = c3_tet_w[tid] * fabs(det);
        } else {
            for (int c = 0; c < 3; ++c) {
                p0[c] = v[c];
                e1[c] = v[3 + c] - v[c];
                e2[c] = v[6 + c] - v[c];
            }
            const double cx = e1[1] * e2[2] - e1[2] * e2[1], cy = e1[2] * e2[0] - e1[0] * e2[2],
                         cz = e1[0] * e2[1] - e1[1] * e2[0];
            const double a = c3_tri_xi[2 * tid], b = c3_tri_xi[2 * tid + 1];
            for (int k = 0; k < 3; ++k) qx[3 * tid + k] = p0[k] + e1[k] * a + e2[k] * b;
            wq = c3_tri_w[tid] * sqrt(cx * cx + cy * cy + cz * cz);
        }
        qw[tid] = wq;
    }
    __syncthreads();
    // functions supported at some point of the element, in overlap-row order
    const int32_t r0 = A.rowptr[o], rl = A.rowptr[o + 1] - r0;
    if (rl > kMaxCand) {
        if (tid == 0) atomicOr(A.flag, 2);
        return;
    }
    for (int base = 0; base < rl; base += kThreads3) {
        const int c = base + tid;
        bool sup = false;
        int32_t j = -1;
        if (c < rl) {
            j = A.col[r0 + c];
            const double xj = A.x[3 * (int64_t)j], yj = A.x[3 * (int64_t)j + 1], zj = A.x[3 * (int64_t)j + 2];
            const double R2 = A.R[j] * A.R[j];
            for (int q = 0; q < nq && !sup; ++q) {
                const double dx = qx[3 * q] - xj, dy = qx[3 * q + 1] - yj, dz = qx[3 * q + 2] - zj;
                sup = dx * dx + dy * dy + dz * dz < R2;
            }
        }
        const unsigned b = __ballot_sync(0xffffffffu, sup);
        if (lane == 0) wcnt[warp] = __popc(b);
        __syncthreads();
        int off = S_sh;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        const int slot = off + __popc(b & ((1u << lane) - 1u));
        if (sup) {
            if (slot < kMaxS3) {
                fidx[slot] = j;
                fx[3 * slot] = A.x[3 * (int64_t)j];
                fx[3 * slot + 1] = A.x[3 * (int64_t)j + 1];
                fx[3 * slot + 2] = A.x[3 * (int64_t)j + 2];
                fR2[slot] = A.R[j] * A.R[j];
                finvh[slot] = 2.0 / A.R[j];
                fV[slot] = A.V[j];
            } else {
                bad = 1;
            }
        }
        __syncthreads();
        if (tid == 0) {
            int t = 0;
            for (int w = 0; w < kThreads3 / 32; ++w) t += wcnt[w];
            S_sh += t;
        }
        __syncthreads();
    }
    if (bad) {
        if (tid == 0) atomicOr(A.flag, 2);
        return;
    }
    const int S = S_sh;
    // RK at every point: one warp per point
    const double s = 0.5 * A.R[o];
    for (int q = warp; q < nq; q += kThreads3 / 32) {
        const double p[3] = {qx[3 * q], qx[3 * q + 1], qx[3 * q + 2]};
        if (!rk3_warp<NP>(p, s, S, fx, fR2, finvh, fV, tab + (int64_t)q * 4 * kMaxS3, kMaxS3, qmk[q])) {
            if (lane == 0) atomicOr(A.flag, 1);
        }
    }
    __syncthreads();
    const int64_t nnz = A.nnz, n = A.n;
    const double st = A.sig_t[o], ss = A.sig_s[o], qv = A.q[o];
    // pairs (a, b): forms summed over the element's points, then added to the pattern
    for (int pidx = tid; pidx < S * S; pidx += kThreads3) {
        const int a = pidx / S, b = pidx - a * S;
        const uint64_t ba = a < 64 ? (uint64_t(1) << a) : 0, bb = b < 64 ? (uint64_t(1) << b) : 0;
        const uint64_t ha = a >= 64 ? (uint64_t(1) << (a - 64)) : 0, hb = b >= 64 ? (uint64_t(1) << (b - 64)) : 0;
        if (BND) {
            double uu = 0.0;
            for (int q = 0; q < nq; ++q) {
                const bool sa = (qmk[q][0] & ba) || (qmk[q][1] & ha), sb = (qmk[q][0] & bb) || (qmk[q][1] & hb);
                if (!(sa && sb)) continue;
                const double *t = tab + (int64_t)q * 4 * kMaxS3;
                uu += qw[q] * t[a] * t[b];
            }
            if (uu == 0.0) continue;
            const int pos = find_col3(A.col, A.rowptr[fidx[a]], A.rowptr[fidx[a] + 1], fidx[b]);
            if (pos < 0) { atomicOr(A.flag, 8); continue; }
            atomicAdd(&A.mats[(21 + A.face[e]) * nnz + pos], uu * fV[b]);
        } else {
            double uu = 0.0, g[3] = {0, 0, 0}, k[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
            for (int q = 0; q < nq; ++q) {
                const bool sa = (qmk[q][0] & ba) || (qmk[q][1] & ha), sb = (qmk[q][0] & bb) || (qmk[q][1] & hb);
                if (!(sa && sb)) continue;
                const double *t = tab + (int64_t)q * 4 * kMaxS3;
                const double w = qw[q], ub = t[b];
                const double da[3] = {w * t[kMaxS3 + a], w * t[2 * kMaxS3 + a], w * t[3 * kMaxS3 + a]};
                const double db[3] = {t[kMaxS3 + b], t[2 * kMaxS3 + b], t[3 * kMaxS3 + b]};
                uu += w * t[a] * ub;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    g[c] += da[c] * ub;
#pragma unroll
                    for (int d = 0; d < 3; ++d) k[3 * c + d] += da[c] * db[d];
                }
            }
            if (uu == 0.0 && g[0] == 0.0 && g[1] == 0.0 && g[2] == 0.0) continue;
            const int pos = find_col3(A.col, A.rowptr[fidx[a]], A.rowptr[fidx[a] + 1], fidx[b]);
            if (pos < 0) { atomicOr(A.flag, 8); continue; }
            const double vb = fV[b], m0 = uu * vb;
            atomicAdd(&A.mats[pos], m0);
            atomicAdd(&A.mats[nnz + pos], st * m0);
            atomicAdd(&A.mats[2 * nnz + pos], ss * m0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double gc = g[c] * vb;
                atomicAdd(&A.mats[(3 + c) * nnz + pos], gc);
                atomicAdd(&A.mats[(6 + c) * nnz + pos], st * gc);
                atomicAdd(&A.mats[(9 + c) * nnz + pos], ss * gc);
            }
#pragma unroll
            for (int c = 0; c < 9; ++c) atomicAdd(&A.mats[(12 + c) * nnz + pos], k[c] * vb);
        }
    }
    // vectors: Q0, Q (volume), B_f (boundary)
    if (tid < S) {
        const int a = tid;
        const uint64_t ba = a < 64 ? (uint64_t(1) << a) : 0, ha = a >= 64 ? (uint64_t(1) << (a - 64)) : 0;
        double v0 = 0.0, vg[3] = {0, 0, 0};
        for (int q = 0; q < nq; ++q) {
            if (!((qmk[q][0] & ba) || (qmk[q][1] & ha))) continue;
            const double *t = tab + (int64_t)q * 4 * kMaxS3;
            v0 += qw[q] * t[a];
            if (!BND)
                for (int c = 0; c < 3; ++c) vg[c] += qw[q] * t[(c + 1) * kMaxS3 + a];
        }
        const int32_t i = fidx[a];
        if (BND) {
            if (v0 != 0.0) atomicAdd(&A.vecs[(4 + A.face[e]) * n + i], v0);
        } else {
            if (v0 != 0.0) atomicAdd(&A.vecs[i], qv * v0);
            for (int c = 0; c < 3; ++c)
                if (vg[c] != 0.0) atomicAdd(&A.vecs[(1 + c) * n + i], qv * vg[c]);
        }
    }
}

// ---------------------------------------------------------------------------
// Volume forms by groups of tetrahedra (the default).
//
// A group is the fan of one cell face, at most kGrpTets tetrahedra: its points
// share most of their functions (about 50 over a fan of 5, against 40 over one
// tetrahedron), so the pattern is looked up and added to once per fan instead of
// once per tetrahedron.  One CTA per group:
//   1. functions supported at some point and their 48-bit point masks (distances
//      in FP32 from the group's centre, FP64 where that could decide wrongly);
//   2. RK functions at every point, four lanes per point over that point's own
//      list of functions; the derivative moments are the third-order moments of
//      the kernel's radial derivative (19 sums instead of 30), M's Cholesky factor
//      once per point;
//   3. the table sqrt(w) (U, dU) is turned into fixed point, 55 bits below each
//      function's largest U and dU in the group, as two signed 28-bit parts;
//   4. every unordered pair a <= b sums the 16 products (u, u_x, u_y, u_z)_a x (u,
//      u_x, u_y, u_z)_b over the group's points in 64-bit integers, exactly but for
//      the products of two low parts (2^-56 of the two functions' largest each);
//   5. the sums are added to the pattern's upper entries (FP64 atomics), the forms
//      G(b, a) to three buffers of their own; k_mirror_3d fills the lower entries
//      (M0 and K are each other's transposes) and applies the trial volumes V_b.
//
// Why integers.  The FP64 units do 1.6 operations per clock and SM (measured), the
// integer multiplier 30 wide products; three of those replace one FP64 FMA.  Per
// tetrahedron the old kernel spent about 350k clocks (pairs twice, 17 operations each;
// 40 warp sums of FP64 values and a Cholesky factor in all 32 lanes per point; 33k
// atomics); now the RK functions bound it.
// Accuracy: fixed point 2^-55 below the function's largest value in the group in place of
// FP64's relative 2^-53 per product and per sum.
// Measured: the kernel at 15^3 (267,000 tetrahedra) 296 -> 51 ms.
// A group with more functions than the table holds goes to k_assemble_3d, element by
// element.
// ---------------------------------------------------------------------------
constexpr int kGrpTets = 6, kGrpPts = 8 * kGrpTets;   // 8 points per tetrahedron
constexpr int kGrpThreads = 256;
constexpr int kGrpEntries = 3200;   // table entries (points x functions) of 32 bytes: two CTAs per SM

// groups of the tetrahedra, in any order: {first, count}.  The thread of a cell's first tetrahedron walks
// the cell; a fan (equal face centre, the first stored vertex) is cut into even parts of at most kGrpTets.
__global__ void k_tet_groups(int64_t ntet, const int32_t *__restrict__ owner, const double *__restrict__ ev,
                             int2 *__restrict__ grp, int *__restrict__ count) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ntet) return;
    const int32_t o = owner[i];
    if (i > 0 && owner[i - 1] == o) return;
    for (int64_t j = i; j < ntet && owner[j] == o;) {
        int64_t k = j + 1;
        while (k < ntet && owner[k] == o && ev[9 * k] == ev[9 * j] && ev[9 * k + 1] == ev[9 * j + 1] &&
               ev[9 * k + 2] == ev[9 * j + 2])
            ++k;
        const int len = (int)(k - j), parts = (len + kGrpTets - 1) / kGrpTets;
        int at = atomicAdd(count, parts);
        for (int q = 0; q < parts; ++q) {
            const int f = (int)((int64_t)len * q / parts), e = (int)((int64_t)len * (q + 1) / parts);
            grp[at + q] = make_int2((int)(j + f), e - f);
        }
        j = k;
    }
}

__device__ __forceinline__ double quad_sum(double v) {   // over the four lanes of a point
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    return v;
}
template <int NP>
__global__ void __launch_bounds__(kGrpThreads, 2) k_assemble_3d_grp(Asm3Args A, const int2 *__restrict__ grp,
                                                                    double *__restrict__ gt,   // [9][nnz]: G, Gt, Gs of (b, a)
                                                                    int *__restrict__ nskip, int32_t *__restrict__ skip) {
    __shared__ double fx[3 * kMaxS3], finvh[kMaxS3], fV[kMaxS3], qx[3 * kGrpPts], qsw[kGrpPts];
    __shared__ float qf[3 * kGrpPts], red_f[4];
    __shared__ int32_t fidx[kMaxS3];
    __shared__ uint64_t fmask[kMaxS3];                 // points at which a function is supported
    __shared__ uint8_t plist[kGrpPts][kMaxS3];         // functions of each point
    __shared__ int pcnt[kGrpPts], wcnt[kGrpThreads / 32];
    __shared__ int16_t xu[kMaxS3], xd[kMaxS3];         // exponents of each function's largest values
    __shared__ int S_sh, over;
    extern __shared__ __align__(16) unsigned char smem_tab[];
    double2 *tab = reinterpret_cast<double2 *>(smem_tab);   // [point][2][S]: (u, u_x), (u_y, u_z)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int2 gr = grp[blockIdx.x];
    const int64_t e0 = gr.x;
    const int nt = gr.y, P = 8 * nt;
    const int32_t o = A.owner[e0];
    const double *g = A.x + 3 * (int64_t)o;
    if (tid == 0) { S_sh = 0; over = 0; }
    if (tid < P) {
        const double *v = A.ev + 9 * (e0 + (tid >> 3));
        const int q = tid & 7;
        double e1[3], e2[3], e3[3];
        for (int c = 0; c < 3; ++c) {
            e1[c] = v[c] - g[c];
            e2[c] = v[3 + c] - g[c];
            e3[c] = v[6 + c] - g[c];
        }
        const double det = e1[0] * (e2[1] * e3[2] - e2[2] * e3[1]) - e1[1] * (e2[0] * e3[2] - e2[2] * e3[0]) +
                           e1[2] * (e2[0] * e3[1] - e2[1] * e3[0]);
        const double a = c3_tet_xi[3 * q], b = c3_tet_xi[3 * q + 1], c = c3_tet_xi[3 * q + 2];
        for (int k = 0; k < 3; ++k) {
            const double d = e1[k] * a + e2[k] * b + e3[k] * c;
            qx[3 * tid + k] = g[k] + d;
            qf[3 * tid + k] = (float)d;   // relative to the generator
        }
        qsw[tid] = sqrt(c3_tet_w[q] * fabs(det));
    }
    __syncthreads();
    if (warp == 0) {   // FP32 bounding sphere around the points' mean, relative to the generator
        float m[3] = {0.0f, 0.0f, 0.0f};
        for (int p = lane; p < P; p += 32)
            for (int k = 0; k < 3; ++k) m[k] += qf[3 * p + k];
        for (int k = 0; k < 3; ++k) {
            for (int x = 16; x > 0; x >>= 1) m[k] += __shfl_xor_sync(0xffffffffu, m[k], x);
            m[k] /= (float)P;
        }
        float r2 = 0.0f;
        for (int p = lane; p < P; p += 32) {
            const float dx = qf[3 * p] - m[0], dy = qf[3 * p + 1] - m[1], dz = qf[3 * p + 2] - m[2];
            r2 = fmaxf(r2, dx * dx + dy * dy + dz * dz);
        }
        for (int x = 16; x > 0; x >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, x));
        if (lane == 0) {
            for (int k = 0; k < 3; ++k) red_f[k] = m[k];
            red_f[3] = sqrtf(r2);
        }
    }
    __syncthreads();
    // 1. functions supported at some point, in overlap-row order (ascending)
    const int32_t r0 = A.rowptr[o], rl = A.rowptr[o + 1] - r0;
    for (int base = 0; base < rl; base += kGrpThreads) {
        const int c = base + tid;
        uint64_t mask = 0;
        int32_t j = -1;
        if (c < rl) {
            j = A.col[r0 + c];
            const double *xj = A.x + 3 * (int64_t)j;
            const double Rj = A.R[j], R2 = Rj * Rj;
            const float fxr = (float)(xj[0] - g[0]), fyr = (float)(xj[1] - g[1]), fzr = (float)(xj[2] - g[2]);
            const float Rf = (float)Rj, R2f = Rf * Rf;
            const float cx = fxr - red_f[0], cy = fyr - red_f[1], cz = fzr - red_f[2], reach = (Rf + red_f[3]) * 1.0001f;
            if (!(cx * cx + cy * cy + cz * cz > reach * reach)) {   // (squares beyond FP32's range: all functions)
                // the coordinates are rounded to 2^-24 of the largest, at most a few R: 1e-4 is far outside
                const float len2 = fxr * fxr + fyr * fyr + fzr * fzr + R2f, slack = 1e-4f * len2;
                for (int q = 0; q < P; ++q) {
                    const float dx = qf[3 * q] - fxr, dy = qf[3 * q + 1] - fyr, dz = qf[3 * q + 2] - fzr;
                    const float r2 = dx * dx + dy * dy + dz * dz;
                    bool sup = r2 < R2f;
                    if (!(fabsf(r2 - R2f) > slack)) {   // close, or beyond FP32's range
                        const double ex = qx[3 * q] - xj[0], ey = qx[3 * q + 1] - xj[1], ez = qx[3 * q + 2] - xj[2];
                        sup = ex * ex + ey * ey + ez * ez < R2;
                    }
                    mask |= (uint64_t)sup << q;
                }
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, mask != 0);
        if (lane == 0) wcnt[warp] = __popc(bal);
        __syncthreads();
        int off = S_sh;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        const int slot = off + __popc(bal & ((1u << lane) - 1u));
        if (mask) {
            if (slot < kMaxS3) {
                fidx[slot] = j;
                for (int k = 0; k < 3; ++k) fx[3 * slot + k] = A.x[3 * (int64_t)j + k];
                finvh[slot] = 2.0 / A.R[j];
                fV[slot] = A.V[j];
                fmask[slot] = mask;
            } else {
                over = 1;
            }
        }
        __syncthreads();
        if (tid == 0)
            for (int w = 0; w < kGrpThreads / 32; ++w) S_sh += wcnt[w];
        __syncthreads();
    }
    const int S = S_sh;
    if (over || S * P > kGrpEntries || rl > kMaxCand) {   // (block-uniform) the element kernel takes these
        if (tid == 0) {
            const int at = atomicAdd(nskip, nt);
            for (int k = 0; k < nt; ++k) skip[at + k] = (int32_t)(e0 + k);
        }
        return;
    }
    // each point's functions; the table starts at zero
    if (tid < P) {
        int n = 0;
        for (int a = 0; a < S; ++a)
            if ((fmask[a] >> tid) & 1) plist[tid][n++] = (uint8_t)a;
        pcnt[tid] = n;
    }
    for (int k = tid; k < P * 2 * S; k += kGrpThreads) tab[k] = make_double2(0.0, 0.0);
    __syncthreads();
    // 2. RK functions: four lanes per point
    const double s = 0.5 * A.R[o], is = 1.0 / s;
    for (int p0 = warp * 8; p0 < P; p0 += kGrpThreads / 4) {   // 8 points per warp (P is a multiple of 8)
        const int p = p0 + (lane >> 2), l4 = lane & 3, cnt = pcnt[p];
        const double px = qx[3 * p], py = qx[3 * p + 1], pz = qx[3 * p + 2];
        double2 *tp = tab + (int64_t)p * 2 * S;
        // moments: m of v W, t of v g s (g: radial derivative over the distance), by monomial
        double m[10], t[19];
#pragma unroll
        for (int k = 0; k < 10; ++k) m[k] = 0.0;
#pragma unroll
        for (int k = 0; k < 19; ++k) t[k] = 0.0;
        for (int k = l4; k < cnt; k += 4) {
            const int a = plist[p][k];
            const double dx = px - fx[3 * a], dy = py - fx[3 * a + 1], dz = pz - fx[3 * a + 2];
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double ir = r2 > 0.0 ? rsqrt(r2) : 0.0;
            const double ih = finvh[a], chi = r2 * ir * ih;
            const double W = w3(chi), gg = dw3(chi) * ih * ir, v = fV[a];
            tp[a] = make_double2(W, gg);
            const double aw = v * W, bw = v * gg * s;
            m[0] += aw;
            const double X = dx * is, Y = dy * is, Z = dz * is;
            const double bx = bw * X, by = bw * Y, bz = bw * Z;
            t[0] += bx; t[1] += by; t[2] += bz;
            if constexpr (NP == 4) {
                const double ax = aw * X, ay = aw * Y, az = aw * Z;
                m[1] += ax; m[2] += ay; m[3] += az;
                m[4] += ax * X; m[5] += ax * Y; m[6] += ax * Z; m[7] += ay * Y; m[8] += ay * Z; m[9] += az * Z;
                const double bxx = bx * X, bxy = bx * Y, bxz = bx * Z, byy = by * Y, byz = by * Z, bzz = bz * Z;
                t[3] += bxx; t[4] += bxy; t[5] += bxz; t[6] += byy; t[7] += byz; t[8] += bzz;
                t[9] += bxx * X; t[10] += bxx * Y; t[11] += bxx * Z; t[12] += bxy * Y; t[13] += bxy * Z; t[14] += bxz * Z;
                t[15] += byy * Y; t[16] += byy * Z; t[17] += byz * Z; t[18] += bzz * Z;
            }
        }
#pragma unroll
        for (int k = 0; k < (NP == 4 ? 10 : 1); ++k) m[k] = quad_sum(m[k]);
#pragma unroll
        for (int k = 0; k < (NP == 4 ? 19 : 3); ++k) t[k] = quad_sum(t[k]);
        double C[4] = {0.0, 0.0, 0.0, 0.0}, Cd[3][4];
        bool ok = true;
        if constexpr (NP == 4) {
            // M = L L^T with reciprocal pivots (m: 1, x, y, z, xx, xy, xz, yy, yz, zz)
            ok = m[0] > 0.0;
            const double i0 = rsqrt(m[0]);
            const double L10 = m[1] * i0, L20 = m[2] * i0, L30 = m[3] * i0;
            const double d1 = m[4] - L10 * L10;
            ok = ok && d1 > 1e-14 * m[4];
            const double i1 = rsqrt(d1), L21 = (m[5] - L20 * L10) * i1, L31 = (m[6] - L30 * L10) * i1;
            const double d2 = m[7] - L20 * L20 - L21 * L21;
            ok = ok && d2 > 1e-14 * m[7];
            const double i2 = rsqrt(d2), L32 = (m[8] - L30 * L20 - L31 * L21) * i2;
            const double d3 = m[9] - L30 * L30 - L31 * L31 - L32 * L32;
            ok = ok && d3 > 1e-14 * m[9];
            const double i3 = rsqrt(d3);
            auto solve = [&](double b0, double b1, double b2, double b3, double *r) {
                const double y0 = b0 * i0, y1 = (b1 - L10 * y0) * i1, y2 = (b2 - L20 * y0 - L21 * y1) * i2;
                const double y3 = (b3 - L30 * y0 - L31 * y1 - L32 * y2) * i3;
                r[3] = y3 * i3;
                r[2] = (y2 - L32 * r[3]) * i2;
                r[1] = (y1 - L21 * r[2] - L31 * r[3]) * i1;
                r[0] = (y0 - L10 * r[1] - L20 * r[2] - L30 * r[3]) * i0;
            };
            solve(1.0, 0.0, 0.0, 0.0, C);
            // Cd_c = -M^-1 D_c C, D_c C [i] = ((i == c + 1) + m_i C_(c+1)) / s + sum_j T_c[i][j] C_j
            // (M C = e_1 takes the first term's sum); T_c[i][j] the third-order moments
            constexpr int T2[3][4] = {{0, 3, 4, 5}, {1, 4, 6, 7}, {2, 5, 7, 8}};   // [c][i]: x_c x_i moment of t
            constexpr int T3[3][3][3] = {{{9, 10, 11}, {10, 12, 13}, {11, 13, 14}},
                                         {{10, 12, 13}, {12, 15, 16}, {13, 16, 17}},
                                         {{11, 13, 14}, {13, 16, 17}, {14, 17, 18}}};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double b[4];
                b[0] = t[c] * C[0];
#pragma unroll
                for (int j = 0; j < 3; ++j) b[0] += t[T2[c][1 + j]] * C[1 + j];
                b[0] += m[0] * C[1 + c] * is;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    b[1 + i] = t[T2[c][1 + i]] * C[0];
#pragma unroll
                    for (int j = 0; j < 3; ++j) b[1 + i] += t[T3[c][i][j]] * C[1 + j];
                    b[1 + i] += ((i == c ? 1.0 : 0.0) + m[1 + i] * C[1 + c]) * is;
                }
                solve(-b[0], -b[1], -b[2], -b[3], Cd[c]);
            }
        } else {
            ok = m[0] > 0.0;
            C[0] = 1.0 / m[0];
#pragma unroll
            for (int c = 0; c < 3; ++c) Cd[c][0] = -t[c] * C[0] * C[0];
        }
        if (!ok) {
            if (l4 == 0) atomicOr(A.flag, 1);
        }
        const double sw = qsw[p];
        for (int k = l4; k < cnt; k += 4) {
            const int a = plist[p][k];
            const double dx = px - fx[3 * a], dy = py - fx[3 * a + 1], dz = pz - fx[3 * a + 2];
            const double2 wg = tp[a];
            const double W = wg.x * sw, gg = wg.y * sw;
            const double X = dx * is, Y = dy * is, Z = dz * is;
            double PC = C[0], ud[3];
            if constexpr (NP == 4) PC += X * C[1] + Y * C[2] + Z * C[3];
            const double h = PC * gg, d[3] = {dx, dy, dz};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double q = Cd[c][0];
                if constexpr (NP == 4) q += C[1 + c] * is + X * Cd[c][1] + Y * Cd[c][2] + Z * Cd[c][3];
                ud[c] = W * q + h * d[c];
            }
            const double u = W * PC;
            if (ok) {
                tp[a] = make_double2(u, ud[0]);
                tp[S + a] = make_double2(ud[1], ud[2]);
            } else {
                tp[a] = make_double2(0.0, 0.0);
            }
        }
    }
    __syncthreads();
    const double st = A.sig_t[o], ss = A.sig_s[o];
    const int64_t nnz = A.nnz, n = A.n;
    // vectors Q0, Q and the scales (before the table changes to fixed point)
    if (tid < S) {
        unsigned mx0 = 0, mx1 = 0;   // high words of the largest |sqrt(w) u|, |sqrt(w) du|
        const double qv = A.q[o];
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
        for (uint64_t bits = fmask[tid]; bits; bits &= bits - 1) {
            const int p = __ffsll((long long)bits) - 1;
            const double2 u = tab[p * 2 * S + tid], w = tab[p * 2 * S + S + tid];
            const double sw = qsw[p];
            v0 += sw * u.x;
            v1 += sw * u.y;
            v2 += sw * w.x;
            v3 += sw * w.y;
            mx0 = max(mx0, abs_hiword(u.x));
            mx1 = max(mx1, max(abs_hiword(u.y), max(abs_hiword(w.x), abs_hiword(w.y))));
        }
        xu[tid] = (int16_t)top_exp(mx0);
        xd[tid] = (int16_t)top_exp(mx1);
        const int32_t i = fidx[tid];
        if (v0 != 0.0) atomicAdd(&A.vecs[i], qv * v0);
        if (v1 != 0.0) atomicAdd(&A.vecs[n + i], qv * v1);
        if (v2 != 0.0) atomicAdd(&A.vecs[2 * n + i], qv * v2);
        if (v3 != 0.0) atomicAdd(&A.vecs[3 * n + i], qv * v3);
    }
    __syncthreads();
    // 3. fixed point, in place: (hi, lo) of u, u_x | u_y, u_z
    int4 *itab = reinterpret_cast<int4 *>(smem_tab);
    for (int k = tid; k < P * S; k += kGrpThreads) {
        const int p = k / S, a = k - p * S;
        if (!((fmask[a] >> p) & 1)) continue;   // zero already
        const int at = p * 2 * S + a;
        const double2 u = tab[at], w = tab[at + S];
        const double sc0 = pow2(55 - xu[a]), sc1 = pow2(55 - xd[a]);   // 48 products of 2^110 fit 64 bits
        const int2 i0 = fixed_parts(u.x, sc0), i1 = fixed_parts(u.y, sc1), i2 = fixed_parts(w.x, sc1), i3 = fixed_parts(w.y, sc1);
        itab[at] = make_int4(i0.x, i0.y, i1.x, i1.y);
        itab[at + S] = make_int4(i2.x, i2.y, i3.x, i3.y);
    }
    __syncthreads();
    // 4. pairs.  value = 2^(e_a + e_b) 2^-110 (A 2^56 + B 2^28) = 2^(e_a + e_b - 57) (8 A + B / 2^25)
    const int nP = S * (S + 1) / 2;
    for (int base = warp * 32; base < nP; base += kGrpThreads) {   // whole warps: the reductions name every lane
        const int pr = base + lane;
        int a = 0, b = 0;
        uint64_t mask = 0;
        if (pr < nP) {
            // row a of the upper triangle: a S - a (a - 1) / 2 <= pr
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
        long long hh[16], hl[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) hh[k] = hl[k] = 0;
        for (uint64_t bits = any; bits; bits &= bits - 1) {
            const int p = __ffsll((long long)bits) - 1;
            const int4 *tp = itab + p * 2 * S;
            const int4 ua = tp[a], va = tp[S + a], ub = tp[b], vb = tp[S + b];
            const int ah[4] = {ua.x, ua.z, va.x, va.z}, al[4] = {ua.y, ua.w, va.y, va.w};
            const int bh[4] = {ub.x, ub.z, vb.x, vb.z}, bl[4] = {ub.y, ub.w, vb.y, vb.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    hh[4 * i + j] = mad_wide(ah[i], bh[j], hh[4 * i + j]);
                    hl[4 * i + j] = mad_wide(ah[i], bl[j], hl[4 * i + j]);
                    hl[4 * i + j] = mad_wide(al[i], bh[j], hl[4 * i + j]);
                }
        }
        if (!mask) continue;
        const int pos = find_col3(A.col, A.rowptr[fidx[a]], A.rowptr[fidx[a] + 1], fidx[b]);
        if (pos < 0) { atomicOr(A.flag, 8); continue; }
        double v[16];
        const double f00 = pow2(xu[a] + xu[b] - 57), f01 = pow2(xu[a] + xd[b] - 57), f10 = pow2(xd[a] + xu[b] - 57),
                     f11 = pow2(xd[a] + xd[b] - 57);
#pragma unroll
        for (int k = 0; k < 16; ++k)
            v[k] = (double)(hh[k] * 8 + ((hl[k] + (1 << 24)) >> 25)) *
                   (k == 0 ? f00 : (k < 4 ? f01 : ((k & 3) == 0 ? f10 : f11)));
        atomicAdd(&A.mats[pos], v[0]);
        atomicAdd(&A.mats[nnz + pos], st * v[0]);
        atomicAdd(&A.mats[2 * nnz + pos], ss * v[0]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double gab = v[4 * (1 + c)], gba = v[1 + c];   // d_c u_a u_b, u_a d_c u_b
            atomicAdd(&A.mats[(3 + c) * nnz + pos], gab);
            atomicAdd(&A.mats[(6 + c) * nnz + pos], st * gab);
            atomicAdd(&A.mats[(9 + c) * nnz + pos], ss * gab);
            atomicAdd(&gt[c * nnz + pos], gba);
            atomicAdd(&gt[(3 + c) * nnz + pos], st * gba);
            atomicAdd(&gt[(6 + c) * nnz + pos], ss * gba);
#pragma unroll
            for (int d = 0; d < 3; ++d) atomicAdd(&A.mats[(12 + 3 * c + d) * nnz + pos], v[4 * (1 + c) + 1 + d]);
        }
    }
}

// Lower entries from the upper ones of the group kernel, and the trial volumes: entry (i, j), i < j, holds
// the sums without V_j; gt holds G(j, i).  One thread per entry of the upper triangle.
__global__ void k_mirror_3d(int64_t n, int64_t nnz, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                            const double *__restrict__ V, const double *__restrict__ gt, double *__restrict__ mats,
                            int *__restrict__ flag) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;   // a warp per row
    if (i >= n) return;
    const double vi = V[i];
    for (int32_t p = rowptr[i] + (threadIdx.x & 31); p < rowptr[i + 1]; p += 32) {
        const int32_t j = col[p];
        if (j < i) continue;
        const double vj = V[j];
        int q = p;
        if (j != i) {
            q = find_col3(col, rowptr[j], rowptr[j + 1], (int32_t)i);
            if (q < 0) { atomicOr(flag, 8); continue; }
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const double v = mats[f * nnz + p];
            mats[f * nnz + p] = v * vj;
            if (q != p) mats[f * nnz + q] = v * vi;
        }
#pragma unroll
        for (int f = 0; f < 9; ++f) {
            const double v = mats[(3 + f) * nnz + p], w = gt[f * nnz + p];
            mats[(3 + f) * nnz + p] = v * vj;
            if (q != p) mats[(3 + f) * nnz + q] = w * vi;
        }
        double k[9];
#pragma unroll
        for (int f = 0; f < 9; ++f) k[f] = mats[(12 + f) * nnz + p];
#pragma unroll
        for (int f = 0; f < 9; ++f) {
            mats[(12 + f) * nnz + p] = k[f] * vj;
            if (q != p) mats[(12 + f) * nnz + q] = k[3 * (f % 3) + f / 3] * vi;
        }
    }
}

// interp[pos(i, j)] = V_j U_j(x_i): one warp per point, candidates from row i
template <int NP>
__global__ void __launch_bounds__(128) k_interp_3d(int64_t n, const double *__restrict__ x,
                                                   const double *__restrict__ R, const double *__restrict__ V,
                                                   const int32_t *__restrict__ rowptr,
                                                   const int32_t *__restrict__ col, double *__restrict__ interp,
                                                   int *__restrict__ flag) {
    constexpr int W = 4;   // warps per block
    __shared__ double fx[W][3 * kMaxS3], fR2[W][kMaxS3], finvh[W][kMaxS3], fV[W][kMaxS3];
    __shared__ int32_t fp[W][kMaxS3];
    __shared__ double tab[W][4 * kMaxS3];
    __shared__ uint64_t mk[W][2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)W + w;
    if (i >= n) return;
    const double p[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    const int32_t r0 = rowptr[i], rl = rowptr[i + 1] - r0;
    int S = 0;
    for (int base = 0; base < rl; base += 32) {
        const int c = base + lane;
        bool sup = false;
        int32_t j = -1;
        if (c < rl) {
            j = col[r0 + c];
            const double dx = p[0] - x[3 * (int64_t)j], dy = p[1] - x[3 * (int64_t)j + 1], dz = p[2] - x[3 * (int64_t)j + 2];
            sup = dx * dx + dy * dy + dz * dz < R[j] * R[j];
        }
        const unsigned b = __ballot_sync(0xffffffffu, sup);
        const int slot = S + __popc(b & ((1u << lane) - 1u));
        if (sup && slot < kMaxS3) {
            fp[w][slot] = r0 + c;
            fx[w][3 * slot] = x[3 * (int64_t)j];
            fx[w][3 * slot + 1] = x[3 * (int64_t)j + 1];
            fx[w][3 * slot + 2] = x[3 * (int64_t)j + 2];
            fR2[w][slot] = R[j] * R[j];
            finvh[w][slot] = 2.0 / R[j];
            fV[w][slot] = V[j];
        }
        S += __popc(b);
    }
    if (S > kMaxS3) {
        if (lane == 0) atomicOr(flag, 2);
        return;
    }
    __syncwarp();
    if (!rk3_warp<NP>(p, 0.5 * R[i], S, fx[w], fR2[w], finvh[w], fV[w], tab[w], kMaxS3, mk[w])) {
        if (lane == 0) atomicOr(flag, 1);
        return;
    }
    __syncwarp();
    for (int a = lane; a < S; a += 32) interp[fp[w][a]] = fV[w][a] * tab[w][a];
}

}  // namespace

static mlpg_status check_flag3(mlpg_ctx *ctx, const char *stage) {
    int flag = 0;
    CU(ctx, cudaMemcpyAsync(&flag, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    CU(ctx, cudaStreamSynchronize(ctx->stream));
    if (flag & 1) return set_err(ctx, MLPG_ERR_RK_SINGULAR, std::string(stage) + ": RK moment matrix singular");
    if (flag & 2) return set_err(ctx, MLPG_ERR_ARG, std::string(stage) + ": too many functions reach one element");
    if (flag & 8) return set_err(ctx, MLPG_ERR_GEOMETRY, std::string(stage) + ": support pair outside the overlap pattern");
    return MLPG_OK;
}

mlpg_status run_interp_3d(mlpg_ctx *ctx) {
    MLPG_TRY(dalloc(ctx, &ctx->interp, ctx->nnz));
    if (!ctx->d_flag) MLPG_TRY(dalloc(ctx, &ctx->d_flag, 1));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->interp, 0, ctx->nnz * sizeof(double), ctx->stream));
    const int64_t blocks = (ctx->n + 3) / 4;
    if (ctx->opt.rk_order == 0)
        k_interp_3d<1><<<(unsigned)blocks, 128, 0, ctx->stream>>>(ctx->n, ctx->x, ctx->R, ctx->V, ctx->rowptr,
                                                                  ctx->col, ctx->interp, ctx->d_flag);
    else
        k_interp_3d<4><<<(unsigned)blocks, 128, 0, ctx->stream>>>(ctx->n, ctx->x, ctx->R, ctx->V, ctx->rowptr,
                                                                  ctx->col, ctx->interp, ctx->d_flag);
    CU_LAUNCH(ctx);
    return check_flag3(ctx, "interpolation");
}

mlpg_status run_assemble_3d(mlpg_ctx *ctx) {
    const int n1 = 2;   // 2x2x2 tetrahedron rule, 2x2 triangle rule (degree 3)
    {
        double xi[3 * kMaxQ3], w[kMaxQ3], ti[2 * kMaxQ3], tw[kMaxQ3];
        tet_rule(n1, xi, w);
        triangle_rule(n1, ti, tw);
        CU(ctx, cudaMemcpyToSymbolAsync(c3_tet_xi, xi, sizeof(double) * 3 * n1 * n1 * n1, 0,
                                        cudaMemcpyHostToDevice, ctx->stream));
        CU(ctx, cudaMemcpyToSymbolAsync(c3_tet_w, w, sizeof(double) * n1 * n1 * n1, 0, cudaMemcpyHostToDevice,
                                        ctx->stream));
        CU(ctx, cudaMemcpyToSymbolAsync(c3_tri_xi, ti, sizeof(double) * 2 * n1 * n1, 0, cudaMemcpyHostToDevice,
                                        ctx->stream));
        CU(ctx, cudaMemcpyToSymbolAsync(c3_tri_w, tw, sizeof(double) * n1 * n1, 0, cudaMemcpyHostToDevice,
                                        ctx->stream));
    }
    ctx->nmats = mlpg_n_matrices(3);
    ctx->nvecs = mlpg_n_vectors(3);
    if (!ctx->mats) MLPG_TRY(dalloc(ctx, &ctx->mats, (size_t)ctx->nmats * ctx->nnz));
    if (!ctx->vecs) MLPG_TRY(dalloc(ctx, &ctx->vecs, (size_t)ctx->nvecs * ctx->n));
    CU(ctx, cudaMemsetAsync(ctx->mats, 0, sizeof(double) * ctx->nmats * ctx->nnz, ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->vecs, 0, sizeof(double) * ctx->nvecs * ctx->n, ctx->stream));
    CU(ctx, cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), ctx->stream));
    Asm3Args a;
    a.n = ctx->n; a.nnz = ctx->nnz;
    a.x = ctx->x; a.R = ctx->R; a.V = ctx->V; a.sig_t = ctx->sig_t; a.sig_s = ctx->sig_s; a.q = ctx->q;
    a.rowptr = ctx->rowptr; a.col = ctx->col;
    a.mats = ctx->mats; a.vecs = ctx->vecs; a.flag = ctx->d_flag;
    // volume elements: groups of tetrahedra, then the elements of groups with too many functions
    a.nelem = ctx->ntet; a.owner = ctx->tet_owner; a.face = nullptr; a.ev = ctx->tet_v; a.nq = n1 * n1 * n1; a.list = nullptr;
    cudaStream_t s = ctx->stream;
    size_t smem = sizeof(double) * (size_t)a.nq * 4 * kMaxS3;
    if (a.nelem > 0) {
        // group list, list of skipped elements, two counters; G of the lower entries
        int2 *grp = nullptr;
        int32_t *skip = nullptr;
        int *cnt = nullptr;
        double *gt = nullptr;
        MLPG_TRY(dalloc(ctx, &grp, a.nelem));
        MLPG_TRY(dalloc(ctx, &skip, a.nelem));
        MLPG_TRY(dalloc(ctx, &cnt, 2));
        MLPG_TRY(assembly_scratch(ctx, &gt));
        CU(ctx, cudaMemsetAsync(cnt, 0, 2 * sizeof(int), s));
        CU(ctx, cudaMemsetAsync(gt, 0, sizeof(double) * 9 * ctx->nnz, s));
        k_tet_groups<<<(unsigned)((a.nelem + 127) / 128), 128, 0, s>>>(a.nelem, a.owner, a.ev, grp, cnt);
        CU_LAUNCH(ctx);
        int ngrp = 0, nskip = 0;
        CU(ctx, cudaMemcpyAsync(&ngrp, cnt, sizeof(int), cudaMemcpyDeviceToHost, s));
        CU(ctx, cudaStreamSynchronize(s));
        const int gsmem = kGrpEntries * 32;
        if (ctx->opt.rk_order == 0) {
            CU(ctx, cudaFuncSetAttribute(k_assemble_3d_grp<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsmem));
            k_assemble_3d_grp<1><<<(unsigned)ngrp, kGrpThreads, gsmem, s>>>(a, grp, gt, cnt + 1, skip);
        } else {
            CU(ctx, cudaFuncSetAttribute(k_assemble_3d_grp<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsmem));
            k_assemble_3d_grp<4><<<(unsigned)ngrp, kGrpThreads, gsmem, s>>>(a, grp, gt, cnt + 1, skip);
        }
        CU_LAUNCH(ctx);
        k_mirror_3d<<<(unsigned)((ctx->n * 32 + 255) / 256), 256, 0, s>>>(ctx->n, ctx->nnz, ctx->rowptr, ctx->col, ctx->V,
                                                                        gt, ctx->mats, ctx->d_flag);
        CU_LAUNCH(ctx);
        CU(ctx, cudaMemcpyAsync(&nskip, cnt + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
        CU(ctx, cudaStreamSynchronize(s));
        if (nskip > 0) {
            a.list = skip;
            if (ctx->opt.rk_order == 0) k_assemble_3d<false, 1><<<(unsigned)nskip, kThreads3, smem, s>>>(a);
            else k_assemble_3d<false, 4><<<(unsigned)nskip, kThreads3, smem, s>>>(a);
            CU_LAUNCH(ctx);
            a.list = nullptr;
        }
    }
    // boundary elements
    a.nelem = ctx->nbtri; a.owner = ctx->tri_owner; a.face = ctx->tri_face; a.ev = ctx->tri_v; a.nq = n1 * n1;
    smem = sizeof(double) * (size_t)a.nq * 4 * kMaxS3;
    if (a.nelem > 0) {
        if (ctx->opt.rk_order == 0) k_assemble_3d<true, 1><<<(unsigned)a.nelem, kThreads3, smem, ctx->stream>>>(a);
        else k_assemble_3d<true, 4><<<(unsigned)a.nelem, kThreads3, smem, ctx->stream>>>(a);
        CU_LAUNCH(ctx);
    }
    return check_flag3(ctx, "assembly");
}

}  // namespace mlpg
