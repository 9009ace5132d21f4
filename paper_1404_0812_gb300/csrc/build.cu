// Batched per-stencil build of the RBF-FD surface Laplacian (Sections 2-5).
//
// GB300 design.  The local algebra must be float64 (kappa_T ~ 1e12 leaves
// about four digits), and GB300's FP64 rate is a few operations per clock
// per SM, so every FP64 warp instruction has to do 32 useful operations.
// One thread owns one stencil ("lane per stencil"): all lanes of a warp run
// the same instruction stream on different stencils, with no shuffles and no
// idle lanes inside the O(m^3) factorisations.  Each lane's matrices live
// in a global scratch area interleaved across the 32 lanes of its warp, so
// every load is one 256-byte coalesced transaction (L1/L2 cached).
// The factorisation is a packed lower Cholesky of Phi with 4x4 register
// tiles (16 FMAs per 8 loads).
//
// Condition number (Section 5, kappa_2 of the symmetric augmented A of
// Eq. rbf_linsys): Phi is positive definite for the Gaussian and IMQ
// kernels, so A = [[Phi, 1], [1^T, 0]] is solved through Phi = L L^T and
// its Schur complement s = 1^T Phi^{-1} 1.  max|lambda(A)| comes from a
// short Lanczos run with A in float32 (on a float32 copy of Phi: the
// dominant eigenvalue is well separated and well conditioned, and a
// relative error of ~1e-6 in kappa moves the root by ~1e-7 in ln eps), and
// 1 / min|lambda(A)| from a float64 Lanczos run with A^{-1}; each run stops
// when its extreme Ritz value settles (relative change 1e-6).  The Ritz
// values of the small tridiagonal are found by Sturm-count bisection in
// float32 (relative accuracy ~1e-7, far below the float64 noise of kappa).
//
// Shape parameter search (Eq. target_cond): F(x) = ln(kappa(A(e^x)) /
// kappa_T) in x = ln(eps * r_s) (coordinates translated to the stencil
// centre and scaled by the stencil radius r_s).  Safeguarded Newton from the
// oracle's starting point (eps_0 = 1 / mean neighbour distance) or from a
// learned prediction: dF/dx comes with every evaluation from the
// Hellmann-Feynman derivative of the smallest eigenvalue (its eigenvector is
// the Ritz vector of the A^{-1} Lanczos run); a bracket and bisection guard
// the steps; the search
// stops when the Newton step is below half the eps tolerance.  Lanes that
// finish take the next stencil from a global counter, so a warp stays full
// until the work runs out.  Groups of different stencil size are processed
// largest first in the same persistent launch.  Node sets that do not fill the
// chip with a lane per stencil take the same steps on teams of lanes (team.cu).
//
// Weights (Eqs. grad_x_f_interp, surface_lap_P1): only the first row of
// L_P = sum_d G^d G^d is needed, so with A symmetric
//   g_d = (A^{-1} [B^d row 0; 0])[:n],  v = sum_d B^{dT} g_d,
//   w = (A^{-1} [v; 0])[:n] / r_s^2,
// four solves and one pass over the pairs, equal in exact arithmetic to
// forming the full G^d (which the oracle does).
#include "dd.cuh"
#include "stencil.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <cstring>

namespace rbffd {
namespace {

// ---------------------------------------------------------------------------
// lane-private scratch, interleaved across the warp
//
// Size of the code.  The warps of an SM are in different phases of their
// stencils, and with the loops unrolled as the compiler likes the search was
// 483 KB of instructions: warps waited longer for instructions than for
// anything else (38 % of their time, 1M nodes in four sizes 421 ms).  So the
// lane functions' loops are not unrolled (unroll 1) where their bodies already
// keep loads in flight, the triangular solves are functions called from several
// places, views and layouts go by value (a reference is read again after every
// store), and the kernel function is a template argument: 192 KB, 385 ms.  Only
// the solves' chunk loops keep the compiler's unrolling (404 ms without, 397
// with, before the other changes).  For the same reason variants with more code
// were slower: the solves' next chunk fetched ahead 461 ms (392 on the smaller
// code, its registers spill), 168 registers for it on three blocks per SM 449 ms.
// ---------------------------------------------------------------------------
struct Lane {
    double* p;   // points at element 0 of this lane
    __device__ __forceinline__ double& operator[](int e) const { return p[(int64_t)e * 32]; }
};

// float32 view of a region of the same scratch: float element e of this lane
// lies at e * 32 + lane floats from the region's start (region start R in
// double units per lane = R * 32 doubles from the warp's base), so a region
// of k doubles per lane holds 2k floats per lane, again one coalesced
// transaction per warp access.
struct LaneF {
    float* p;
    __device__ __forceinline__ float& operator[](int e) const { return p[(int64_t)e * 32]; }
};

__device__ __forceinline__ LaneF float_view(const Lane& S, int region) {
    const int lane = threadIdx.x & 31;
    return LaneF{reinterpret_cast<float*>(S.p - lane + (int64_t)region * 32) + lane};
}

struct Layout {
    int m;       // padded stencil size (multiple of 4)
    int P;       // m (m + 1) / 2
    int R2, L, PH, XS, NS, U, ID, Q0, Q2, GV, HV, QB, RV;
    int PF, FV;  // float32 regions (search only): copy of Phi, three Lanczos vectors
    int size;    // doubles per lane
};

// full = true: the weights kernel's layout; full = false: the search's, which
// adds the Lanczos basis, the Ritz vector and the float32 regions of the
// lambda_max run (both hold the Phi copy, normals and gradient vectors: the
// search computes the weights from its last factorisation).
__host__ __device__ inline Layout make_layout(int m, bool full) {
    Layout l;
    l.m = m;
    l.P = m * (m + 1) / 2;
    int o = 0;
    l.R2 = o; o += l.P;
    l.L = o; o += l.P;
    l.PH = o; o += l.P;
    l.XS = o; o += 3 * m;
    l.U = o; o += m;
    l.ID = o; o += m;
    l.Q0 = o; o += m;
    l.Q2 = o; o += m;
    l.NS = o; o += 3 * m;
    l.GV = o; o += 3 * m;
    l.HV = o; o += 3 * m;
    l.QB = l.RV = l.PF = l.FV = -1;
    if (!full) {
        l.QB = o; o += LANCZOS_KMAX * m;   // Lanczos basis
        l.RV = o; o += m;
        l.PF = o; o += (l.P + 1) / 2;      // P floats
        l.FV = o; o += (3 * m + 1) / 2;    // 3 m floats
    }
    l.size = o;
    return l;
}

// ---------------------------------------------------------------------------
// stencil geometry: centre-translated, r_s-scaled coordinates and normals
// ---------------------------------------------------------------------------
__device__ Geo load_geometry(const Lane S, const Layout ly, int n, const int32_t* __restrict__ idx,
                             int64_t off, int npad, int64_t lr, const double* __restrict__ X,
                             const double* __restrict__ NR, bool with_normals) {
    int c = idx[ell_elem(off, npad, lr, 0)];
    double cx = X[3 * (int64_t)c], cy = X[3 * (int64_t)c + 1], cz = X[3 * (int64_t)c + 2];
    double rs2 = 0.0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        int k = idx[ell_elem(off, npad, lr, j)];
        double dx = X[3 * (int64_t)k] - cx, dy = X[3 * (int64_t)k + 1] - cy,
               dz = X[3 * (int64_t)k + 2] - cz;
        S[ly.XS + j] = dx;
        S[ly.XS + ly.m + j] = dy;
        S[ly.XS + 2 * ly.m + j] = dz;
        rs2 = fmax(rs2, dx * dx + dy * dy + dz * dz);
        if (with_normals) {
            double nx = NR[3 * (int64_t)k], ny = NR[3 * (int64_t)k + 1], nz = NR[3 * (int64_t)k + 2];
            double inv = rsqrt(nx * nx + ny * ny + nz * nz);
            S[ly.NS + j] = nx * inv;
            S[ly.NS + ly.m + j] = ny * inv;
            S[ly.NS + 2 * ly.m + j] = nz * inv;
        }
    }
    Geo g;
    g.rs = sqrt(rs2);
    double inv = 1.0 / g.rs;
    double sum = 0.0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        double x = S[ly.XS + j] * inv, y = S[ly.XS + ly.m + j] * inv, z = S[ly.XS + 2 * ly.m + j] * inv;
        S[ly.XS + j] = x;
        S[ly.XS + ly.m + j] = y;
        S[ly.XS + 2 * ly.m + j] = z;
        if (j > 0) sum += sqrt(x * x + y * y + z * z);
    }
    g.mean_d = sum / (double)(n - 1);
    // pairwise squared distances (lower triangle, diagonal 0)
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        double xi = S[ly.XS + i], yi = S[ly.XS + ly.m + i], zi = S[ly.XS + 2 * ly.m + i];
        int base = pk(i, 0);
#pragma unroll 1
        for (int j = 0; j < i; ++j) {
            double dx = xi - S[ly.XS + j], dy = yi - S[ly.XS + ly.m + j], dz = zi - S[ly.XS + 2 * ly.m + j];
            S[ly.R2 + base + j] = dx * dx + dy * dy + dz * dz;
        }
        S[ly.R2 + base + i] = 0.0;
    }
    return g;
}

// Phi(eps) into region dst (lower packed, m x m, identity on the padding);
// optionally a copy into region cpy and a float32 copy into region fcpy.
__device__ void assemble_phi(const Lane S, const Layout ly, int n, int kernel, double eps_s,
                             int dst, int cpy, int fcpy = -1) {
    double e2 = eps_s * eps_s;
    const LaneF F = float_view(S, fcpy >= 0 ? fcpy : 0);
#pragma unroll 1
    for (int i = 0; i < ly.m; ++i) {
        int base = pk(i, 0);
        if (i < n) {
            int j = 0;
#pragma unroll 1
            for (; j + 4 <= i; j += 4) {   // four loads ahead of the stores
                double v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = S[ly.R2 + base + j + q];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = phi_of(kernel, e2, v[q]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    S[dst + base + j + q] = v[q];
                    if (cpy >= 0) S[cpy + base + j + q] = v[q];
                    if (fcpy >= 0) F[base + j + q] = (float)v[q];
                }
            }
#pragma unroll 1
            for (; j < i; ++j) {
                double v = phi_of(kernel, e2, S[ly.R2 + base + j]);
                S[dst + base + j] = v;
                if (cpy >= 0) S[cpy + base + j] = v;
                if (fcpy >= 0) F[base + j] = (float)v;
            }
        } else {
#pragma unroll 1
            for (int j = 0; j < i; ++j) {
                S[dst + base + j] = 0.0;
                if (cpy >= 0) S[cpy + base + j] = 0.0;
                if (fcpy >= 0) F[base + j] = 0.f;
            }
        }
        S[dst + base + i] = 1.0;
        if (cpy >= 0) S[cpy + base + i] = 1.0;
        if (fcpy >= 0) F[base + i] = 1.f;
    }
}

// acc[a][b] -= sum_{k < jb} L(ib + a, k) L(jb + b, k) for the first R rows
// of the tile (software-pipelined: the loads of step k + 1 are in flight
// while the 4 R FMAs of step k issue)
template <int R>
__device__ __forceinline__ void chol_tile_accumulate(const Lane& S, int L, int ib, int jb, double (&acc)[R][4]) {
    const int ra = L + pk(ib, 0), rb = L + pk(jb, 0);
    double xa[R], yb[4];
#pragma unroll
    for (int a = 0; a < R; ++a) xa[a] = S[ra + a * ib + a * (a + 1) / 2];
#pragma unroll
    for (int b = 0; b < 4; ++b) yb[b] = S[rb + b * jb + b * (b + 1) / 2];
#pragma unroll 1
    for (int k = 0; k < jb; ++k) {
        double xn[R], yn[4];
        const int kn = k + 1 < jb ? k + 1 : k;
#pragma unroll
        for (int a = 0; a < R; ++a) xn[a] = S[ra + a * ib + a * (a + 1) / 2 + kn];
#pragma unroll
        for (int b = 0; b < 4; ++b) yn[b] = S[rb + b * jb + b * (b + 1) / 2 + kn];
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fma(-xa[a], yb[b], acc[a][b]);
#pragma unroll
        for (int a = 0; a < R; ++a) xa[a] = xn[a];
#pragma unroll
        for (int b = 0; b < 4; ++b) yb[b] = yn[b];
    }
}

// The diagonal tile (ib = jb): its lower half only, ten of sixteen FMAs and
// half the loads of a step.
__device__ __forceinline__ void chol_diag_accumulate(const Lane& S, int L, int jb, double (&acc)[4][4]) {
    const int r = L + pk(jb, 0);
    double x[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) x[a] = S[r + a * jb + a * (a + 1) / 2];
#pragma unroll 1
    for (int k = 0; k < jb; ++k) {
        double xn[4];
        const int kn = k + 1 < jb ? k + 1 : k;
#pragma unroll
        for (int a = 0; a < 4; ++a) xn[a] = S[r + a * jb + a * (a + 1) / 2 + kn];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b <= a; ++b) acc[a][b] = fma(-x[a], x[b], acc[a][b]);
#pragma unroll
        for (int a = 0; a < 4; ++a) x[a] = xn[a];
    }
}

// Off-diagonal tile (ib > jb): rows ib .. ib + R - 1 of column block jb,
// from the diagonal block's factor Ld and 1 / L_ii.  R < 4 only in the last
// row block, whose other rows are padding (identity rows of Phi: their L
// entries stay the zeros the assembly wrote, and no real row reads them).
template <int R>
__device__ __forceinline__ void chol_tile_offdiag(const Lane S, const Layout ly, int ib, int jb,
                                                  const double (&Ld)[4][4]) {
    const int L = ly.L;
    double acc[R][4];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = S[L + pk(ib + a, jb + b)];
    if (jb > 0) chol_tile_accumulate<R>(S, L, ib, jb, acc);
#pragma unroll
    for (int a = 0; a < R; ++a) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double v = acc[a][b];
#pragma unroll
            for (int c = 0; c < b; ++c) v = fma(-acc[a][c], Ld[b][c], v);
            acc[a][b] = v * S[ly.ID + jb + b];
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) S[L + pk(ib + a, jb + b)] = acc[a][b];
    }
}

// In-place packed Cholesky Phi = L L^T (left-looking, 4x4 register tiles).
// ID receives 1 / L_ii.  Returns false when a pivot is not positive.  Rows
// n .. m-1 are padding (identity in Phi and in L): the off-diagonal tiles of
// the last row block leave them out.
__device__ bool cholesky(const Lane S, const Layout ly, int n) {
    const int m = ly.m, L = ly.L;
    bool ok = true;
#pragma unroll 1
    for (int jb = 0; jb < m; jb += 4) {
        double Ld[4][4];
        {
            // diagonal block (all four rows, padding included: it sets 1 / L_ii = 1 there)
            const int ib = jb;
            double acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = (a >= b) ? S[L + pk(ib + a, jb + b)] : 0.0;
            if (jb > 0) chol_diag_accumulate(S, L, jb, acc);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                double d = acc[b][b];
                if (!(d > 0.0)) {
                    ok = false;
                    d = 1.0;
                }
                double l = sqrt(d);
                double il = 1.0 / l;
                acc[b][b] = l;
                S[ly.ID + jb + b] = il;
#pragma unroll
                for (int a = b + 1; a < 4; ++a) acc[a][b] *= il;
#pragma unroll
                for (int c = b + 1; c < 4; ++c)
#pragma unroll
                    for (int a = c; a < 4; ++a) acc[a][c] = fma(-acc[a][b], acc[c][b], acc[a][c]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b <= a; ++b) {
                    Ld[a][b] = acc[a][b];
                    S[L + pk(jb + a, jb + b)] = acc[a][b];
                }
        }
#pragma unroll 1
        for (int ib = jb + 4; ib < m; ib += 4) {
            const int rows = n - ib;   // >= 1: padding is less than one block
            if (rows >= 4) chol_tile_offdiag<4>(S, ly, ib, jb, Ld);
            else if (rows == 3) chol_tile_offdiag<3>(S, ly, ib, jb, Ld);
            else if (rows == 2) chol_tile_offdiag<2>(S, ly, ib, jb, Ld);
            else chol_tile_offdiag<1>(S, ly, ib, jb, Ld);
        }
        if (!ok) return false;
    }
    return true;
}

// x_d <- Phi^{-1} x_d for NR right-hand sides (regions V0 + d VS, length m) using
// L and ID: forward L y = x, then backward L^T x = y, in blocks of four rows.
// A chunk of C = 4 / NR columns (forward) or rows (backward) is loaded before
// its FMAs issue, so each step keeps 4 C + NR C loads in flight for 4 C NR
// FMAs; every row still sums its columns in increasing order (forward) and
// receives the blocks' updates from the last block down (backward), whatever
// NR is, so a right-hand side gets the same bits alone or with others.
template <int NR>
__device__ __noinline__ void chol_solve_multi(const Lane S, const Layout ly, int V0, int VS) {
    constexpr int C = NR == 1 ? 4 : NR == 2 ? 2 : 1;
    const int m = ly.m, L = ly.L;
    for (int ib = 0; ib < m; ib += 4) {   // forward
        double t[4][NR];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int d = 0; d < NR; ++d) t[a][d] = S[V0 + d * VS + ib + a];
        const int r = pk(ib, 0);   // row ib + a starts at r + a ib + a (a + 1) / 2
        for (int k = 0; k < ib; k += C) {   // ib is a multiple of 4, hence of C
            double y[C][NR], l[4][C];
#pragma unroll
            for (int q = 0; q < C; ++q)
#pragma unroll
                for (int d = 0; d < NR; ++d) y[q][d] = S[V0 + d * VS + k + q];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int q = 0; q < C; ++q) l[a][q] = S[L + r + a * ib + a * (a + 1) / 2 + k + q];
#pragma unroll
            for (int q = 0; q < C; ++q)
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int d = 0; d < NR; ++d) t[a][d] = fma(-l[a][q], y[q][d], t[a][d]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < a; ++c) {
                const double l = S[L + pk(ib + a, ib + c)];
#pragma unroll
                for (int d = 0; d < NR; ++d) t[a][d] = fma(-l, t[c][d], t[a][d]);
            }
            const double id = S[ly.ID + ib + a];
#pragma unroll
            for (int d = 0; d < NR; ++d) {
                t[a][d] *= id;
                S[V0 + d * VS + ib + a] = t[a][d];
            }
        }
    }
    for (int kb = m - 4; kb >= 0; kb -= 4) {   // backward
        double t[4][NR];
#pragma unroll
        for (int b = 3; b >= 0; --b) {
#pragma unroll
            for (int d = 0; d < NR; ++d) t[b][d] = S[V0 + d * VS + kb + b];
#pragma unroll
            for (int c = b + 1; c < 4; ++c) {
                const double l = S[L + pk(kb + c, kb + b)];
#pragma unroll
                for (int d = 0; d < NR; ++d) t[b][d] = fma(-l, t[c][d], t[b][d]);
            }
            const double id = S[ly.ID + kb + b];
#pragma unroll
            for (int d = 0; d < NR; ++d) {
                t[b][d] *= id;
                S[V0 + d * VS + kb + b] = t[b][d];
            }
        }
        const int r0 = pk(kb, 0), r1 = pk(kb + 1, 0), r2 = pk(kb + 2, 0), r3 = pk(kb + 3, 0);
        for (int i = 0; i < kb; i += C) {
            double l[4][C], v[C][NR];
#pragma unroll
            for (int q = 0; q < C; ++q) {
                l[0][q] = S[L + r0 + i + q];
                l[1][q] = S[L + r1 + i + q];
                l[2][q] = S[L + r2 + i + q];
                l[3][q] = S[L + r3 + i + q];
#pragma unroll
                for (int d = 0; d < NR; ++d) v[q][d] = S[V0 + d * VS + i + q];
            }
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int q = 0; q < C; ++q)
#pragma unroll
                    for (int d = 0; d < NR; ++d) v[q][d] = fma(-l[b][q], t[b][d], v[q][d]);
#pragma unroll
            for (int q = 0; q < C; ++q)
#pragma unroll
                for (int d = 0; d < NR; ++d) S[V0 + d * VS + i + q] = v[q][d];
        }
    }
}

// x <- Phi^{-1} x (x in region V of length m)
__device__ void chol_solve(const Lane S, const Layout ly, int V) {
    chol_solve_multi<1>(S, ly, V, 0);
}

// y = Phi x in float32 from the packed float32 copy F of Phi, x and y at
// float offsets x, y of V.  Rows in blocks of four (four independent FMA
// chains; each x_j loaded once per block): columns left of the block from
// the block's rows, the 4 x 4 diagonal block, and columns right of it from
// the rows below (symmetry).  The padding rows of Phi are the identity and
// entries n..m-1 of x are zero, so the loops run to m.
__device__ void phi_mul_f32(const LaneF F, const LaneF V, int x, int y, int m) {
    for (int ib = 0; ib < m; ib += 4) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const int r = pk(ib, 0);   // row ib + a starts at r + a ib + a (a + 1) / 2
        for (int j = 0; j < ib; ++j) {
            const float xj = V[x + j];
#pragma unroll
            for (int a = 0; a < 4; ++a) acc[a] = fmaf(F[r + a * ib + a * (a + 1) / 2 + j], xj, acc[a]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float xc = V[x + ib + c];
#pragma unroll
            for (int a = 0; a < 4; ++a)
                acc[a] = fmaf(F[a >= c ? pk(ib + a, ib + c) : pk(ib + c, ib + a)], xc, acc[a]);
        }
        for (int j = ib + 4; j < m; ++j) {
            const float xj = V[x + j];
            const int rj = pk(j, ib);
#pragma unroll
            for (int a = 0; a < 4; ++a) acc[a] = fmaf(F[rj + a], xj, acc[a]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) V[y + ib + a] = acc[a];
    }
}

// max|lambda(A)| of A = [[Phi, 1], [1^T, 0]] by Lanczos in float32 on the
// float32 copy of Phi (region PF, written by assemble_phi) with vectors in
// region FV (m entries each plus a border scalar).  The start vector is
// mostly the constant vector, close to the dominant eigenvector when Phi is
// nearly flat (Phi ~ 1 1^T), plus a 1 % oscillation so that no eigenvector
// is missed; two steps can then settle.  The dominant eigenvalue is well
// conditioned (Weyl: float32 rounding of Phi and of the products moves it
// by ~sqrt(m) 6e-8 relative), so float32 costs kappa no accuracy that the
// root finder would notice and takes the run off the float64 pipe.
__device__ double lanczos_max_f32(const Lane S, const Layout ly, int n, double rtol) {
    const int m = ly.m;
    const LaneF F = float_view(S, ly.PF), V = float_view(S, ly.FV);
    float al[LANCZOS_KMAX], b2[LANCZOS_KMAX];
    double alpha_d[LANCZOS_KMAX], beta_d[LANCZOS_KMAX];
    int qp = 0, q_ = m, w = 2 * m;
    float nrm2 = 0.f;
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        const float v = i < n ? 1.0f + 0.01f * (__cosf(1.7f * (float)i + 0.3f) + 0.1f) : 0.f;
        V[q_ + i] = v;
        V[qp + i] = 0.f;
        nrm2 = fmaf(v, v, nrm2);
    }
    float qb = 0.1f, qpb = 0.f;
    nrm2 = fmaf(qb, qb, nrm2);
    const float inrm = rsqrtf(nrm2);
#pragma unroll 1
    for (int i = 0; i < n; ++i) V[q_ + i] *= inrm;
    qb *= inrm;
    float beta = 0.f;
    double prev = -1.0, ext = 0.0;
#pragma unroll 1
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        // [Phi q + qb 1; 1^T q]
        phi_mul_f32(F, V, q_, w, m);
        float sum = 0.f;
#pragma unroll 1
        for (int i = 0; i < n; ++i) sum += V[q_ + i];
        float wb = fmaf(-beta, qpb, sum);
        float ap[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int i = 0; i < m; i += 4) {
            float v[4], x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = V[w + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = V[qp + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = fmaf(-beta, x[q], i + q < n ? v[q] + qb : v[q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = V[q_ + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                V[w + i + q] = v[q];
                ap[q] = fmaf(x[q], v[q], ap[q]);
            }
        }
        const float a = fmaf(qb, wb, (ap[0] + ap[1]) + (ap[2] + ap[3]));
        float bp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int i = 0; i < m; i += 4) {
            float v[4], x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = V[w + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = V[q_ + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = fmaf(-a, x[q], v[q]);
                V[w + i + q] = v[q];
                bp[q] = fmaf(v[q], v[q], bp[q]);
            }
        }
        wb = fmaf(-a, qb, wb);
        const float bn = sqrtf(fmaf(wb, wb, (bp[0] + bp[1]) + (bp[2] + bp[3])));
        alpha_d[j] = a;
        beta_d[j] = bn;
        // scaled tridiagonal (Gershgorin bound as the scale)
        double G = 0.0;
#pragma unroll 1
        for (int i = 0; i <= j; ++i) {
            double r = fabs(alpha_d[i]) + (i < j ? beta_d[i] : 0.0) + (i > 0 ? beta_d[i - 1] : 0.0);
            G = fmax(G, r);
        }
        const double ig = 1.0 / G;
#pragma unroll 1
        for (int i = 0; i <= j; ++i) {
            al[i] = (float)(alpha_d[i] * ig);
            const float bb = (float)(beta_d[i] * ig);
            b2[i] = bb * bb;
        }
        ext = tri_max_abs(al, b2, j + 1, G);
        if (j + 1 >= 2 && fabs(ext - prev) <= rtol * ext) break;
        // an invariant subspace to float32 precision: the residual bounds the
        // error of the Ritz value by bn
        if (bn <= 1e-6f * fabsf(a)) break;
        prev = ext;
        beta = bn;
        const float ib = 1.f / bn;
        const int t = qp;
        qp = q_;
        q_ = w;
        w = t;
        qpb = qb;
#pragma unroll 1
        for (int i = 0; i < n; ++i) V[q_ + i] *= ib;
        qb = wb * ib;
    }
    return ext;
}

// Start vector of the A^{-1} Lanczos run, normalised, in region QB (m
// entries) with its border entry returned: the previous evaluation's Ritz
// vector (region RV, border *vb) when warm, else the stencil's
// pseudo-random vector.
__device__ double lanczos_inv_start(const Lane S, const Layout ly, int n, bool warm, const double* vb,
                                    uint64_t seed) {
    const int m = ly.m;
    double nrm2 = 0.0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        double v = i < n ? (warm ? S[ly.RV + i] : unit_hash(seed * 131u + i)) : 0.0;
        S[ly.QB + i] = v;
        nrm2 += v * v;
    }
    double qb = warm ? *vb : unit_hash(seed * 131u + n);
    nrm2 += qb * qb;
    double inrm = rsqrt(nrm2);
#pragma unroll 1
    for (int i = 0; i < n; ++i) S[ly.QB + i] *= inrm;
    return qb * inrm;
}

// Lanczos with A^{-1} keeping its basis (regions QB + j m, borders in
// qbord[]) from the start vector in QB (border qb0; with w0_ready its first
// Phi^{-1} product is already in region Q2): returns the signed Ritz value
// theta of largest magnitude and writes the unit Ritz vector (m entries,
// border in *vb) to region RV.
__device__ double lanczos_inv_ritz(const Lane S, const Layout ly, int n, double s, double rtol, bool warm,
                                   double qb0, bool w0_ready, double* vb, double lmax = 0.0,
                                   double acc_lo = 0.0, double acc_hi = 0.0, bool* early = nullptr) {
    const int m = ly.m, w = ly.Q2;
    float al[LANCZOS_KMAX], b2[LANCZOS_KMAX];
    double alpha_d[LANCZOS_KMAX], beta_d[LANCZOS_KMAX], qbord[LANCZOS_KMAX + 1];
    qbord[0] = qb0;
    const int kmin = warm ? 2 : LANCZOS_KMIN;
    double beta = 0.0, prev = -1.0, ext = 0.0;
    int k = 0;
#pragma unroll 1
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        const int qj = ly.QB + j * m, qp = ly.QB + (j - 1) * m;
        // [c; d] = A^{-1} [f; g]: c0 = Phi^{-1} f, d = (1^T c0 - g) / s, c = c0 - d u
        if (j > 0 || !w0_ready) {
#pragma unroll 1
            for (int i = 0; i < m; i += 4) {
                double v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = S[qj + i + q];
#pragma unroll
                for (int q = 0; q < 4; ++q) S[w + i + q] = v[q];
            }
            chol_solve(S, ly, w);
        }
        double sp[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (int i = 0; i < m; i += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q) sp[q] += S[w + i + q];
        double dd = ((sp[0] + sp[1]) + (sp[2] + sp[3]) - qbord[j]) / s;
        double wb = dd;
        double ap[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (int i = 0; i < m; i += 4) {   // the loads of four elements ahead of the stores
            double v[4], x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = S[w + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = S[ly.U + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + q < n) v[q] = fma(-dd, x[q], v[q]);
            if (j > 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) x[q] = S[qp + i + q];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = fma(-beta, x[q], v[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = S[qj + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                S[w + i + q] = v[q];
                ap[q] = fma(x[q], v[q], ap[q]);
            }
        }
        if (j > 0) wb = fma(-beta, qbord[j - 1], wb);
        double a = fma(qbord[j], wb, (ap[0] + ap[1]) + (ap[2] + ap[3]));
        double bp[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (int i = 0; i < m; i += 4) {
            double v[4], x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = S[w + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = S[qj + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = fma(-a, x[q], v[q]);
                S[w + i + q] = v[q];
                bp[q] = fma(v[q], v[q], bp[q]);
            }
        }
        wb = fma(-a, qbord[j], wb);
        double bn = sqrt(fma(wb, wb, (bp[0] + bp[1]) + (bp[2] + bp[3])));
        alpha_d[j] = a;
        beta_d[j] = bn;
        k = j + 1;
        // the extreme eigenvalue, at the steps whose tests use it: the stops
        // from kmin on (which compare with the step before) and the early
        // acceptance
        const bool last = bn <= 1e-14 * fabs(a) || j + 1 == LANCZOS_KMAX;
        if (j + 1 >= kmin - 1 || last || (early && early_accept_factor(j + 1) > 0.0)) {
            double G = 0.0;
#pragma unroll 1
            for (int i = 0; i <= j; ++i) {
                double r = fabs(alpha_d[i]) + (i < j ? beta_d[i] : 0.0) + (i > 0 ? beta_d[i - 1] : 0.0);
                G = fmax(G, r);
            }
            double ig = 1.0 / G;
#pragma unroll 1
            for (int i = 0; i <= j; ++i) {
                al[i] = (float)(alpha_d[i] * ig);
                float bb = (float)(beta_d[i] * ig);
                b2[i] = bb * bb;
            }
            ext = tri_extreme(al, b2, j + 1, G);
        }
        if (early && j + 1 < kmin) {
            // early acceptance of a learned guess (see early_accept_factor);
            // the caller needs no Ritz vector then
            const double est = lmax * fabs(ext);
            if (est >= acc_lo && est <= early_accept_factor(j + 1) * acc_hi) {
                *early = true;
                return ext;
            }
        }
        if (j + 1 >= kmin && fabs(fabs(ext) - prev) <= rtol * fabs(ext)) break;
        if (last) break;
        prev = fabs(ext);
        beta = bn;
        const double ib = 1.0 / bn;
        const int qn = ly.QB + (j + 1) * m;
#pragma unroll 1
        for (int i = 0; i < m; i += 4) {
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = S[w + i + q];
#pragma unroll
            for (int q = 0; q < 4; ++q) S[qn + i + q] = v[q] * ib;
        }
        qbord[j + 1] = wb * ib;
    }
    // Ritz vector  v = sum_j y_j q_j
    double y[LANCZOS_KMAX];
    tri_eigvec(alpha_d, beta_d, k, ext, y);
    double vbr = 0.0, nv = 0.0;
#pragma unroll 1
    for (int j = 0; j < k; ++j) vbr = fma(y[j], qbord[j], vbr);
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        double v = 0.0;
#pragma unroll 1
        for (int j = 0; j < k; ++j) v = fma(y[j], S[ly.QB + j * m + i], v);
        S[ly.RV + i] = v;
        nv = fma(v, v, nv);
    }
    nv = fma(vbr, vbr, nv);
    double inv = nv > 0.0 ? rsqrt(nv) : 0.0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) S[ly.RV + i] *= inv;
    *vb = vbr * inv;
    return ext;
}

// d lambda / d eps_s = v^T (dA/d eps_s) v for the unit eigenvector v in RV
// (Hellmann-Feynman; the border of A does not depend on eps).
__device__ double eig_derivative(const Lane S, const Layout ly, int n, int kernel, double eps_s) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int i = 1; i < n; ++i) {
        const int base = pk(i, 0);
        const double vi = S[ly.RV + i];
        double row[4] = {0.0, 0.0, 0.0, 0.0};
        int j = 0;
#pragma unroll 1
        for (; j + 4 <= i; j += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                double ph = S[ly.PH + base + j + q];
                double g = kernel == RBFFD_GAUSSIAN ? 2.0 * ph : ph * ph * ph;   // -dphi/(eps r^2)
                row[q] = fma(g * S[ly.R2 + base + j + q], S[ly.RV + j + q], row[q]);
            }
        }
#pragma unroll 1
        for (; j < i; ++j) {
            double ph = S[ly.PH + base + j];
            double g = kernel == RBFFD_GAUSSIAN ? 2.0 * ph : ph * ph * ph;
            row[0] = fma(g * S[ly.R2 + base + j], S[ly.RV + j], row[0]);
        }
        acc[i & 3] = fma(vi, (row[0] + row[1]) + (row[2] + row[3]), acc[i & 3]);
    }
    // dPhi_ij/d eps = -eps r_ij^2 phi^3 (IMQ) or -2 eps r_ij^2 phi (Gaussian);
    // the double sum over i != j is twice the lower-triangle sum
    return -2.0 * eps_s * ((acc[0] + acc[1]) + (acc[2] + acc[3]));
}

// kappa_2(A(eps_s)) (+inf when Phi is not numerically positive definite)
// and dF/dx, F = ln(kappa / kappa_T), x = ln eps_s: the derivative of
// -ln|lambda_min| by Hellmann-Feynman with the Ritz vector of the A^{-1}
// Lanczos run (d ln lambda_max / dx is ~1% of it on these stencils and is
// left out: Newton then still converges, linearly at rate ~0.01).  The Ritz
// vector stays in RV as the next evaluation's start vector.
// With acc_hi > 0 (a learned first guess) the A^{-1} run may stop early and
// set *early when the guess is proven acceptable (see early_accept_factor);
// kappa is then the run's lower estimate and no Ritz vector is formed.
__device__ double eval_kappa(const Lane S, const Layout ly, int n, int kernel, double eps_s, bool warm,
                             double* vb, double* theta_out, double* schur, uint64_t seed,
                             double acc_lo = 0.0, double acc_hi = 0.0, bool* early = nullptr) {
    double* dF = theta_out;
    *dF = NAN;
    *schur = 0.0;
    assemble_phi(S, ly, n, kernel, eps_s, ly.L, ly.PH, ly.PF);
    if (!cholesky(S, ly, n)) return INFINITY;
    // u = Phi^{-1} 1 and the A^{-1} run's first product Phi^{-1} q_0 in one
    // pass over L
    const double qb0 = lanczos_inv_start(S, ly, n, warm, vb, seed);
#pragma unroll 1
    for (int i = 0; i < ly.m; ++i) {
        S[ly.U + i] = i < n ? 1.0 : 0.0;
        S[ly.Q2 + i] = S[ly.QB + i];
    }
    chol_solve_multi<2>(S, ly, ly.U, ly.Q2 - ly.U);
    double s = 0.0;
#pragma unroll 1
    for (int i = 0; i < n; ++i) s += S[ly.U + i];
    if (!(s > 0.0)) return INFINITY;
    *schur = s;
    // the A run first: its estimate turns the A^{-1} run's Ritz values into
    // running estimates of kappa for the early acceptance
    double lmax = lanczos_max_f32(S, ly, n, LANCZOS_RTOL);
    double theta = lanczos_inv_ritz(S, ly, n, s, LANCZOS_RTOL, warm, qb0, true, vb, lmax, acc_lo, acc_hi,
                                    acc_hi > 0.0 ? early : nullptr);
    double k = lmax * fabs(theta);
    if (!isfinite(k)) return INFINITY;
    *dF = theta;   // the caller turns it into dF/dx with kappa_slope() when needed
    return k;
}

// dF/dx from the Ritz vector left in RV by eval_kappa (theta = its Ritz value)
__device__ inline double kappa_slope(const Lane S, const Layout ly, int n, int kernel, double eps_s,
                                     double theta) {
    return -eps_s * theta * eig_derivative(S, ly, n, kernel, eps_s);
}

// [c; d] = A^{-1} [f; 0] in place on region V (first n entries)
__device__ void aug_solve0(const Lane S, const Layout ly, int n, int V, double s) {
    chol_solve(S, ly, V);
    double sum = 0.0;
#pragma unroll 1
    for (int i = 0; i < n; ++i) sum += S[V + i];
    double d = sum / s;
#pragma unroll 1
    for (int i = 0; i < n; ++i) S[V + i] = fma(-d, S[ly.U + i], S[V + i]);
}

// Three right-hand sides (regions V, V + m, V + 2m) solved together: every
// element of L is loaded once for three FMAs.
__device__ void chol_solve_x3(const Lane S, const Layout ly, int V) {
    chol_solve_multi<3>(S, ly, V, ly.m);
}

__device__ void aug_solve0_x3(const Lane S, const Layout ly, int n, int V, double s) {
    const int m = ly.m;
    chol_solve_x3(S, ly, V);
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        double sum = 0.0;
#pragma unroll 1
        for (int i = 0; i < n; ++i) sum += S[V + d * m + i];
        double dd = sum / s;
#pragma unroll 1
        for (int i = 0; i < n; ++i) S[V + d * m + i] = fma(-dd, S[ly.U + i], S[V + d * m + i]);
    }
}

// First row of L_P from a factorised Phi(eps_s) (regions L, ID, U = Phi^{-1} 1,
// Schur complement s, the Phi copy PH, scaled coordinates XS and normals NS):
//   g_d = (A^{-1} [B^d row 0; 0])[:n],  h_i = P_i g_i,
//   v_j = sum_i psi_ij (x_i - x_j) . h_i,  w = (A^{-1} [v; 0])[:n].
// Leaves the scaled weights (times r_s^2) in region Q0.
__device__ void first_row_weights(const Lane S, const Layout ly, int n, int kernel, double eps_s, double s) {
    const int XS = ly.XS, m = ly.m;
    const double e2 = eps_s * eps_s;
    // centre projector P_0 = I - n_0 n_0^T; rhs_d,j = psi(r_0j) [P_0 (x_0 - x_j)]_d
    double n0x = S[ly.NS], n0y = S[ly.NS + m], n0z = S[ly.NS + 2 * m];
#pragma unroll 1
    for (int d = 0; d < 3; ++d)
#pragma unroll 1
        for (int i = 0; i < m; ++i) S[ly.GV + d * m + i] = 0.0;
#pragma unroll 1
    for (int j = 1; j < n; ++j) {
        double ph = S[ly.PH + pk(j, 0)];
        double ps = psi_from_phi(kernel, e2, ph);
        double dx = -S[XS + j], dy = -S[XS + m + j], dz = -S[XS + 2 * m + j];   // x_0 - x_j
        double nd = n0x * dx + n0y * dy + n0z * dz;
        S[ly.GV + j] = ps * (dx - n0x * nd);
        S[ly.GV + m + j] = ps * (dy - n0y * nd);
        S[ly.GV + 2 * m + j] = ps * (dz - n0z * nd);
    }
    aug_solve0_x3(S, ly, n, ly.GV, s);
    // h_i = P_i g_i
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        double gx = S[ly.GV + i], gy = S[ly.GV + m + i], gz = S[ly.GV + 2 * m + i];
        double nx = S[ly.NS + i], ny = S[ly.NS + m + i], nz = S[ly.NS + 2 * m + i];
        double nd = nx * gx + ny * gy + nz * gz;
        S[ly.HV + i] = gx - nx * nd;
        S[ly.HV + m + i] = gy - ny * nd;
        S[ly.HV + 2 * m + i] = gz - nz * nd;
    }
    const int V = ly.Q0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) S[V + i] = 0.0;
    // pair (i, j), j < i: v_j += psi (x_i - x_j) . h_i ; v_i += psi (x_j - x_i) . h_j,
    // summed with psi_shape and scaled by psi_scale at the end.
    // Rows in blocks of four: x_j, h_j and v_j are loaded once per column for
    // the four rows (a third of the scratch accesses of one row at a time).
    // Every v_j still receives the rows' contributions in row order and every
    // row sums its own in column order, so the result is the same bit for bit.
    int i = 0;
#pragma unroll 1
    for (; i + 4 <= n; i += 4) {
        double xi[4], yi[4], zi[4], hx[4], hy[4], hz[4], vi[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            xi[a] = S[XS + i + a];
            yi[a] = S[XS + m + i + a];
            zi[a] = S[XS + 2 * m + i + a];
            hx[a] = S[ly.HV + i + a];
            hy[a] = S[ly.HV + m + i + a];
            hz[a] = S[ly.HV + 2 * m + i + a];
            vi[a] = 0.0;
        }
        const int r0 = pk(i, 0);   // row i + a starts at r0 + a i + a (a + 1) / 2
#pragma unroll 1
        for (int j = 0; j < i; ++j) {
            const double xj = S[XS + j], yj = S[XS + m + j], zj = S[XS + 2 * m + j];
            const double hjx = S[ly.HV + j], hjy = S[ly.HV + m + j], hjz = S[ly.HV + 2 * m + j];
            double vj = S[V + j];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const double ps = psi_shape(kernel, S[ly.PH + r0 + a * i + a * (a + 1) / 2 + j]);
                const double dx = xi[a] - xj, dy = yi[a] - yj, dz = zi[a] - zj;
                vj = fma(ps, dx * hx[a] + dy * hy[a] + dz * hz[a], vj);
                vi[a] = fma(-ps, dx * hjx + dy * hjy + dz * hjz, vi[a]);
            }
            S[V + j] = vj;
        }
        // the pairs inside the block, row by row
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < a; ++c) {
                const int j = i + c;
                const double ps = psi_shape(kernel, S[ly.PH + pk(i + a, j)]);
                const double dx = xi[a] - S[XS + j], dy = yi[a] - S[XS + m + j], dz = zi[a] - S[XS + 2 * m + j];
                const double hjx = S[ly.HV + j], hjy = S[ly.HV + m + j], hjz = S[ly.HV + 2 * m + j];
                S[V + j] = fma(ps, dx * hx[a] + dy * hy[a] + dz * hz[a], S[V + j]);
                vi[a] = fma(-ps, dx * hjx + dy * hjy + dz * hjz, vi[a]);
            }
            S[V + i + a] += vi[a];
        }
    }
#pragma unroll 1
    for (; i < n; ++i) {
        double xi = S[XS + i], yi = S[XS + m + i], zi = S[XS + 2 * m + i];
        double hx = S[ly.HV + i], hy = S[ly.HV + m + i], hz = S[ly.HV + 2 * m + i];
        double vi = 0.0;
        int base = pk(i, 0);
#pragma unroll 1
        for (int j = 0; j < i; ++j) {
            double ps = psi_shape(kernel, S[ly.PH + base + j]);
            double dx = xi - S[XS + j], dy = yi - S[XS + m + j], dz = zi - S[XS + 2 * m + j];
            double hjx = S[ly.HV + j], hjy = S[ly.HV + m + j], hjz = S[ly.HV + 2 * m + j];
            S[V + j] = fma(ps, dx * hx + dy * hy + dz * hz, S[V + j]);
            vi = fma(-ps, dx * hjx + dy * hjy + dz * hjz, vi);
        }
        S[V + i] += vi;
    }
    const double cs = psi_scale(kernel, e2);
#pragma unroll 1
    for (int j = 0; j < n; ++j) S[V + j] *= cs;
    aug_solve0(S, ly, n, V, s);
}

template <int KERNEL>
__global__ void __launch_bounds__(128, 4) search_kernel(SearchArgs A) {
    const int lane_id = threadIdx.x & 31;
    const int64_t warp_global = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    Lane S{A.scratch + warp_global * 32 * (int64_t)A.lane_size + lane_id};
    int g = 0;
    Layout ly = make_layout(A.gi.npad[0], false);
    bool have = false;
    int64_t lr = 0, r = 0;
    int n = A.gi.n[0];
    Search st;
    Geo geo;
    geo.rs = 1.0;
    double tol_s = 0.0;
    bool learned = false;
    double vborder = 0.0;     // border entry of the Ritz vector in RV
    while (true) {
        if (!have) {
            unsigned long long t = atomicAdd(&A.counters[g], 1ull);
            int64_t cnt = A.gi.row_begin[g + 1] - A.gi.row_begin[g];
            if ((int64_t)t < cnt) {
                have = true;
                lr = (int64_t)t;
                r = A.gi.row_begin[g] + lr;
                geo = load_geometry(S, ly, n, A.idx, A.gi.ell_off[g], A.gi.npad[g], lr, A.X, A.NR, true);
                tol_s = A.tol * geo.rs;
                st.phase = PH_FIRST;
                st.evals = 0;
                st.status = RBFFD_STENCIL_OK;
                st.lo = -INFINITY;
                st.hi = INFINITY;
                st.dx_prev = INFINITY;
                st.f_prev = INFINITY;
                st.ulo = A.xlo;
                st.uhi = A.xhi;
                float gs = A.guess_rows ? A.guess_rows[r] : NAN;
                learned = isfinite(gs);
                st.x_next = clampd(learned ? learned_start(gs, n) : log(1.0 / geo.mean_d), A.xlo, A.xhi);
            }
        }
        if (__ballot_sync(0xffffffffu, have) == 0) {
            if (++g >= A.gi.ngroups) break;
            ly = make_layout(A.gi.npad[g], false);
            n = A.gi.n[g];
            continue;
        }
        if (have) {
            double dF, schur;
            // every evaluation starts its A^{-1} Lanczos run cold: a start from
            // the previous Ritz vector can stay on that eigenvalue's branch
            // when the two smallest eigenvalues cross, and then misjudge kappa
            const double eps_s = exp(st.x_next);
            const double acc_lo = A.acc_lo * A.kT * (1.0 + ACCEPT_MARGIN);
            const double acc_hi = A.acc_hi * A.kT * (1.0 - ACCEPT_MARGIN);
            double theta;
            const bool first_guess = learned && st.phase == PH_FIRST;
            bool early = false;
            double k = eval_kappa(S, ly, n, KERNEL, eps_s, false, &vborder, &theta, &schur,
                                  (uint64_t)A.row_node[r], acc_lo, first_guess ? acc_hi : 0.0, &early);
            // the slope is needed unless a learned guess is accepted now
            const bool accept_now = first_guess && (early || (k >= acc_lo && k <= acc_hi));
            dF = (isfinite(k) && !accept_now) ? kappa_slope(S, ly, n, KERNEL, eps_s, theta) : NAN;
            search_update(st, F_of(k, A.kT), dF, k, tol_s, A.max_evals, acc_lo, acc_hi, learned, n);
            if (st.phase == PH_DONE) {
                // the search stopped at its last evaluated point, whose
                // factorisation is still in scratch: the weights follow
                const int node = A.row_node[r];
                const int npad = A.gi.npad[g];
                const int64_t off = A.gi.ell_off[g];
                const bool valid = isfinite(st.k_ret) && schur > 0.0;
                if (valid) first_row_weights(S, ly, n, KERNEL, exp(st.x_ret), schur);
                const double inv_rs2 = 1.0 / (geo.rs * geo.rs);
#pragma unroll 1
                for (int j = 0; j < npad; ++j) {
                    double w = (valid && j < n) ? S[ly.Q0 + j] * inv_rs2 : 0.0;
                    A.w64[ell_elem(off, npad, lr, j)] = w;
                    A.w32[ell_elem(off, npad, lr, j)] = (float)w;
                }
                A.eps[node] = exp(st.x_ret) / geo.rs;
                A.kappa[node] = st.k_ret;
                A.evals[node] = st.evals;
                A.status[node] = valid ? st.status : RBFFD_STENCIL_SINGULAR;
                have = false;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// weights at a fixed eps per stencil
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128, 4) weights_kernel(WeightArgs A) {
    const int lane_id = threadIdx.x & 31;
    const int64_t warp_global = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    Lane S{A.scratch + warp_global * 32 * (int64_t)A.lane_size + lane_id};
    const int64_t R = A.gi.row_begin[A.gi.ngroups];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < R; r += stride) {
        const int g = group_of_row(A.gi, r);
        const int n = A.gi.n[g], npad = A.gi.npad[g];
        const int64_t lr = r - A.gi.row_begin[g], off = A.gi.ell_off[g];
        const Layout ly = make_layout(npad, true);
        Geo geo = load_geometry(S, ly, n, A.idx, off, npad, lr, A.X, A.NR, true);
        int node = A.row_node[r];
        double eps_s = A.eps_node[node] * geo.rs;
        assemble_phi(S, ly, n, A.kernel, eps_s, ly.L, ly.PH);
        bool ok = cholesky(S, ly, n) && isfinite(eps_s) && eps_s > 0.0;
        double s = 0.0;
        if (ok) {
            for (int i = 0; i < ly.m; ++i) S[ly.U + i] = i < n ? 1.0 : 0.0;
            chol_solve(S, ly, ly.U);
            for (int i = 0; i < n; ++i) s += S[ly.U + i];
            ok = s > 0.0 && isfinite(s);
        }
        if (!ok) {
            A.status[node] = RBFFD_STENCIL_SINGULAR;
            atomicAdd(A.nfail, 1);
            for (int j = 0; j < npad; ++j) {
                A.w64[ell_elem(off, npad, lr, j)] = 0.0;
                A.w32[ell_elem(off, npad, lr, j)] = 0.f;
            }
            continue;
        }
        first_row_weights(S, ly, n, A.kernel, eps_s, s);
        const int V = ly.Q0;
        double inv_rs2 = 1.0 / (geo.rs * geo.rs);
        for (int j = 0; j < npad; ++j) {
            double w = j < n ? S[V + j] * inv_rs2 : 0.0;
            A.w64[ell_elem(off, npad, lr, j)] = w;
            A.w32[ell_elem(off, npad, lr, j)] = (float)w;
        }
    }
}

struct LaunchShape {
    int threads, blocks;
};

LaunchShape launch_shape(const rbffd_build_opts& o, int64_t rows) {
    LaunchShape ls;
    ls.threads = o.block_threads > 0 ? o.block_threads : 128;
    // 4 x 128 threads: 16 resident warps per SM, which the kernels' launch
    // bounds (<= 128 registers per thread) allow; more warps in flight hide
    // more of the latency of the lanes' scratch loads
    int bps = o.blocks_per_sm > 0 ? o.blocks_per_sm : 4;
    int64_t want = (int64_t)sm_count() * bps;
    int64_t need = (rows + ls.threads - 1) / ls.threads;
    ls.blocks = (int)std::max<int64_t>(1, std::min(want, need));
    return ls;
}

}  // namespace

rbffd_status build_search(rbffd_op* op, const double* nodes, const double* normals,
                          const rbffd_build_opts& o, const float* guess_rows, cudaStream_t st) {
    const GroupInfo& gi = op->gi;
    LaunchShape ls = launch_shape(o, op->N);
    RBFFD_CHECK_ARG(ls.threads % 32 == 0 && ls.threads <= 128, "block_threads must be 32..128, x32");
    unsigned long long* ctr = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&ctr, RBFFD_MAX_GROUPS * sizeof(unsigned long long), st));
    RBFFD_CUDA_TRY(cudaMemsetAsync(ctr, 0, RBFFD_MAX_GROUPS * sizeof(unsigned long long), st));
    SearchArgs A;
    A.X = nodes;
    A.NR = normals;
    A.w64 = op->w64;
    A.w32 = op->w32;
    A.idx = op->idx;
    A.row_node = op->row_node;
    A.gi = gi;
    A.kernel = o.kernel;
    A.kT = o.kappa_target;
    A.tol = o.eps_tol;
    A.xlo = o.eps_lo > 0.0 ? log(o.eps_lo) : -INFINITY;
    A.xhi = o.eps_hi > 0.0 ? log(o.eps_hi) : INFINITY;
    A.acc_lo = o.accept_lo;
    A.acc_hi = o.accept_hi;
    A.max_evals = o.max_evals;
    A.guess_rows = guess_rows;
    A.counters = ctr;
    A.eps = op->eps;
    A.kappa = op->kappa;
    A.evals = op->evals;
    A.status = op->status;
    // Operators that do not fill the chip with a lane per stencil go to the team
    // kernel, unless the caller chose the lane kernel's launch shape.  One kernel
    // takes all groups, largest stencils first: a launch per group was slower
    // (1M nodes in four sizes, learned: 476 against 421 ms), because the last
    // stencils of a large group then run alone.
    int mmax = 0;
    for (int g = 0; g < gi.ngroups; ++g) mmax = std::max(mmax, gi.npad[g]);
    const bool shaped = o.block_threads > 0 || o.blocks_per_sm > 0;
    if (!shaped && team_lanes(mmax, op->N, guess_rows != nullptr) > 0) {
        rbffd_status s = team_search(A, mmax, op->N, st);
        if (s != RBFFD_OK) return s;
    } else {
        const Layout ly = make_layout(mmax, false);
        const int64_t lanes = (int64_t)ls.blocks * ls.threads;
        RBFFD_CUDA_TRY(pool_alloc(&A.scratch, (size_t)lanes * ly.size * sizeof(double), st));
        A.lane_size = ly.size;
        if (A.kernel == RBFFD_GAUSSIAN) search_kernel<RBFFD_GAUSSIAN><<<ls.blocks, ls.threads, 0, st>>>(A);
        else search_kernel<RBFFD_IMQ><<<ls.blocks, ls.threads, 0, st>>>(A);
        note_launch();
        RBFFD_CUDA_TRY(cudaGetLastError());
        RBFFD_CUDA_TRY(cudaFreeAsync(A.scratch, st));
    }
    RBFFD_CUDA_TRY(cudaFreeAsync(ctr, st));
    return RBFFD_OK;
}

rbffd_status build_weights(rbffd_op* op, const double* nodes, const double* normals,
                           const rbffd_build_opts& o, const double* eps_node, cudaStream_t st) {
    const GroupInfo& gi = op->gi;
    LaunchShape ls = launch_shape(o, op->N);
    RBFFD_CHECK_ARG(ls.threads % 32 == 0 && ls.threads <= 128, "block_threads must be 32..128, x32");
    int* nfail = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&nfail, sizeof(int), st));
    RBFFD_CUDA_TRY(cudaMemsetAsync(nfail, 0, sizeof(int), st));
    TeamWeightArgs B;
    memset(&B, 0, sizeof(B));
    WeightArgs& A = B.w;
    A.X = nodes;
    A.NR = normals;
    A.idx = op->idx;
    A.row_node = op->row_node;
    A.gi = gi;
    A.kernel = o.kernel;
    A.eps_node = eps_node;
    A.w64 = op->w64;
    A.w32 = op->w32;
    A.status = op->status;
    A.nfail = nfail;
    int mmax = 0;
    for (int g = 0; g < gi.ngroups; ++g) mmax = std::max(mmax, gi.npad[g]);
    const bool shaped = o.block_threads > 0 || o.blocks_per_sm > 0;
    if (!shaped && team_weight_lanes(mmax, op->N) > 0) {
        rbffd_status s = team_weights(B, 0, st);
        if (s != RBFFD_OK) return s;
    } else {
        const Layout ly = make_layout(mmax, true);
        const int64_t lanes = (int64_t)ls.blocks * ls.threads;
        RBFFD_CUDA_TRY(pool_alloc(&A.scratch, (size_t)lanes * ly.size * sizeof(double), st));
        A.lane_size = ly.size;
        weights_kernel<<<ls.blocks, ls.threads, 0, st>>>(A);
        note_launch();
        RBFFD_CUDA_TRY(cudaGetLastError());
        RBFFD_CUDA_TRY(cudaFreeAsync(A.scratch, st));
    }
    int hf = 0;
    RBFFD_CUDA_TRY(cudaMemcpyAsync(&hf, nfail, sizeof(int), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    RBFFD_CUDA_TRY(cudaFreeAsync(nfail, st));
    if (hf) {
        set_error("%d stencils have a local matrix that is not numerically positive definite", hf);
        return RBFFD_ESINGULAR;
    }
    return RBFFD_OK;
}

}  // namespace rbffd

// ---------------------------------------------------------------------------
// Allocation-free weights for caller-supplied stencils
// (rbffd_stencil_weights_noalloc).  The scratch lives in a fixed array in the
// library's device image instead of memory obtained at run time.
// ---------------------------------------------------------------------------
namespace rbffd {
namespace {

constexpr int64_t NOALLOC_SCRATCH_DOUBLES = (int64_t)4 << 20;   // 32 MiB of float64
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_SCRATCH_DOUBLES];
static __device__ int g_noalloc_fail;   // rows that failed in the current call

// Device address of the scratch array, looked up once per device.
constexpr int NOALLOC_MAX_DEVICES = 64;
double* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};
int* g_noalloc_fail_ptr[NOALLOC_MAX_DEVICES] = {};
std::mutex g_noalloc_mu;

}  // namespace
}  // namespace rbffd

extern "C" rbffd_status rbffd_stencil_weights_noalloc(const double* nodes, const double* normals, int64_t N,
                                                      const int32_t* stencils, int64_t rows, int n,
                                                      const double* eps, int kernel, double* weights,
                                                      void* stream) {
    using namespace rbffd;
    RBFFD_CHECK_ARG(nodes && normals && stencils && eps && weights, "NULL argument");
    RBFFD_CHECK_ARG(kernel == RBFFD_GAUSSIAN || kernel == RBFFD_IMQ, "kernel");
    RBFFD_CHECK_ARG(N >= 2 && rows >= 0, "N must be >= 2 and rows >= 0");
    if (n < 2 || n > RBFFD_MAX_N || n > N) {
        set_error("rbffd_stencil_weights_noalloc: stencil size %d outside [2, min(N, %d)]", n, RBFFD_MAX_N);
        return RBFFD_EINVAL;
    }
    if (rows == 0) return RBFFD_OK;
    int dev = 0;
    RBFFD_CUDA_TRY(cudaGetDevice(&dev));
    RBFFD_CHECK_ARG(dev >= 0 && dev < NOALLOC_MAX_DEVICES, "device ordinal");
    double* scratch;
    int* fail;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            // with this device current: the symbols' device addresses
            void* p = nullptr;
            void* f = nullptr;
            RBFFD_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
            RBFFD_CUDA_TRY(cudaGetSymbolAddress(&f, g_noalloc_fail));
            g_noalloc_fail_ptr[dev] = static_cast<int*>(f);
            g_noalloc_ptr[dev] = static_cast<double*>(p);
        }
        scratch = g_noalloc_ptr[dev];
        fail = g_noalloc_fail_ptr[dev];
    }
    cudaStream_t st = as_stream(stream);
    // the failure counter must start at zero; the scratch itself is written
    // before it is read in every row, so it is not cleared
    RBFFD_CUDA_TRY(cudaMemsetAsync(fail, 0, sizeof(int), st));
    TeamWeightArgs B;
    memset(&B, 0, sizeof(B));
    B.w.X = nodes;
    B.w.NR = normals;
    B.w.scratch = scratch;
    B.w.kernel = kernel;
    B.w.eps_node = eps;
    B.w.w64 = weights;
    B.w.nfail = fail;
    B.stencils = stencils;
    B.N = N;
    B.rows = rows;
    B.n = n;
    const rbffd_status s = team_weights(B, NOALLOC_SCRATCH_DOUBLES, st);
    if (s != RBFFD_OK) return s;
    int hfail = 0;
    RBFFD_CUDA_TRY(cudaMemcpyAsync(&hfail, fail, sizeof(int), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    if (hfail) {
        set_error("%d stencils have an out-of-range index or a local matrix that is not positive definite "
                  "(their weights are NaN)", hfail);
        return RBFFD_ESINGULAR;
    }
    return RBFFD_OK;
}

// ---------------------------------------------------------------------------
// Double-double build (rbffd_build_opts.precision = RBFFD_PREC_DD): the same
// search and weights with every step that the condition number amplifies --
// geometry, Phi, its Cholesky factor, the A^{-1} solves, the weights -- in
// double-double arithmetic (unit roundoff ~1e-32), for target condition
// numbers beyond float64 (Section 6 computes its kappa_T = 1e18 / 1e20
// weights in quad precision and then rounds them to float64, as this path
// does).  The A Lanczos run (lambda_max, well conditioned), the tridiagonal
// eigenvalues and the Hellmann-Feynman slope stay in float64 / float32.
// Plain loops: these builds are for the high-kappa studies, not for speed.
// ---------------------------------------------------------------------------
namespace rbffd {
namespace {

// lane-interleaved storage of double-double elements: element e of a lane
// occupies float64 slots 2e (hi) and 2e + 1 (lo) of that lane
struct LaneDD {
    double* p;
    __device__ __forceinline__ dd get(int e) const {
        return dd{p[(int64_t)(2 * e) * 32], p[(int64_t)(2 * e + 1) * 32]};
    }
    __device__ __forceinline__ void set(int e, dd v) const {
        p[(int64_t)(2 * e) * 32] = v.hi;
        p[(int64_t)(2 * e + 1) * 32] = v.lo;
    }
    __device__ __forceinline__ double hi(int e) const { return p[(int64_t)(2 * e) * 32]; }
};

struct LayoutDD {
    int m, P;
    int XS, NS, R2, L, PH, U, ID, V0, V1, V2, QB, RV, GV, HV;
    int size;   // double-double elements per lane
};

__host__ __device__ inline LayoutDD make_layout_dd(int m) {
    LayoutDD l;
    l.m = m;
    l.P = m * (m + 1) / 2;
    int o = 0;
    l.XS = o; o += 3 * m;
    l.NS = o; o += 3 * m;
    l.R2 = o; o += l.P;
    l.L = o; o += l.P;
    l.PH = o; o += l.P;
    l.U = o; o += m;
    l.ID = o; o += m;
    l.V0 = o; o += m;
    l.V1 = o; o += m;
    l.V2 = o; o += m;
    l.QB = o; o += LANCZOS_KMAX * m;
    l.RV = o; o += m;
    l.GV = o; o += 3 * m;
    l.HV = o; o += 3 * m;
    l.size = o;
    return l;
}

// centre-translated (exact differences), r_s-scaled coordinates, unit
// normals and pairwise squared distances, all in double-double
__device__ Geo geometry_dd(const LaneDD& S, const LayoutDD& ly, int n, const int32_t* __restrict__ idx,
                           int64_t off, int npad, int64_t lr, const double* __restrict__ X,
                           const double* __restrict__ NR) {
    const int m = ly.m;
    int c = idx[ell_elem(off, npad, lr, 0)];
    const double cx = X[3 * (int64_t)c], cy = X[3 * (int64_t)c + 1], cz = X[3 * (int64_t)c + 2];
    double rs2 = 0.0;
    for (int j = 0; j < n; ++j) {
        int k = idx[ell_elem(off, npad, lr, j)];
        dd d0 = two_sum(X[3 * (int64_t)k], -cx), d1 = two_sum(X[3 * (int64_t)k + 1], -cy),
           d2 = two_sum(X[3 * (int64_t)k + 2], -cz);
        S.set(ly.XS + j, d0);
        S.set(ly.XS + m + j, d1);
        S.set(ly.XS + 2 * m + j, d2);
        rs2 = fmax(rs2, d0.hi * d0.hi + d1.hi * d1.hi + d2.hi * d2.hi);
        double nx = NR[3 * (int64_t)k], ny = NR[3 * (int64_t)k + 1], nz = NR[3 * (int64_t)k + 2];
        double inv = rsqrt(nx * nx + ny * ny + nz * nz);
        S.set(ly.NS + j, dd_of(nx * inv));
        S.set(ly.NS + m + j, dd_of(ny * inv));
        S.set(ly.NS + 2 * m + j, dd_of(nz * inv));
    }
    Geo g;
    g.rs = sqrt(rs2);
    const double inv = 1.0 / g.rs;
    double sum = 0.0;
    for (int j = 0; j < n; ++j) {
        dd x = S.get(ly.XS + j) * inv, y = S.get(ly.XS + m + j) * inv, z = S.get(ly.XS + 2 * m + j) * inv;
        S.set(ly.XS + j, x);
        S.set(ly.XS + m + j, y);
        S.set(ly.XS + 2 * m + j, z);
        if (j > 0) sum += sqrt(x.hi * x.hi + y.hi * y.hi + z.hi * z.hi);
    }
    g.mean_d = sum / (double)(n - 1);
    for (int i = 0; i < n; ++i) {
        const dd xi = S.get(ly.XS + i), yi = S.get(ly.XS + m + i), zi = S.get(ly.XS + 2 * m + i);
        for (int j = 0; j < i; ++j) {
            dd dx = xi - S.get(ly.XS + j), dy = yi - S.get(ly.XS + m + j), dz = zi - S.get(ly.XS + 2 * m + j);
            S.set(ly.R2 + pk(i, j), dx * dx + dy * dy + dz * dz);
        }
        S.set(ly.R2 + pk(i, i), dd_of(0.0));
    }
    return g;
}

__device__ __forceinline__ dd phi_dd(int kernel, dd e2r2) {
    return kernel == RBFFD_GAUSSIAN ? dd_exp(-e2r2) : dd_of(1.0) / dd_sqrt(dd_of(1.0) + e2r2);
}
__device__ __forceinline__ dd psi_from_phi_dd(int kernel, dd e2, dd ph) {
    return kernel == RBFFD_GAUSSIAN ? -(e2 * ph * 2.0) : -(e2 * ph * ph * ph);
}

// Phi(eps_s) into L and PH (packed lower, identity on the padding)
__device__ void assemble_dd(const LaneDD& S, const LayoutDD& ly, int n, int kernel, double eps_s) {
    const dd e2 = two_prod(eps_s, eps_s);
    for (int i = 0; i < ly.m; ++i) {
        for (int j = 0; j < i; ++j) {
            dd v = i < n ? phi_dd(kernel, e2 * S.get(ly.R2 + pk(i, j))) : dd_of(0.0);
            S.set(ly.L + pk(i, j), v);
            S.set(ly.PH + pk(i, j), v);
        }
        S.set(ly.L + pk(i, i), dd_of(1.0));
        S.set(ly.PH + pk(i, i), dd_of(1.0));
    }
}

// in-place packed Cholesky, L_ij = (A_ij - sum_{k<j} L_ik L_jk) / L_jj;
// ID receives 1 / L_jj.  false when a pivot is not positive.
__device__ bool cholesky_dd(const LaneDD& S, const LayoutDD& ly) {
    const int m = ly.m;
    for (int j = 0; j < m; ++j) {
        dd d = S.get(ly.L + pk(j, j));
        for (int k = 0; k < j; ++k) {
            dd l = S.get(ly.L + pk(j, k));
            d = fms(d, l, l);
        }
        if (!(d.hi > 0.0)) return false;
        dd ljj = dd_sqrt(d);
        dd il = dd_of(1.0) / ljj;
        S.set(ly.L + pk(j, j), ljj);
        S.set(ly.ID + j, il);
        for (int i = j + 1; i < m; ++i) {
            dd s = S.get(ly.L + pk(i, j));
            for (int k = 0; k < j; ++k) s = fms(s, S.get(ly.L + pk(i, k)), S.get(ly.L + pk(j, k)));
            S.set(ly.L + pk(i, j), s * il);
        }
    }
    return true;
}

// V <- Phi^{-1} V
__device__ void chol_solve_dd(const LaneDD& S, const LayoutDD& ly, int V) {
    const int m = ly.m;
    for (int i = 0; i < m; ++i) {
        dd t = S.get(V + i);
        for (int k = 0; k < i; ++k) t = fms(t, S.get(ly.L + pk(i, k)), S.get(V + k));
        S.set(V + i, t * S.get(ly.ID + i));
    }
    for (int i = m - 1; i >= 0; --i) {
        dd t = S.get(V + i);
        for (int k = i + 1; k < m; ++k) t = fms(t, S.get(ly.L + pk(k, i)), S.get(V + k));
        S.set(V + i, t * S.get(ly.ID + i));
    }
}

// [c; d] = A^{-1} [f; g] with c in V (first n entries), d returned:
// c0 = Phi^{-1} f, d = (1^T c0 - g) / s, c = c0 - d u
__device__ dd aug_solve_dd(const LaneDD& S, const LayoutDD& ly, int n, int V, dd g, dd s) {
    chol_solve_dd(S, ly, V);
    dd sum = dd_of(0.0);
    for (int i = 0; i < n; ++i) sum = sum + S.get(V + i);
    dd d = (sum - g) / s;
    for (int i = 0; i < n; ++i) S.set(V + i, fms(S.get(V + i), d, S.get(ly.U + i)));
    return d;
}

// Lanczos on A^{-1} from the stencil's pseudo-random start (as the float64
// search does): returns the Ritz value of largest magnitude and leaves the
// Ritz vector (float64 values as hi parts) in RV with its border in *vb.
__device__ double lanczos_inv_dd(const LaneDD& S, const LayoutDD& ly, int n, dd s, uint64_t seed, double* vb) {
    const int m = ly.m;
    float al[LANCZOS_KMAX], b2[LANCZOS_KMAX];
    double alpha_d[LANCZOS_KMAX], beta_d[LANCZOS_KMAX];
    dd qbord[LANCZOS_KMAX + 1];
    dd nrm2 = dd_of(0.0);
    for (int i = 0; i < m; ++i) {
        dd v = dd_of(i < n ? unit_hash(seed * 131u + i) : 0.0);
        S.set(ly.QB + i, v);
        nrm2 = nrm2 + v * v;
    }
    dd qb = dd_of(unit_hash(seed * 131u + n));
    nrm2 = nrm2 + qb * qb;
    dd inrm = dd_of(1.0) / dd_sqrt(nrm2);
    for (int i = 0; i < n; ++i) S.set(ly.QB + i, S.get(ly.QB + i) * inrm);
    qbord[0] = qb * inrm;
    dd beta = dd_of(0.0);
    double prev = -1.0, ext = 0.0;
    int k = 0;
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        const int qj = ly.QB + j * m, qp = ly.QB + (j - 1) * m;
        for (int i = 0; i < m; ++i) S.set(ly.V0 + i, S.get(qj + i));
        dd wb = aug_solve_dd(S, ly, n, ly.V0, qbord[j], s);
        if (j > 0) {
            for (int i = 0; i < m; ++i) S.set(ly.V0 + i, fms(S.get(ly.V0 + i), beta, S.get(qp + i)));
            wb = fms(wb, beta, qbord[j - 1]);
        }
        dd a = qbord[j] * wb;
        for (int i = 0; i < m; ++i) a = a + S.get(qj + i) * S.get(ly.V0 + i);
        dd bn2 = dd_of(0.0);
        for (int i = 0; i < m; ++i) {
            dd v = fms(S.get(ly.V0 + i), a, S.get(qj + i));
            S.set(ly.V0 + i, v);
            bn2 = bn2 + v * v;
        }
        wb = fms(wb, a, qbord[j]);
        bn2 = bn2 + wb * wb;
        dd bn = dd_sqrt(bn2);
        alpha_d[j] = a.hi;
        beta_d[j] = bn.hi;
        k = j + 1;
        double G = 0.0;
        for (int i = 0; i <= j; ++i)
            G = fmax(G, fabs(alpha_d[i]) + (i < j ? beta_d[i] : 0.0) + (i > 0 ? beta_d[i - 1] : 0.0));
        const double ig = 1.0 / G;
        for (int i = 0; i <= j; ++i) {
            al[i] = (float)(alpha_d[i] * ig);
            float bb = (float)(beta_d[i] * ig);
            b2[i] = bb * bb;
        }
        ext = tri_extreme(al, b2, j + 1, G);
        if (j + 1 >= LANCZOS_KMIN && fabs(fabs(ext) - prev) <= LANCZOS_RTOL * fabs(ext)) break;
        if (bn.hi <= 1e-30 * fabs(a.hi) || j + 1 == LANCZOS_KMAX) break;
        prev = fabs(ext);
        beta = bn;
        const dd ib = dd_of(1.0) / bn;
        const int qn = ly.QB + (j + 1) * m;
        for (int i = 0; i < m; ++i) S.set(qn + i, S.get(ly.V0 + i) * ib);
        qbord[j + 1] = wb * ib;
    }
    double y[LANCZOS_KMAX];
    tri_eigvec(alpha_d, beta_d, k, ext, y);
    double vbr = 0.0, nv = 0.0;
    for (int j = 0; j < k; ++j) vbr = fma(y[j], qbord[j].hi, vbr);
    for (int i = 0; i < m; ++i) {
        double v = 0.0;
        for (int j = 0; j < k; ++j) v = fma(y[j], S.hi(ly.QB + j * m + i), v);
        S.set(ly.RV + i, dd_of(v));
        nv = fma(v, v, nv);
    }
    nv = fma(vbr, vbr, nv);
    const double inv = nv > 0.0 ? rsqrt(nv) : 0.0;
    for (int i = 0; i < m; ++i) S.set(ly.RV + i, dd_of(S.hi(ly.RV + i) * inv));
    *vb = vbr * inv;
    return ext;
}

// lambda_max of A by Lanczos on A (well conditioned: float64 products with
// the hi parts of Phi), from the near-constant start of the float64 search
__device__ double lanczos_max_dd(const LaneDD& S, const LayoutDD& ly, int n) {
    const int m = ly.m;
    float al[LANCZOS_KMAX], b2[LANCZOS_KMAX];
    double alpha_d[LANCZOS_KMAX], beta_d[LANCZOS_KMAX];
    // float64 vectors in the lo slots of V1 (q), V2 (q_prev) and GV (w)
    auto Q = [&](int r, int i) -> double& { return S.p[(int64_t)(2 * (r + i) + 1) * 32]; };
    const int q_ = ly.V1, qp = ly.V2, w = ly.GV;
    double nrm2 = 0.0;
    for (int i = 0; i < m; ++i) {
        double v = i < n ? 1.0 + 0.01 * (cos(1.7 * i + 0.3) + 0.1) : 0.0;
        Q(q_, i) = v;
        Q(qp, i) = 0.0;
        nrm2 += v * v;
    }
    double qb = 0.1, qpb = 0.0;
    nrm2 += qb * qb;
    double inrm = rsqrt(nrm2);
    for (int i = 0; i < n; ++i) Q(q_, i) *= inrm;
    qb *= inrm;
    double beta = 0.0, prev = -1.0, ext = 0.0;
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        // w = Phi q + qb 1 (rows < n), border 1^T q
        double sumq = 0.0;
        for (int i = 0; i < m; ++i) {
            double acc = 0.0;
            for (int k = 0; k < m; ++k) acc = fma(S.hi(ly.PH + (i >= k ? pk(i, k) : pk(k, i))), Q(q_, k), acc);
            Q(w, i) = i < n ? acc + qb : acc;
            if (i < n) sumq += Q(q_, i);
        }
        double wb = sumq;
        double a = 0.0;
        for (int i = 0; i < m; ++i) {
            Q(w, i) = fma(-beta, Q(qp, i), Q(w, i));
            a = fma(Q(q_, i), Q(w, i), a);
        }
        wb = fma(-beta, qpb, wb);
        a = fma(qb, wb, a);
        double bn = 0.0;
        for (int i = 0; i < m; ++i) {
            Q(w, i) = fma(-a, Q(q_, i), Q(w, i));
            bn = fma(Q(w, i), Q(w, i), bn);
        }
        wb = fma(-a, qb, wb);
        bn = sqrt(fma(wb, wb, bn));
        alpha_d[j] = a;
        beta_d[j] = bn;
        double G = 0.0;
        for (int i = 0; i <= j; ++i)
            G = fmax(G, fabs(alpha_d[i]) + (i < j ? beta_d[i] : 0.0) + (i > 0 ? beta_d[i - 1] : 0.0));
        const double ig = 1.0 / G;
        for (int i = 0; i <= j; ++i) {
            al[i] = (float)(alpha_d[i] * ig);
            float bb = (float)(beta_d[i] * ig);
            b2[i] = bb * bb;
        }
        ext = tri_max_abs(al, b2, j + 1, G);
        if (j + 1 >= 2 && fabs(ext - prev) <= LANCZOS_RTOL * ext) break;
        if (bn <= 1e-14 * fabs(a)) break;
        prev = ext;
        beta = bn;
        const double ib = 1.0 / bn;
        for (int i = 0; i < m; ++i) {
            Q(qp, i) = Q(q_, i);
            Q(q_, i) = Q(w, i) * ib;
        }
        qpb = qb;
        qb = wb * ib;
    }
    return ext;
}

// d(-ln lambda_min)/dx by Hellmann-Feynman (float64, hi parts), as the
// float64 search computes it
__device__ double kappa_slope_dd(const LaneDD& S, const LayoutDD& ly, int n, int kernel, double eps_s,
                                 double theta) {
    double acc = 0.0;
    for (int i = 1; i < n; ++i) {
        double row = 0.0;
        for (int j = 0; j < i; ++j) {
            double ph = S.hi(ly.PH + pk(i, j));
            double g = kernel == RBFFD_GAUSSIAN ? 2.0 * ph : ph * ph * ph;
            row = fma(g * S.hi(ly.R2 + pk(i, j)), S.hi(ly.RV + j), row);
        }
        acc = fma(S.hi(ly.RV + i), row, acc);
    }
    return -eps_s * theta * (-2.0 * eps_s * acc);
}

// kappa_2(A(eps_s)) in double-double; theta (the A^{-1} Ritz value) and the
// Schur complement s = 1^T Phi^{-1} 1 for the weights
__device__ double eval_kappa_dd(const LaneDD& S, const LayoutDD& ly, int n, int kernel, double eps_s,
                                double* theta_out, dd* schur, uint64_t seed) {
    *theta_out = NAN;
    *schur = dd_of(0.0);
    assemble_dd(S, ly, n, kernel, eps_s);
    if (!cholesky_dd(S, ly)) return INFINITY;
    for (int i = 0; i < ly.m; ++i) S.set(ly.U + i, dd_of(i < n ? 1.0 : 0.0));
    chol_solve_dd(S, ly, ly.U);
    dd s = dd_of(0.0);
    for (int i = 0; i < n; ++i) s = s + S.get(ly.U + i);
    if (!(s.hi > 0.0)) return INFINITY;
    *schur = s;
    double vb;
    double theta = lanczos_inv_dd(S, ly, n, s, seed, &vb);
    double lmax = lanczos_max_dd(S, ly, n);
    double k = lmax * fabs(theta);
    if (!isfinite(k)) return INFINITY;
    *theta_out = theta;
    return k;
}

// first row of L_P from the factorised Phi(eps_s) (the reassociated
// four-solve form of the float64 path), into V0 (first n entries)
__device__ void weights_dd(const LaneDD& S, const LayoutDD& ly, int n, int kernel, double eps_s, dd s) {
    const int m = ly.m, XS = ly.XS;
    const dd e2 = two_prod(eps_s, eps_s);
    const dd n0x = S.get(ly.NS), n0y = S.get(ly.NS + m), n0z = S.get(ly.NS + 2 * m);
    // rhs_d,j = psi(r_0j) [P_0 (x_0 - x_j)]_d in V0, V1, V2
    const int G[3] = {ly.V0, ly.V1, ly.V2};
    for (int d = 0; d < 3; ++d)
        for (int i = 0; i < m; ++i) S.set(G[d] + i, dd_of(0.0));
    for (int j = 1; j < n; ++j) {
        dd ps = psi_from_phi_dd(kernel, e2, S.get(ly.PH + pk(j, 0)));
        dd dx = -S.get(XS + j), dy = -S.get(XS + m + j), dz = -S.get(XS + 2 * m + j);
        dd nd = n0x * dx + n0y * dy + n0z * dz;
        S.set(G[0] + j, ps * fms(dx, n0x, nd));
        S.set(G[1] + j, ps * fms(dy, n0y, nd));
        S.set(G[2] + j, ps * fms(dz, n0z, nd));
    }
    for (int d = 0; d < 3; ++d) aug_solve_dd(S, ly, n, G[d], dd_of(0.0), s);
    // h_i = P_i g_i
    for (int i = 0; i < n; ++i) {
        dd gx = S.get(G[0] + i), gy = S.get(G[1] + i), gz = S.get(G[2] + i);
        dd nx = S.get(ly.NS + i), ny = S.get(ly.NS + m + i), nz = S.get(ly.NS + 2 * m + i);
        dd nd = nx * gx + ny * gy + nz * gz;
        S.set(ly.HV + i, fms(gx, nx, nd));
        S.set(ly.HV + m + i, fms(gy, ny, nd));
        S.set(ly.HV + 2 * m + i, fms(gz, nz, nd));
    }
    // v_j = sum_i psi_ij (x_i - x_j) . h_i
    for (int i = 0; i < m; ++i) S.set(ly.GV + i, dd_of(0.0));
    for (int i = 0; i < n; ++i) {
        const dd xi = S.get(XS + i), yi = S.get(XS + m + i), zi = S.get(XS + 2 * m + i);
        const dd hx = S.get(ly.HV + i), hy = S.get(ly.HV + m + i), hz = S.get(ly.HV + 2 * m + i);
        dd vi = S.get(ly.GV + i);
        for (int j = 0; j < i; ++j) {
            dd ps = psi_from_phi_dd(kernel, e2, S.get(ly.PH + pk(i, j)));
            dd dx = xi - S.get(XS + j), dy = yi - S.get(XS + m + j), dz = zi - S.get(XS + 2 * m + j);
            dd hjx = S.get(ly.HV + j), hjy = S.get(ly.HV + m + j), hjz = S.get(ly.HV + 2 * m + j);
            S.set(ly.GV + j, S.get(ly.GV + j) + ps * (dx * hx + dy * hy + dz * hz));
            vi = vi - ps * (dx * hjx + dy * hjy + dz * hjz);
        }
        S.set(ly.GV + i, vi);
    }
    for (int i = 0; i < m; ++i) S.set(ly.V0 + i, S.get(ly.GV + i));
    aug_solve_dd(S, ly, n, ly.V0, dd_of(0.0), s);
}

struct SearchDDArgs {
    SearchArgs a;                // inputs, outputs and search options as for the float64 kernel
    const double* eps_fixed;     // node order: weights at these eps (no search), or NULL
};

__global__ void __launch_bounds__(64) search_dd_kernel(SearchDDArgs D) {
    const SearchArgs& A = D.a;
    const int lane_id = threadIdx.x & 31;
    const int64_t warp_global = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    LaneDD S{A.scratch + warp_global * 32 * (int64_t)A.lane_size * 2 + lane_id};
    for (int g = 0; g < A.gi.ngroups; ++g) {
        const LayoutDD ly = make_layout_dd(A.gi.npad[g]);
        const int n = A.gi.n[g], npad = A.gi.npad[g];
        const int64_t off = A.gi.ell_off[g];
        const int64_t cnt = A.gi.row_begin[g + 1] - A.gi.row_begin[g];
        while (true) {
            const int64_t lr = (int64_t)atomicAdd(&A.counters[g], 1ull);
            if (lr >= cnt) break;
            const int64_t r = A.gi.row_begin[g] + lr;
            const int node = A.row_node[r];
            Geo geo = geometry_dd(S, ly, n, A.idx, off, npad, lr, A.X, A.NR);
            Search st;
            st.phase = PH_FIRST;
            st.evals = 0;
            st.status = RBFFD_STENCIL_OK;
            st.lo = -INFINITY;
            st.hi = INFINITY;
            st.dx_prev = INFINITY;
            st.f_prev = INFINITY;
            st.ulo = A.xlo;
            st.uhi = A.xhi;
            dd schur = dd_of(0.0);
            bool valid;
            double eps_w;   // the eps_s whose factorisation is in scratch
            if (D.eps_fixed) {
                // weights at the given eps: factorise, no kappa
                const double eps_s = D.eps_fixed[node] * geo.rs;
                eps_w = eps_s;
                assemble_dd(S, ly, n, A.kernel, eps_s);
                valid = isfinite(eps_s) && eps_s > 0.0 && cholesky_dd(S, ly);
                if (valid) {
                    for (int i = 0; i < ly.m; ++i) S.set(ly.U + i, dd_of(i < n ? 1.0 : 0.0));
                    chol_solve_dd(S, ly, ly.U);
                    for (int i = 0; i < n; ++i) schur = schur + S.get(ly.U + i);
                    valid = schur.hi > 0.0;
                }
                st.x_ret = log(eps_s);
                st.k_ret = NAN;
                st.status = RBFFD_STENCIL_OK;
            } else {
                const double tol_s = A.tol * geo.rs;
                const float gs = A.guess_rows ? A.guess_rows[r] : NAN;
                const bool learned = isfinite(gs);
                st.x_next = clampd(learned ? learned_start(gs, n) : log(1.0 / geo.mean_d), A.xlo, A.xhi);
                const double acc_lo = A.acc_lo * A.kT * (1.0 + ACCEPT_MARGIN);
                const double acc_hi = A.acc_hi * A.kT * (1.0 - ACCEPT_MARGIN);
                while (st.phase != PH_DONE) {
                    const double eps_s = exp(st.x_next);
                    double theta;
                    const double k = eval_kappa_dd(S, ly, n, A.kernel, eps_s, &theta, &schur, (uint64_t)node);
                    const bool accept_now = learned && st.phase == PH_FIRST && k >= acc_lo && k <= acc_hi;
                    const double dF = (isfinite(k) && !accept_now) ? kappa_slope_dd(S, ly, n, A.kernel, eps_s, theta)
                                                                   : NAN;
                    search_update(st, F_of(k, A.kT), dF, k, tol_s, A.max_evals, acc_lo, acc_hi, learned, n);
                }
                // the search stops at its last evaluated point, still factorised
                valid = isfinite(st.k_ret) && schur.hi > 0.0;
                eps_w = exp(st.x_ret);
            }
            if (valid) weights_dd(S, ly, n, A.kernel, eps_w, schur);
            const double inv_rs2 = 1.0 / (geo.rs * geo.rs);
            for (int j = 0; j < npad; ++j) {
                const double w = (valid && j < n) ? (S.get(ly.V0 + j) * inv_rs2).hi : 0.0;
                A.w64[ell_elem(off, npad, lr, j)] = w;
                A.w32[ell_elem(off, npad, lr, j)] = (float)w;
            }
            if (!D.eps_fixed) {
                A.eps[node] = exp(st.x_ret) / geo.rs;
                A.kappa[node] = st.k_ret;
                A.evals[node] = st.evals;
            }
            A.status[node] = valid ? st.status : RBFFD_STENCIL_SINGULAR;
        }
    }
}

}  // namespace

rbffd_status build_search_dd(rbffd_op* op, const double* nodes, const double* normals,
                             const rbffd_build_opts& o, const float* guess_rows, const double* eps_fixed,
                             cudaStream_t st) {
    const GroupInfo& gi = op->gi;
    int mmax = 0;
    for (int g = 0; g < gi.ngroups; ++g) mmax = std::max(mmax, gi.npad[g]);
    const LayoutDD ly = make_layout_dd(mmax);
    // one 64-thread block per SM: double-double scratch is large (~46 KB
    // per lane at n = 31, ~0.5 MB at n = 128)
    const int threads = 64;
    const int64_t need = (op->N + threads - 1) / threads;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sm_count(), need));
    const int64_t lanes = (int64_t)blocks * threads;
    double* scratch = nullptr;
    unsigned long long* ctr = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&scratch, (size_t)lanes * ly.size * 2 * sizeof(double), st));
    RBFFD_CUDA_TRY(pool_alloc(&ctr, RBFFD_MAX_GROUPS * sizeof(unsigned long long), st));
    RBFFD_CUDA_TRY(cudaMemsetAsync(ctr, 0, RBFFD_MAX_GROUPS * sizeof(unsigned long long), st));
    SearchDDArgs D;
    SearchArgs& A = D.a;
    A.X = nodes;
    A.NR = normals;
    A.w64 = op->w64;
    A.w32 = op->w32;
    A.idx = op->idx;
    A.row_node = op->row_node;
    A.gi = gi;
    A.scratch = scratch;
    A.lane_size = ly.size;
    A.kernel = o.kernel;
    A.kT = o.kappa_target;
    A.tol = o.eps_tol;
    A.xlo = o.eps_lo > 0.0 ? log(o.eps_lo) : -INFINITY;
    A.xhi = o.eps_hi > 0.0 ? log(o.eps_hi) : INFINITY;
    A.acc_lo = o.accept_lo;
    A.acc_hi = o.accept_hi;
    A.max_evals = o.max_evals;
    A.guess_rows = guess_rows;
    A.counters = ctr;
    A.eps = op->eps;
    A.kappa = op->kappa;
    A.evals = op->evals;
    A.status = op->status;
    D.eps_fixed = eps_fixed;
    search_dd_kernel<<<blocks, threads, 0, st>>>(D);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    RBFFD_CUDA_TRY(cudaFreeAsync(scratch, st));
    RBFFD_CUDA_TRY(cudaFreeAsync(ctr, st));
    return RBFFD_OK;
}

}  // namespace rbffd
