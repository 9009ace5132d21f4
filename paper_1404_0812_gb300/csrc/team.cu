// Operator build with a team of T lanes per stencil, for node sets that do not
// fill the chip with one lane per stencil (build.cu).
//
// What bounds it.  One float64 warp instruction occupies its scheduler's
// float64 unit for 64 clocks on this GPU whatever the number of active lanes,
// and its result is ready after the same 64 clocks (measured: a chain of
// dependent FMAs runs at the unit's full rate).  One warp per scheduler
// therefore saturates the unit, and what counts is how few float64 warp
// instructions a stencil needs and how evenly the stencils spread over the
// 608 schedulers.  A lane per stencil needs the fewest per stencil, but its
// shortest possible build is one stencil's whole instruction stream (n = 31,
// five evaluations: 175k instructions, 5.4 ms), and 2,562 stencils are 81
// warps.  T lanes of a warp share a stencil here, 32 / T stencils per warp:
// rows of the factorisation and of the solves go to the lanes, scalars are
// computed by every lane of the team.  Loads, shuffles and integer work hide
// under the float64 instructions.
//
// Same results.  Every element of the factor, of a solve and of a sum receives
// its float64 operations in the order of the lane-per-stencil kernels
// (increasing column in the factorisation and the forward solves, blocks of
// four rows from the last to the first in the backward solves, four partial
// sums by index mod 4 in the dot products), so an operator has the same bits
// whichever kernel built it.
//
// The warp runs its teams in step: loops have the same trip count for all, a
// team that is done repeats its last evaluation (the same values again), and
// its weights are formed when enough of the warp's teams are done.
#include "stencil.cuh"

#include <algorithm>
#include <cmath>

namespace rbffd {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// Regions of a team: global scratch (matrices, coordinates, normals, Lanczos
// basis) and shared memory (vectors).  Element e of team t lies at region + e * S + t, S = 32 / T
// teams per warp: lanes of a team on consecutive elements, or teams on the
// same element, make one contiguous access.
struct TeamLayout {
    int m, P;
    int R2, L, PH, XS, NS, QB, PF, size;          // global, doubles (PF: P floats)
    int W, U, ID, G, AL, BE, QBD, Y, A32, vsize;  // shared, doubles (G: three vectors; A32: two float arrays)
};

__host__ __device__ inline TeamLayout team_layout(int m, bool search) {
    TeamLayout l;
    l.m = m;
    l.P = m * (m + 1) / 2;
    int o = 0;
    l.R2 = o; o += search ? l.P : 0;   // the weights alone form Phi in place
    l.L = o; o += l.P;
    l.PH = o; o += l.P;
    l.XS = o; o += 3 * m;
    l.NS = o; o += 3 * m;
    l.QB = o; o += search ? LANCZOS_KMAX * m : 0;
    l.PF = o; o += search ? (l.P + 1) / 2 : 0;
    l.size = o;
    o = 0;
    l.W = o; o += m;
    l.U = o; o += m;
    l.ID = o; o += m;
    l.G = o; o += 3 * m;
    l.AL = o; o += search ? LANCZOS_KMAX : 0;
    l.BE = o; o += search ? LANCZOS_KMAX : 0;
    l.QBD = o; o += search ? LANCZOS_KMAX + 1 : 0;
    l.Y = o; o += search ? LANCZOS_KMAX : 0;
    l.A32 = o; o += search ? LANCZOS_KMAX : 0;
    l.vsize = o;
    return l;
}

template <int TL>
struct Team {
    static constexpr int T = TL, S = 32 / T;
    double* g;   // the team's element 0 of the warp's global scratch
    double* v;   // the same in shared memory
    int l, t;    // lane of the team, team of the warp
    __device__ __forceinline__ double& G(int e) const { return g[e * S]; }
    __device__ __forceinline__ double& V(int e) const { return v[e * S]; }
    // float32 views of a global / shared region
    __device__ __forceinline__ float& GF(int region, int e) const {
        return (reinterpret_cast<float*>(g - t + region * S) + t)[e * S];
    }
    __device__ __forceinline__ float& VF(int region, int e) const {
        return (reinterpret_cast<float*>(v - t + region * S) + t)[e * S];
    }
    // value of the team's lane k
    template <typename X>
    __device__ __forceinline__ X from(X x, int k) const {
        return __shfl_sync(FULL, x, k * S + t);
    }
    __device__ __forceinline__ double team_max(double x) const {
#pragma unroll
        for (int o = S; o < 32; o <<= 1) x = fmax(x, __shfl_xor_sync(FULL, x, o));
        return x;
    }
    // the four partial sums (index mod 4) of lanes 0..3, combined
    template <typename X>
    __device__ __forceinline__ X sum4(X x) const {
        const X a = from(x, 0), b = from(x, 1), c = from(x, 2), d = from(x, 3);
        return (a + b) + (c + d);
    }
};

// ---------------------------------------------------------------------------
// geometry
// ---------------------------------------------------------------------------

// centre-translated, r_s-scaled coordinates, unit normals and pairwise
// squared distances of the teams with `on`; node(j) gives the stencil's j-th
// node.  The mean distance is summed in index order.
template <typename Tm, typename Node>
__device__ Geo team_geometry(const Tm& C, const TeamLayout& ly, int n, bool on, bool want_mean, Node node,
                             const double* __restrict__ X, const double* __restrict__ NR) {
    constexpr int T = Tm::T;
    const int m = ly.m, XV = ly.G;   // the coordinates stay in shared memory while the pairs are formed
    double rs2 = 0.0;
    if (on) {
        const int c = node(0);
        const double cx = X[3 * (int64_t)c], cy = X[3 * (int64_t)c + 1], cz = X[3 * (int64_t)c + 2];
#pragma unroll 1
        for (int j = C.l; j < n; j += T) {
            const int k = node(j);
            const double dx = X[3 * (int64_t)k] - cx, dy = X[3 * (int64_t)k + 1] - cy,
                         dz = X[3 * (int64_t)k + 2] - cz;
            C.V(XV + j) = dx;
            C.V(XV + m + j) = dy;
            C.V(XV + 2 * m + j) = dz;
            rs2 = fmax(rs2, dx * dx + dy * dy + dz * dz);
            const double nx = NR[3 * (int64_t)k], ny = NR[3 * (int64_t)k + 1], nz = NR[3 * (int64_t)k + 2];
            const double inv = rsqrt(nx * nx + ny * ny + nz * nz);
            C.G(ly.NS + j) = nx * inv;
            C.G(ly.NS + m + j) = ny * inv;
            C.G(ly.NS + 2 * m + j) = nz * inv;
        }
    }
    rs2 = C.team_max(rs2);
    Geo g;
    g.rs = sqrt(rs2);
    g.mean_d = 0.0;
    const double inv = 1.0 / g.rs;
    if (on)
#pragma unroll 1
        for (int j = C.l; j < n; j += T) {
            const double x = C.V(XV + j) * inv, y = C.V(XV + m + j) * inv, z = C.V(XV + 2 * m + j) * inv;
            C.V(XV + j) = x;
            C.V(XV + m + j) = y;
            C.V(XV + 2 * m + j) = z;
            C.G(ly.XS + j) = x;
            C.G(ly.XS + m + j) = y;
            C.G(ly.XS + 2 * m + j) = z;
            if (want_mean) C.V(ly.W + j) = sqrt(x * x + y * y + z * z);
        }
    __syncwarp();
    if (want_mean) {
        double sum = 0.0;
#pragma unroll 1
        for (int j = 1; j < n; ++j) sum += C.V(ly.W + j);
        g.mean_d = sum / (double)(n - 1);
    }
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const double xi = C.V(XV + i), yi = C.V(XV + m + i), zi = C.V(XV + 2 * m + i);
        const int base = ly.R2 + pk(i, 0);
#pragma unroll 1
        for (int j = C.l; j <= i; j += T) {
            const double dx = xi - C.V(XV + j), dy = yi - C.V(XV + m + j), dz = zi - C.V(XV + 2 * m + j);
            if (on) C.G(base + j) = dx * dx + dy * dy + dz * dz;   // 0 on the diagonal
        }
    }
    __syncwarp();
    return g;
}

// Phi(eps) into the factor and PH (and float32 into PF), identity on the
// padding.  The packed elements go to the lanes one after the other, whatever
// their row.
template <typename Tm>
__device__ void team_assemble(const Tm& C, const TeamLayout& ly, int n, int kernel, double eps_s, bool f32) {
    constexpr int T = Tm::T;
    const double e2 = eps_s * eps_s;
    const int real = pk(n, 0);
#pragma unroll 2
    for (int e = C.l; e < real; e += T) {
        const double v = phi_of(kernel, e2, C.G(ly.R2 + e));
        C.G(ly.L + e) = v;
        C.G(ly.PH + e) = v;
        if (f32) C.GF(ly.PF, e) = (float)v;
    }
#pragma unroll 1
    for (int e = real + C.l; e < ly.P; e += T) {
        C.G(ly.L + e) = 0.0;
        C.G(ly.PH + e) = 0.0;
        if (f32) C.GF(ly.PF, e) = 0.f;
    }
    __syncwarp();
#pragma unroll 1
    for (int i = C.l; i < ly.m; i += T) {
        const int e = pk(i, i);
        C.G(ly.L + e) = 1.0;
        C.G(ly.PH + e) = 1.0;
        if (f32) C.GF(ly.PF, e) = 1.f;
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// factorisation and solves
// ---------------------------------------------------------------------------

// acc[q][b] -= sum_{k < jb} L(row q, k) L(jb + b, k) for CH rows of a lane; the
// loads of the next four columns are issued before the FMAs of these four
// (16 CH FMAs of 64 clocks each hide them)
template <int CH, typename Tm>
__device__ __forceinline__ void team_accumulate(const Tm& C, int L, const int (&row)[CH], int jb,
                                                double (&acc)[CH][4]) {
    const int c0 = L + pk(jb, 0), c1 = L + pk(jb + 1, 0), c2 = L + pk(jb + 2, 0), c3 = L + pk(jb + 3, 0);
    constexpr int UN = CH > 2 ? 2 : 4;   // columns in flight
    double x[CH][UN], y[4][UN];
    auto load = [&](int k) {
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            y[0][u] = C.G(c0 + k + u);
            y[1][u] = C.G(c1 + k + u);
            y[2][u] = C.G(c2 + k + u);
            y[3][u] = C.G(c3 + k + u);
#pragma unroll
            for (int q = 0; q < CH; ++q) x[q][u] = C.G(row[q] + k + u);
        }
    };
    if (jb > 0) load(0);
    for (int k = 0; k < jb; k += UN) {
        double xc[CH][UN], yc[4][UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
#pragma unroll
            for (int b = 0; b < 4; ++b) yc[b][u] = y[b][u];
#pragma unroll
            for (int q = 0; q < CH; ++q) xc[q][u] = x[q][u];
        }
        if (k + UN < jb) load(k + UN);
#pragma unroll
        for (int u = 0; u < UN; ++u)
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[q][b] = fma(-xc[q][u], yc[b][u], acc[q][b]);
    }
}

// rows r0 + l + T q (q < CH) of column block jb, below its first chunk
template <int CH, typename Tm>
__device__ __forceinline__ void team_chol_rows(const Tm& C, const TeamLayout& ly, int jb, int r0,
                                               const double (&lc)[4][4], const double (&il)[4]) {
    constexpr int T = Tm::T;
    int row[CH];
    double acc[CH][4];
#pragma unroll
    for (int q = 0; q < CH; ++q) {
        const int r = min(r0 + C.l + T * q, ly.m - 1);
        row[q] = ly.L + pk(r, 0);
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[q][b] = C.G(row[q] + jb + b);
    }
    team_accumulate<CH>(C, ly.L, row, jb, acc);
    __syncwarp();   // lanes clamped to the last row have read it before its owner writes
#pragma unroll
    for (int q = 0; q < CH; ++q) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double v = acc[q][b];
#pragma unroll
            for (int c = 0; c < b; ++c) v = fma(-acc[q][c], lc[b][c], v);
            acc[q][b] = v * il[b];
        }
        if (r0 + C.l + T * q < ly.m) {
#pragma unroll
            for (int b = 0; b < 4; ++b) C.G(row[q] + jb + b) = acc[q][b];
        }
    }
}

// In-place packed Cholesky Phi = L L^T by blocks of four columns, a row per
// lane (left-looking); ID receives 1 / L_ii.  False when a pivot of the team
// is not positive.
template <typename Tm>
__device__ __noinline__ bool team_cholesky(const Tm C, int m, bool search) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, search);
    bool ok = true;
    for (int jb = 0; jb < m; jb += 4) {
        // the chunk that holds the diagonal block: lanes 0..3 its rows
        const int r = jb + C.l, rr = min(r, m - 1);
        const int row[1] = {ly.L + pk(rr, 0)};
        double acc[1][4], il[4], lc[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[0][b] = jb + b <= rr ? C.G(row[0] + jb + b) : 0.0;
        team_accumulate<1>(C, ly.L, row, jb, acc);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double d = C.from(acc[0][b], b);
            if (!(d > 0.0)) {
                ok = false;
                d = 1.0;
            }
            const double lb = sqrt(d);
            il[b] = 1.0 / lb;
            acc[0][b] = C.l == b ? lb : acc[0][b] * il[b];
#pragma unroll
            for (int c = b + 1; c < 4; ++c) {
                lc[c][b] = C.from(acc[0][b], c);
                acc[0][c] = fma(-acc[0][b], lc[c][b], acc[0][c]);
            }
        }
        if (r < m) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (jb + b <= r) C.G(row[0] + jb + b) = acc[0][b];
        }
        if (C.l < 4) C.V(ly.ID + jb + C.l) = C.l == 0 ? il[0] : C.l == 1 ? il[1] : C.l == 2 ? il[2] : il[3];
        int r0 = jb + T;
        for (; r0 + 2 * T < m; r0 += 3 * T) team_chol_rows<3>(C, ly, jb, r0, lc, il);
        if (r0 + T < m) team_chol_rows<2>(C, ly, jb, r0, lc, il);
        else if (r0 < m) team_chol_rows<1>(C, ly, jb, r0, lc, il);
        __syncwarp();
    }
    return ok;
}

// x_d <- Phi^{-1} x_d for NR right-hand sides (shared regions R0, R0 + RS,
// ...).  Forward: blocks of T rows, a row per lane, columns in increasing
// order.  Backward: blocks of four rows solved by every lane, then the rows
// above updated, a row per lane.
template <int NR, typename Tm>
__device__ __noinline__ void team_solve(const Tm C, int m, bool search, int R0, int RS) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, search);
    const int L = ly.L;
    constexpr int UN = 8;   // columns whose loads are in flight
    for (int ib = 0; ib < m; ib += T) {
        const int r = ib + C.l, rr = min(r, m - 1);
        const int base = L + pk(rr, 0);
        double t[NR], a[UN], lr[T];
#pragma unroll
        for (int d = 0; d < NR; ++d) t[d] = C.V(R0 + d * RS + rr);
#pragma unroll
        for (int u = 0; u < UN; ++u) a[u] = u < ib ? C.G(base + u) : 0.0;
#pragma unroll
        for (int c = 0; c < T; ++c) lr[c] = c < C.l && ib + c < m ? C.G(base + ib + c) : 0.0;
        for (int k = 0; k < ib; k += UN) {
            double ac[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) ac[u] = a[u];
#pragma unroll
            for (int u = 0; u < UN; ++u) a[u] = k + UN + u < ib ? C.G(base + k + UN + u) : 0.0;
#pragma unroll
            for (int h = 0; h < UN; h += 4)
                if (k + h < ib) {   // ib is a multiple of four
#pragma unroll
                    for (int u = h; u < h + 4; ++u)
#pragma unroll
                        for (int d = 0; d < NR; ++d) t[d] = fma(-ac[u], C.V(R0 + d * RS + k + u), t[d]);
                }
        }
        const double id = C.V(ly.ID + rr);
#pragma unroll
        for (int c = 0; c < T; ++c)
            if (ib + c < m) {
#pragma unroll
                for (int d = 0; d < NR; ++d) {
                    const double y = C.from(t[d] * id, c);
                    t[d] = C.l == c ? y : fma(-lr[c], y, t[d]);
                }
            }
        __syncwarp();
        if (r < m) {
#pragma unroll
            for (int d = 0; d < NR; ++d) C.V(R0 + d * RS + r) = t[d];
        }
        __syncwarp();
    }
    for (int kb = m - 4; kb >= 0; kb -= 4) {
        const int r0 = L + pk(kb, 0), r1 = L + pk(kb + 1, 0), r2 = L + pk(kb + 2, 0), r3 = L + pk(kb + 3, 0);
        // the first updates' factor entries go out before the block's chain
        double a[4];
        int i = C.l;
        const int i0 = min(i, kb);   // a valid element also where the lane has no row
        a[0] = C.G(r0 + i0);
        a[1] = C.G(r1 + i0);
        a[2] = C.G(r2 + i0);
        a[3] = C.G(r3 + i0);
        const double d10 = C.G(r1 + kb), d20 = C.G(r2 + kb), d21 = C.G(r2 + kb + 1), d30 = C.G(r3 + kb),
                     d31 = C.G(r3 + kb + 1), d32 = C.G(r3 + kb + 2);
        double t[4][NR];
#pragma unroll
        for (int d = 0; d < NR; ++d) {
            const int R = R0 + d * RS + kb;
            t[3][d] = C.V(R + 3) * C.V(ly.ID + kb + 3);
            t[2][d] = fma(-d32, t[3][d], C.V(R + 2)) * C.V(ly.ID + kb + 2);
            t[1][d] = fma(-d31, t[3][d], fma(-d21, t[2][d], C.V(R + 1))) * C.V(ly.ID + kb + 1);
            t[0][d] = fma(-d30, t[3][d], fma(-d20, t[2][d], fma(-d10, t[1][d], C.V(R)))) * C.V(ly.ID + kb);
        }
        __syncwarp();
        if (C.l < 4) {
#pragma unroll
            for (int d = 0; d < NR; ++d)
                C.V(R0 + d * RS + kb + C.l) = C.l == 0 ? t[0][d] : C.l == 1 ? t[1][d] : C.l == 2 ? t[2][d] : t[3][d];
        }
        while (i - C.l < kb) {   // uniform over the warp
            const int in = min(i + T, kb);
            const double b0 = C.G(r0 + in), b1 = C.G(r1 + in), b2 = C.G(r2 + in), b3 = C.G(r3 + in);
            if (i < kb) {
#pragma unroll
                for (int d = 0; d < NR; ++d) {
                    double x = C.V(R0 + d * RS + i);
                    x = fma(-a[0], t[0][d], x);
                    x = fma(-a[1], t[1][d], x);
                    x = fma(-a[2], t[2][d], x);
                    x = fma(-a[3], t[3][d], x);
                    C.V(R0 + d * RS + i) = x;
                }
            }
            a[0] = b0;
            a[1] = b1;
            a[2] = b2;
            a[3] = b3;
            i += T;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// condition number
// ---------------------------------------------------------------------------

// Ritz value of largest magnitude (signed) of the k x k tridiagonal in AL, BE
// (float64): the lane-per-stencil kernel's float32 bisections, LV levels per
// round: half of the team's lanes bisect for the top eigenvalue, half for the
// bottom one, each lane testing one midpoint of the next LV levels, and the
// team then follows the branches that one lane would take.  (Several midpoints
// per lane and more levels per round were slower: the divisions of one lane's
// midpoints do not overlap.)
template <typename Tm>
__device__ __noinline__ double team_tri_extreme(const Tm C, int AL, int BE, int A32, int k) {
    constexpr int T = Tm::T, S = Tm::S;
    constexpr int LV = T >= 32 ? 4 : T >= 16 ? 3 : T >= 8 ? 2 : 1, HALF = T / 2, LEVELS = 26;
    // scale (Gershgorin bound)
    double G = 0.0;
#pragma unroll 1
    for (int i = C.l; i < k; i += T) {
        const double r = fabs(C.V(AL + i)) + (i < k - 1 ? C.V(BE + i) : 0.0) + (i > 0 ? C.V(BE + i - 1) : 0.0);
        G = fmax(G, r);
    }
    G = C.team_max(G);
    const double ig = 1.0 / G;
#pragma unroll 1
    for (int i = C.l; i < k; i += T) {
        C.VF(A32, i) = (float)(C.V(AL + i) * ig);
        const float bb = (float)(C.V(BE + i) * ig);
        C.VF(A32, LANCZOS_KMAX + i) = bb * bb;
    }
    __syncwarp();
    const bool top = C.l < HALF;
    const int node = (top ? C.l : C.l - HALF) + 1;   // heap index of this lane's midpoint, 1 = the next
    const int depth = 31 - __clz(node);
    float lo = -1.f, hi = 1.f;
#pragma unroll 1
    for (int done = 0; done < LEVELS; done += LV) {
        const int lv = min(LV, LEVELS - done);
        // this lane's midpoint: the path of its heap index from the root
        float a = lo, b = hi, x = 0.5f * (a + b);
#pragma unroll
        for (int d = 1; d <= LV; ++d)
            if (d <= depth) {
                if ((node >> (depth - d)) & 1) a = x; else b = x;
                x = 0.5f * (a + b);
            }
        float dd = C.VF(A32, 0) - x;
        int cnt = dd < 0.f ? 1 : 0;
#pragma unroll 1
        for (int i = 1; i < k; ++i) {
            if (dd == 0.f) dd = -1e-30f;
            dd = (C.VF(A32, i) - x) - C.VF(A32, LANCZOS_KMAX + i - 1) / dd;
            if (dd < 0.f) ++cnt;
        }
        // up: the eigenvalue lies above this midpoint (top: fewer than k below; bottom: none below)
        const unsigned votes = __ballot_sync(FULL, top ? cnt < k : cnt < 1);
        int h = 1;
#pragma unroll 1
        for (int d = 0; d < lv; ++d) {
            const bool up = (votes >> (((top ? 0 : HALF) + h - 1) * S + C.t)) & 1u;
            const float c = 0.5f * (lo + hi);
            if (up) lo = c; else hi = c;
            h = 2 * h + (up ? 1 : 0);
        }
    }
    const float v = 0.5f * (lo + hi);
    const float vt = C.from(v, 0), vb = C.from(v, HALF);
    __syncwarp();
    return G * (double)(fabsf(vt) >= fabsf(vb) ? vt : vb);
}

// max|lambda(A)| by Lanczos in float32 (lanczos_max_f32 of build.cu); the
// vectors are floats of region G.  A team that is done repeats its steps
// without effect until the warp is.
template <typename Tm>
__device__ __noinline__ double team_lanczos_max(const Tm C, int m, int n, double rtol) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, true);
    const int FV = ly.G;
    int qp = 0, q_ = m, w = 2 * m;
    for (int i = C.l; i < m; i += T) {
        C.VF(FV, q_ + i) = i < n ? 1.0f + 0.01f * (__cosf(1.7f * (float)i + 0.3f) + 0.1f) : 0.f;
        C.VF(FV, qp + i) = 0.f;
    }
    __syncwarp();
    float nrm2 = 0.f;
    for (int i = 0; i < m; ++i) nrm2 = fmaf(C.VF(FV, q_ + i), C.VF(FV, q_ + i), nrm2);
    float qb = 0.1f, qpb = 0.f;
    nrm2 = fmaf(qb, qb, nrm2);
    const float inrm = rsqrtf(nrm2);
    __syncwarp();
    for (int i = C.l; i < n; i += T) C.VF(FV, q_ + i) *= inrm;
    qb *= inrm;
    __syncwarp();
    float beta = 0.f;
    double prev = -1.0, ext = 0.0;
    bool done = false;
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        // Phi q, four rows per lane at a time, columns in increasing order
        for (int i0 = C.l; i0 - C.l < m; i0 += 4 * T) {
            int row[4], e[4];   // e: element (max(row, k), min(row, k)) of the packed triangle
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                row[q] = min(i0 + T * q, m - 1);
                e[q] = pk(row[q], 0);
            }
            for (int k = 0; k < m; k += 4) {
                float f[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        f[u][q] = C.GF(ly.PF, e[q]);
                        e[q] += k + u < row[q] ? 1 : k + u + 1;
                    }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float x = C.VF(FV, q_ + k + u);
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q] = fmaf(f[u][q], x, acc[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + T * q < m) C.VF(FV, w + i0 + T * q) = acc[q];
        }
        float sum = 0.f;
        for (int i = 0; i < n; ++i) sum += C.VF(FV, q_ + i);
        for (int i = C.l; i < m; i += T) {
            float v = C.VF(FV, w + i);
            if (i < n) v += qb;
            C.VF(FV, w + i) = fmaf(-beta, C.VF(FV, qp + i), v);
        }
        float wb = fmaf(-beta, qpb, sum);
        __syncwarp();
        float ap = 0.f;
        for (int i = C.l & 3; i < m; i += 4) ap = fmaf(C.VF(FV, q_ + i), C.VF(FV, w + i), ap);
        const float a = fmaf(qb, wb, C.sum4(ap));
        __syncwarp();
        for (int i = C.l; i < m; i += T) C.VF(FV, w + i) = fmaf(-a, C.VF(FV, q_ + i), C.VF(FV, w + i));
        __syncwarp();
        float bp = 0.f;
        for (int i = C.l & 3; i < m; i += 4) bp = fmaf(C.VF(FV, w + i), C.VF(FV, w + i), bp);
        wb = fmaf(-a, qb, wb);
        const float bn = sqrtf(fmaf(wb, wb, C.sum4(bp)));
        if (C.l == 0) {
            C.V(ly.AL + j) = a;
            C.V(ly.BE + j) = bn;
        }
        __syncwarp();
        const double e = team_tri_extreme(C, ly.AL, ly.BE, ly.A32, j + 1);
        if (!done) {
            ext = fabs(e);
            if (j + 1 >= 2 && fabs(ext - prev) <= rtol * ext) done = true;
            else if (bn <= 1e-6f * fabsf(a)) done = true;
            prev = ext;
        }
        if (__all_sync(FULL, done)) break;
        beta = bn;
        const float ib = 1.f / bn;
        const int s = qp;
        qp = q_;
        q_ = w;
        w = s;
        qpb = qb;
        for (int i = C.l; i < n; i += T) C.VF(FV, q_ + i) *= ib;
        qb = wb * ib;
        __syncwarp();
    }
    __syncwarp();
    return ext;
}

// start vector of the A^{-1} run in region q (border returned)
template <typename Tm>
__device__ double team_lanczos_start(const Tm& C, const TeamLayout& ly, int n, int q, uint64_t seed) {
    constexpr int T = Tm::T;
    const int m = ly.m;
#pragma unroll 1
    for (int i = C.l; i < m; i += T) C.V(q + i) = i < n ? unit_hash(seed * 131u + i) : 0.0;
    __syncwarp();
    double nrm2 = 0.0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        const double v = C.V(q + i);
        nrm2 += v * v;
    }
    double qb = unit_hash(seed * 131u + n);
    nrm2 += qb * qb;
    const double inrm = rsqrt(nrm2);
    __syncwarp();
#pragma unroll 1
    for (int i = C.l; i < n; i += T) C.V(q + i) *= inrm;
    __syncwarp();
    return qb * inrm;
}

// Ritz vector of the k-step run's Ritz value ext: unit, in region RV
template <typename Tm>
__device__ __noinline__ void team_ritz_vector(const Tm C, int m, int k, double ext) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, true);
    const int RV = ly.G + 2 * m;
    {
        double al[LANCZOS_KMAX], be[LANCZOS_KMAX], y[LANCZOS_KMAX];
#pragma unroll 1
        for (int i = 0; i < k; ++i) {
            al[i] = C.V(ly.AL + i);
            be[i] = C.V(ly.BE + i);
        }
        tri_eigvec(al, be, k, ext, y);
        __syncwarp();
        if (C.l == 0)
#pragma unroll 1
            for (int i = 0; i < k; ++i) C.V(ly.Y + i) = y[i];
    }
    __syncwarp();
    double vbr = 0.0;
#pragma unroll 1
    for (int j = 0; j < k; ++j) vbr = fma(C.V(ly.Y + j), C.V(ly.QBD + j), vbr);
#pragma unroll 1
    for (int i = C.l; i < m; i += T) {
        double v = 0.0;
#pragma unroll 1
        for (int j = 0; j < k; ++j) v = fma(C.V(ly.Y + j), C.G(ly.QB + j * m + i), v);
        C.V(RV + i) = v;
    }
    __syncwarp();
    double nv = 0.0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        const double v = C.V(RV + i);
        nv = fma(v, v, nv);
    }
    nv = fma(vbr, vbr, nv);
    const double inv = nv > 0.0 ? rsqrt(nv) : 0.0;
    __syncwarp();
#pragma unroll 1
    for (int i = C.l; i < m; i += T) C.V(RV + i) *= inv;
    __syncwarp();
}

// Lanczos with A^{-1} (lanczos_inv_ritz of build.cu, cold start): returns the
// signed Ritz value of largest magnitude, the unit Ritz vector in region RV
// (G + 2m).  The first product Phi^{-1} q_0 is in W.  The extreme eigenvalue
// is evaluated only at the steps whose tests use it.
template <typename Tm>
__device__ __noinline__ double team_lanczos_inv(const Tm C, int m, int n, double s, double rtol, double qb0,
                                                bool active, bool try_early, double lmax, double acc_lo,
                                                double acc_hi, bool* early) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, true);
    const int W = ly.W;
    int cur = ly.G, old = ly.G + m;
    for (int i = C.l; i < m; i += T) C.G(ly.QB + i) = C.V(cur + i);
    if (C.l == 0) C.V(ly.QBD) = qb0;
    __syncwarp();
    double beta = 0.0, prev = -1.0, ext = 0.0;
    int k = 1;
    bool done = !active;
    const bool any_early = __any_sync(FULL, active && try_early);
    for (int j = 0; j < LANCZOS_KMAX; ++j) {
        if (j > 0) {
            for (int i = C.l; i < m; i += T) C.V(W + i) = C.V(cur + i);
            __syncwarp();
            team_solve<1>(C, m, true, W, m);
        }
        double sp = 0.0;
        for (int i = C.l & 3; i < m; i += 4) sp += C.V(W + i);
        const double qbj = C.V(ly.QBD + j);
        const double dd = (C.sum4(sp) - qbj) / s;
        __syncwarp();
        for (int i = C.l; i < m; i += T) {
            double v = C.V(W + i);
            if (i < n) v = fma(-dd, C.V(ly.U + i), v);
            if (j > 0) v = fma(-beta, C.V(old + i), v);
            C.V(W + i) = v;
        }
        double wb = dd;
        __syncwarp();
        double ap = 0.0;
        for (int i = C.l & 3; i < m; i += 4) ap = fma(C.V(cur + i), C.V(W + i), ap);
        if (j > 0) wb = fma(-beta, C.V(ly.QBD + j - 1), wb);
        const double a = fma(qbj, wb, C.sum4(ap));
        __syncwarp();
        for (int i = C.l; i < m; i += T) C.V(W + i) = fma(-a, C.V(cur + i), C.V(W + i));
        __syncwarp();
        double bp = 0.0;
        for (int i = C.l & 3; i < m; i += 4) {
            const double v = C.V(W + i);
            bp = fma(v, v, bp);
        }
        wb = fma(-a, qbj, wb);
        const double bn = sqrt(fma(wb, wb, C.sum4(bp)));
        if (C.l == 0) {
            C.V(ly.AL + j) = a;
            C.V(ly.BE + j) = bn;
        }
        __syncwarp();
        const bool last = bn <= 1e-14 * fabs(a) || j + 1 == LANCZOS_KMAX;
        const bool need = j + 1 >= LANCZOS_KMIN - 1 || (any_early && early_accept_factor(j + 1) > 0.0) || last;
        if (__any_sync(FULL, need && !done)) {
            const double e = team_tri_extreme(C, ly.AL, ly.BE, ly.A32, j + 1);
            if (!done) {
                ext = e;
                k = j + 1;
                if (try_early && j + 1 < LANCZOS_KMIN) {
                    const double est = lmax * fabs(ext);
                    if (est >= acc_lo && est <= early_accept_factor(j + 1) * acc_hi) {
                        *early = true;
                        done = true;
                    }
                }
                if (j + 1 >= LANCZOS_KMIN && fabs(fabs(ext) - prev) <= rtol * fabs(ext)) done = true;
                if (last) done = true;
                prev = fabs(ext);
            }
        }
        if (__all_sync(FULL, done)) break;
        beta = bn;
        const double ib = 1.0 / bn;
        const int nx = old;
        old = cur;
        cur = nx;
        for (int i = C.l; i < m; i += T) {
            const double v = C.V(W + i) * ib;
            C.V(cur + i) = v;
            C.G(ly.QB + (j + 1) * m + i) = v;
        }
        if (C.l == 0) C.V(ly.QBD + j + 1) = wb * ib;
        __syncwarp();
    }
    // the slope needs the Ritz vector, unless the guess was accepted early
    if (__any_sync(FULL, active && !*early)) team_ritz_vector(C, m, k, ext);
    return ext;
}

// d lambda / d eps_s with the Ritz vector in RV (eig_derivative of build.cu):
// a row per lane, then the rows' products added by row mod 4 in row order
template <typename Tm>
__device__ __noinline__ double team_eig_derivative(const Tm C, int m, int n, int kernel, double eps_s) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, true);
    const int RV = ly.G + 2 * m;
    double acc = 0.0;   // partial sum (row mod 4 = l & 3)
    for (int i0 = 0; i0 < n; i0 += T) {
        const int i = i0 + C.l;
        double p = 0.0;
        if (i > 0 && i < n) {
            const int base = pk(i, 0);
            double row[4] = {0.0, 0.0, 0.0, 0.0};
            int j = 0;
#pragma unroll 2
            for (; j + 4 <= i; j += 4) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double ph = C.G(ly.PH + base + j + q);
                    const double g = kernel == RBFFD_GAUSSIAN ? 2.0 * ph : ph * ph * ph;
                    row[q] = fma(g * C.G(ly.R2 + base + j + q), C.V(RV + j + q), row[q]);
                }
            }
            for (; j < i; ++j) {
                const double ph = C.G(ly.PH + base + j);
                const double g = kernel == RBFFD_GAUSSIAN ? 2.0 * ph : ph * ph * ph;
                row[0] = fma(g * C.G(ly.R2 + base + j), C.V(RV + j), row[0]);
            }
            p = (row[0] + row[1]) + (row[2] + row[3]);
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < T; h += 4) {
            const int k = h + (C.l & 3), ik = i0 + k;
            const double pk_ = C.from(p, k);
            if (ik > 0 && ik < n) acc = fma(C.V(RV + ik), pk_, acc);
        }
    }
    return -2.0 * eps_s * C.sum4(acc);
}

// ---------------------------------------------------------------------------
// weights
// ---------------------------------------------------------------------------

// [c; d] = A^{-1} [f; 0] for NR right-hand sides (regions R0, R0 + m, ...):
// the solves, then the sums over the real entries in index order, a
// right-hand side per lane
template <int NR, typename Tm>
__device__ void team_aug_solve0(const Tm& C, const TeamLayout& ly, bool search, int n, int R0, double s) {
    constexpr int T = Tm::T;
    const int m = ly.m;
    team_solve<NR>(C, m, search, R0, m);
    double sum = 0.0;
    const int mine = R0 + (C.l % NR) * m;
    for (int i = 0; i < n; ++i) sum += C.V(mine + i);
    const double d = sum / s;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        const double dq = C.from(d, q);
        for (int i = C.l; i < n; i += T) C.V(R0 + q * m + i) = fma(-dq, C.V(ly.U + i), C.V(R0 + q * m + i));
    }
    __syncwarp();
}

// First row of L_P (first_row_weights of build.cu) into region W, scaled by
// r_s^2.  PH is overwritten with the shape of psi; every entry v_j sums the
// other nodes' terms in index order, the order in which the lane-per-stencil
// kernel's pair loop reaches it.
template <typename Tm>
__device__ __noinline__ void team_row_weights(const Tm C, int m, bool search, int n, int kernel, double eps_s,
                                              double s) {
    constexpr int T = Tm::T;
    const TeamLayout ly = team_layout(m, search);
    const int XS = ly.XS, GV = ly.G;
    const double e2 = eps_s * eps_s;
    const double n0x = C.G(ly.NS), n0y = C.G(ly.NS + m), n0z = C.G(ly.NS + 2 * m);
    for (int j = C.l; j < m; j += T) {
        double gx = 0.0, gy = 0.0, gz = 0.0;
        if (j > 0 && j < n) {
            const double ph = C.G(ly.PH + pk(j, 0));
            const double ps = psi_from_phi(kernel, e2, ph);
            const double dx = -C.G(XS + j), dy = -C.G(XS + m + j), dz = -C.G(XS + 2 * m + j);
            const double nd = n0x * dx + n0y * dy + n0z * dz;
            gx = ps * (dx - n0x * nd);
            gy = ps * (dy - n0y * nd);
            gz = ps * (dz - n0z * nd);
        }
        C.V(GV + j) = gx;
        C.V(GV + m + j) = gy;
        C.V(GV + 2 * m + j) = gz;
    }
    __syncwarp();
    team_aug_solve0<3>(C, ly, search, n, GV, s);
    // h_i = P_i g_i, in place
    for (int i = C.l; i < n; i += T) {
        const double gx = C.V(GV + i), gy = C.V(GV + m + i), gz = C.V(GV + 2 * m + i);
        const double nx = C.G(ly.NS + i), ny = C.G(ly.NS + m + i), nz = C.G(ly.NS + 2 * m + i);
        const double nd = nx * gx + ny * gy + nz * gz;
        C.V(GV + i) = gx - nx * nd;
        C.V(GV + m + i) = gy - ny * nd;
        C.V(GV + 2 * m + i) = gz - nz * nd;
    }
    if (kernel != RBFFD_GAUSSIAN)
        for (int e = C.l; e < pk(n, 0); e += T) C.G(ly.PH + e) = psi_shape(kernel, C.G(ly.PH + e));
    __syncwarp();
    const double cs = psi_scale(kernel, e2);
    for (int j0 = 0; j0 < m; j0 += T) {
        const int j = j0 + C.l, jj = min(j, n - 1);
        const double xj = C.G(XS + jj), yj = C.G(XS + m + jj), zj = C.G(XS + 2 * m + jj);
        double v = 0.0;
        int e = ly.PH + pk(jj, 0);   // element (max(jj, c), min(jj, c))
#pragma unroll 4
        for (int c = 0; c < n; ++c) {
            const double ps = C.G(e);
            e += c < jj ? 1 : c + 1;
            const double dx = C.G(XS + c) - xj, dy = C.G(XS + m + c) - yj, dz = C.G(XS + 2 * m + c) - zj;
            const double u = fma(ps, dx * C.V(GV + c) + dy * C.V(GV + m + c) + dz * C.V(GV + 2 * m + c), v);
            if (c != jj) v = u;
        }
        if (j < m) C.V(ly.W + j) = j < n ? v * cs : 0.0;
    }
    __syncwarp();
    team_aug_solve0<1>(C, ly, search, n, ly.W, s);
}

// u = Phi^{-1} 1 (with W solved beside it when TWO) and the Schur complement
// 1^T u summed in index order
template <bool TWO, typename Tm>
__device__ double team_schur(const Tm& C, const TeamLayout& ly, bool search, int n) {
    for (int i = C.l; i < ly.m; i += Tm::T) C.V(ly.U + i) = i < n ? 1.0 : 0.0;
    __syncwarp();
    team_solve<TWO ? 2 : 1>(C, ly.m, search, ly.U, ly.W - ly.U);
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += C.V(ly.U + i);
    return s;
}

// ---------------------------------------------------------------------------
// kernels (one warp per block)
// ---------------------------------------------------------------------------

template <typename Tm>
__device__ __forceinline__ Tm make_team(double* scratch, int64_t warp, int size, double* shared) {
    Tm C;
    const int lane = threadIdx.x & 31;
    C.l = lane / Tm::S;
    C.t = lane % Tm::S;
    C.g = scratch + warp * (int64_t)size * Tm::S + C.t;
    C.v = shared + C.t;
    return C;
}

// Search and weights.  `refill`: teams that must be done before the warp
// forms their weights and takes new stencils.
template <int T>
__global__ void __launch_bounds__(32) team_search_kernel(SearchArgs A, int refill) {
    extern __shared__ __align__(16) double team_smem[];
    using Tm = Team<T>;
    const Tm C = make_team<Tm>(A.scratch, blockIdx.x, A.lane_size, team_smem);
    const double acc_lo = A.acc_lo * A.kT * (1.0 + ACCEPT_MARGIN);
    const double acc_hi = A.acc_hi * A.kT * (1.0 - ACCEPT_MARGIN);
#pragma unroll 1
    for (int g = 0; g < A.gi.ngroups; ++g) {
        const int n = A.gi.n[g], m = A.gi.npad[g];
        const TeamLayout ly = team_layout(m, true);
        const int64_t off = A.gi.ell_off[g], cnt = A.gi.row_begin[g + 1] - A.gi.row_begin[g];
        bool have = false, more = true;   // this team holds a stencil; stencils may be left
        int64_t lr = 0;
        int node = 0;
        Search st;
        st.phase = PH_DONE;
        st.x_next = st.x_ret = 0.0;
        Geo geo;
        geo.rs = 1.0;
        geo.mean_d = 1.0;
        double tol_s = 0.0;
        bool learned = false;
        while (true) {
            // ---- teams without a stencil take the next ones
            bool fresh = false;
            const unsigned want = __ballot_sync(FULL, !have && C.l == 0);
            if (more && want) {
                unsigned long long first = 0;
                if ((threadIdx.x & 31) == 0) first = atomicAdd(&A.counters[g], (unsigned long long)__popc(want));
                first = __shfl_sync(FULL, first, 0);
                lr = have ? lr : (int64_t)first + __popc(want & ((1u << C.t) - 1u));
                fresh = !have && lr < cnt;
                more = (int64_t)first + __popc(want) < cnt;
                have = have || fresh;
            }
            if (!__any_sync(FULL, have)) break;
            if (__any_sync(FULL, fresh)) {
                const int64_t r = A.gi.row_begin[g] + (fresh ? lr : 0);
                const float gs = fresh && A.guess_rows ? A.guess_rows[r] : NAN;
                const bool mean = __any_sync(FULL, fresh && !isfinite(gs));
                const Geo gn = team_geometry(
                    C, ly, n, fresh, mean, [&](int j) { return A.idx[ell_elem(off, m, lr, j)]; }, A.X, A.NR);
                if (fresh) {
                    geo = gn;
                    node = A.row_node[r];
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
                    learned = isfinite(gs);
                    st.x_next = clampd(learned ? learned_start(gs, n) : log(1.0 / geo.mean_d), A.xlo, A.xhi);
                }
            }
            // ---- one evaluation of kappa for every team
            const double eps_s = exp(st.x_next);
            const bool running = have && st.phase != PH_DONE;
            const bool first_guess = running && learned && st.phase == PH_FIRST;
            team_assemble(C, ly, n, A.kernel, eps_s, true);
            const bool spd = team_cholesky(C, m, true);
            const double lmax = team_lanczos_max(C, m, n, LANCZOS_RTOL);
            const double qb0 = team_lanczos_start(C, ly, n, ly.G, (uint64_t)node);
#pragma unroll 1
            for (int i = C.l; i < m; i += T) C.V(ly.W + i) = C.V(ly.G + i);
            const double s = team_schur<true>(C, ly, true, n);
            const bool sound = spd && s > 0.0;
            const double schur = sound ? s : 0.0;
            bool early = false;
            const double theta = team_lanczos_inv(C, m, n, s, LANCZOS_RTOL, qb0, running && sound, first_guess, lmax,
                                                  acc_lo, acc_hi, &early);
            double k = sound ? lmax * fabs(theta) : INFINITY;
            if (!isfinite(k)) k = INFINITY;
            const bool accept_now = first_guess && (early || (k >= acc_lo && k <= acc_hi));
            const bool slope = running && isfinite(k) && !accept_now;
            double dF = NAN;
            if (__any_sync(FULL, slope)) {
                const double d = -eps_s * theta * team_eig_derivative(C, m, n, A.kernel, eps_s);
                if (slope) dF = d;
            }
            if (running) search_update(st, F_of(k, A.kT), dF, k, tol_s, A.max_evals, acc_lo, acc_hi, learned, n);
            // ---- weights of the teams that are done, from their last factorisation
            const bool finished = have && st.phase == PH_DONE;
            const int ndone = __popc(__ballot_sync(FULL, finished && C.l == 0));
            const int nhave = __popc(__ballot_sync(FULL, have && C.l == 0));
            if (ndone >= min(refill, nhave)) {
                team_row_weights(C, m, true, n, A.kernel, exp(st.x_ret), s);
                if (finished) {
                    const bool valid = isfinite(st.k_ret) && schur > 0.0;
                    const double inv_rs2 = 1.0 / (geo.rs * geo.rs);
#pragma unroll 1
                    for (int j = C.l; j < m; j += T) {
                        const double w = (valid && j < n) ? C.V(ly.W + j) * inv_rs2 : 0.0;
                        const int64_t e = ell_elem(off, m, lr, j);
                        A.w64[e] = w;
                        A.w32[e] = (float)w;
                    }
                    if (C.l == 0) {
                        A.eps[node] = exp(st.x_ret) / geo.rs;
                        A.kappa[node] = st.k_ret;
                        A.evals[node] = st.evals;
                        A.status[node] = valid ? st.status : RBFFD_STENCIL_SINGULAR;
                    }
                    have = false;
                }
                __syncwarp();
            }
        }
    }
}

// Weights at given shape parameters: the rows of an operator (idx in its
// sliced layout; failed rows get zeros and their status), or rows x n
// stencils as a dense array (failed rows get NaN).
template <int T>
__global__ void __launch_bounds__(32) team_weights_kernel(TeamWeightArgs B) {
    extern __shared__ __align__(16) double team_smem[];
    using Tm = Team<T>;
    constexpr int S = Tm::S;
    const WeightArgs& A = B.w;
    const Tm C = make_team<Tm>(A.scratch, blockIdx.x, A.lane_size, team_smem);
    const bool dense = B.stencils != nullptr;
    const int groups = dense ? 1 : A.gi.ngroups;
#pragma unroll 1
    for (int g = 0; g < groups; ++g) {
        const int n = dense ? B.n : A.gi.n[g], m = (n + 3) / 4 * 4;
        const TeamLayout ly = team_layout(m, false);
        const int64_t off = dense ? 0 : A.gi.ell_off[g], row0 = dense ? 0 : A.gi.row_begin[g];
        const int64_t cnt = dense ? B.rows : A.gi.row_begin[g + 1] - row0;
#pragma unroll 1
        for (int64_t first = (int64_t)blockIdx.x * S; first < cnt; first += (int64_t)gridDim.x * S) {
            const int64_t lr = first + C.t;
            const bool have = lr < cnt;
            bool ok = have;
            const int32_t* row = dense ? B.stencils + (have ? lr : 0) * n : nullptr;
            if (dense) {
                if (have)
#pragma unroll 1
                    for (int j = C.l; j < n; j += T) ok = ok && row[j] >= 0 && (int64_t)row[j] < B.N;
                // every lane of the team has to agree
                const unsigned bad = __ballot_sync(FULL, have && !ok);
                unsigned mine = 0;
#pragma unroll
                for (int k = 0; k < T; ++k) mine |= 1u << (k * S + C.t);
                ok = have && !(bad & mine);
            }
            const Geo geo = team_geometry(
                C, ly, n, ok, false, [&](int j) { return dense ? row[j] : A.idx[ell_elem(off, m, lr, j)]; }, A.X, A.NR);
            const int64_t node = dense ? lr : have ? A.row_node[row0 + lr] : 0;
            const double eps_s = ok ? A.eps_node[node] * geo.rs : 1.0;
            team_assemble(C, ly, n, A.kernel, eps_s, false);
            ok = team_cholesky(C, m, false) && ok && isfinite(eps_s) && eps_s > 0.0;
            const double s = team_schur<false>(C, ly, false, n);
            ok = ok && s > 0.0 && isfinite(s);
            team_row_weights(C, m, false, n, A.kernel, eps_s, s);
            const double inv_rs2 = 1.0 / (geo.rs * geo.rs);
            if (have && !ok && C.l == 0) {
                atomicAdd(A.nfail, 1);
                if (!dense) A.status[node] = RBFFD_STENCIL_SINGULAR;
            }
            if (have && dense) {
#pragma unroll 1
                for (int j = C.l; j < n; j += T) A.w64[lr * n + j] = ok ? C.V(ly.W + j) * inv_rs2 : NAN;
            } else if (have) {
#pragma unroll 1
                for (int j = C.l; j < m; j += T) {
                    const double w = ok && j < n ? C.V(ly.W + j) * inv_rs2 : 0.0;
                    const int64_t e = ell_elem(off, m, lr, j);
                    A.w64[e] = w;
                    A.w32[e] = (float)w;
                }
            }
            __syncwarp();
        }
    }
}

// one-warp blocks resident on the chip with the given shared memory each
rbffd_status resident_warps(const void* kernel, size_t smem, int* warps) {
    RBFFD_TRY(allow_shared(kernel));
    int per_sm = 0;
    RBFFD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32, smem));
    *warps = std::max(1, per_sm) * sm_count();
    return RBFFD_OK;
}

template <int T>
rbffd_status search_with(SearchArgs A, int mmax, int64_t rows, cudaStream_t st) {
    constexpr int S = Team<T>::S;
    const TeamLayout ly = team_layout(mmax, true);
    const size_t smem = (size_t)ly.vsize * S * sizeof(double);
    int warps = 0;
    rbffd_status r = resident_warps((const void*)team_search_kernel<T>, smem, &warps);
    if (r != RBFFD_OK) return r;
    warps = (int)std::min<int64_t>(warps, (rows + S - 1) / S);
    RBFFD_CUDA_TRY(pool_alloc(&A.scratch, (size_t)warps * S * ly.size * sizeof(double), st));
    A.lane_size = ly.size;
    team_search_kernel<T><<<warps, 32, smem, st>>>(A, std::max(1, S / 2));
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    RBFFD_CUDA_TRY(cudaFreeAsync(A.scratch, st));
    return RBFFD_OK;
}

template <int T>
rbffd_status weights_with(TeamWeightArgs B, int mmax, int64_t rows, int64_t scratch_doubles, cudaStream_t st) {
    constexpr int S = Team<T>::S;
    const TeamLayout ly = team_layout(mmax, false);
    const size_t smem = (size_t)ly.vsize * S * sizeof(double);
    int warps = 0;
    rbffd_status r = resident_warps((const void*)team_weights_kernel<T>, smem, &warps);
    if (r != RBFFD_OK) return r;
    warps = (int)std::min<int64_t>(warps, (rows + S - 1) / S);
    B.w.lane_size = ly.size;
    double* own = nullptr;
    if (scratch_doubles > 0) {
        warps = (int)std::min<int64_t>(warps, scratch_doubles / ((int64_t)ly.size * S));
        RBFFD_CHECK_ARG(warps >= 1, "scratch too small for the stencil size");
    } else {
        RBFFD_CUDA_TRY(pool_alloc(&own, (size_t)warps * S * ly.size * sizeof(double), st));
        B.w.scratch = own;
    }
    team_weights_kernel<T><<<warps, 32, smem, st>>>(B);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    if (own) RBFFD_CUDA_TRY(cudaFreeAsync(own, st));
    return RBFFD_OK;
}

}  // namespace

// Measured on one GB300 (sphere, IMQ, kappa_T 1e12, plain search; ms for a
// lane / 4 / 8 / 16 lanes per stencil, the chosen one marked):
//   n = 31:   1.3k 17.3/-/3.6/2.9*   5k 23.7/8.0/6.2*/8.2   10k 23.5/8.9*/10.0/16.9
//             20k 30.8/17.0*/22.2/35.4   80k 80.7*/60.2/88.1/-   320k 296*/249/391/-
//   n = 50:   5k 60.7/20.1/13.0*/15.8   10k 90.1/29.1/23.4*/31.7   20k 83.3/32.3*/35.8/63.3
//             50k 103/78.0*/93.6/-   160k 264*/241/352/-   320k 468*/446/691/-
//   n = 58:   10k 86.2/29.5/24.1*/34.0   25k 95.2/56.3/55.9*/-   50k 109*/101/113/-   80k 157*/161/184/-
//   n = 78:   5k 122/34.4/25.7*/25.5   25k 154/129/89.6*/-   50k 187*/261/184/-
//   n = 101:  5k 180/80/46.6/39.3*   20k 205/215/127*/129   80k 399*/758/447/-
// Few stencils want many lanes each (all schedulers busy), many want few
// (fewer float64 instructions per stencil).  From n = 57 the vectors of eight
// teams of 4 lanes leave too few warps per SM.  With fewer evaluations per
// stencil the lane kernel catches up earlier (torus, kappa_T 1e8, lane / team:
// n = 15 20k 4.7/6.1, 51k 9.6/12.4; n = 31 51k 23.2/31.1; n = 50 51k 63.7/63.0,
// 120k sphere 132/152), so it takes over there.  From learned guesses (about
// one evaluation each) it is the other way round, since few rounds leave its
// long instruction stream exposed (n = 31: 80k 24.9/14.2, 250k 40.7/34.6; n = 50:
// 160k 98.9/57.0, 250k 71.0/67.5; n = 101: 50k 144/65.2, 80k 127/96, 160k 264/271).
int team_lanes(int m, int64_t rows, bool guesses) {
    if (rows < 900) return 32;
    if (rows < (m > 80 ? 12000 : 3500)) return 16;
    if (m > 56) return rows < (guesses ? 100000 : 40000) ? 8 : 0;
    if (rows < (m > 32 ? 18000 : 8000)) return 8;
    return rows < (guesses ? 250000 : m > 36 ? 80000 : m > 24 ? 40000 : 25000) ? 4 : 0;
}

rbffd_status team_search(SearchArgs A, int mmax, int64_t rows, cudaStream_t st) {
    switch (team_lanes(mmax, rows, A.guess_rows != nullptr)) {
        case 4: return search_with<4>(A, mmax, rows, st);
        case 16: return search_with<16>(A, mmax, rows, st);
        case 32: return search_with<32>(A, mmax, rows, st);
        default: return search_with<8>(A, mmax, rows, st);
    }
}

// The weights at given shape parameters, one factorisation and five solves per
// stencil (sphere, IMQ; ms for a lane / 4 / 8 / 16 / 32 lanes per stencil):
//   n = 31:   700 1.14/0.38/0.24/0.18/0.17*   2.6k 1.15/0.42/0.31*/0.42/0.53
//             10k 1.35/1.01/0.96*/1.13/1.67   40k 2.63*/2.71/3.05/4.01/6.30
//   n = 50:   10k 4.05/2.59/2.39*/2.68/3.55   100k 14.6*/16.8/18.5/-/-
//   n = 101:  2k 18.2/5.66/3.04/2.18*/2.75   20k 26.2/25.8/18.9*/19.8/23.9   100k 73*/114/85/-/-
int team_weight_lanes(int m, int64_t rows) {
    if (rows < 1200) return m > 80 ? 16 : 32;
    if (rows < 3500 && m > 60) return 16;
    return rows < (m > 60 ? 50000 : 25000) ? 8 : 0;
}

// scratch_doubles > 0: the caller's scratch (B.w.scratch) of that many
// doubles, nothing is allocated; 0: scratch from the pool
rbffd_status team_weights(TeamWeightArgs B, int64_t scratch_doubles, cudaStream_t st) {
    int mmax = 0;
    int64_t rows = B.rows;
    if (B.stencils) {
        mmax = (B.n + 3) / 4 * 4;
    } else {
        rows = B.w.gi.row_begin[B.w.gi.ngroups];
#pragma unroll 1
        for (int g = 0; g < B.w.gi.ngroups; ++g) mmax = std::max(mmax, B.w.gi.npad[g]);
    }
    int T = std::max(8, team_weight_lanes(mmax, rows));
    // a fixed scratch holds so many teams: enough lanes per team for a warp per scheduler
    if (scratch_doubles > 0)
        while (T < 32 && scratch_doubles / team_layout(mmax, false).size * T < (int64_t)4 * 32 * sm_count()) T *= 2;
    switch (T) {
        case 16: return weights_with<16>(B, mmax, rows, scratch_doubles, st);
        case 32: return weights_with<32>(B, mmax, rows, scratch_doubles, st);
        default: return weights_with<8>(B, mmax, rows, scratch_doubles, st);
    }
}

}  // namespace rbffd
