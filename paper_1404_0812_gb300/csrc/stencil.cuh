// Device code that every build kernel shares: the radial kernels, the
// tridiagonal eigenvalue helpers, the per-stencil root finder and the kernels'
// argument blocks (Sections 2 and 5).
#pragma once

#include "common.cuh"

#include <cmath>

namespace rbffd {
namespace {

constexpr int LANCZOS_KMAX = 24;
constexpr double LANCZOS_RTOL = 1e-6;       // relative change that stops a Lanczos run
// The A^{-1} run never stops before this many steps: when the second
// smallest |eigenvalue| of A is within a factor 0.6-0.9 of the smallest, the
// top Ritz value can sit on the second one for several steps (the component
// of lambda_min's eigenvector grows by (1 + 2 sqrt(gap))^k per step), and
// stopping on a stalled value misjudges kappa by 10-40 %.
constexpr int LANCZOS_KMIN = 10;
constexpr double ACCEPT_MARGIN = 1e-4;      // shrink the accept band by this
// Early acceptance of a learned first guess.  Every Ritz value of the A^{-1}
// run is a lower bound of 1 / min|lambda(A)| (and the A run's of
// max|lambda(A)|), so the running estimate k_j = lambda_max theta_j never
// exceeds kappa: k_j >= accept_lo kappa_T already proves the lower edge.
// The upper edge needs the run's shortfall bounded: over 1.5M first
// evaluations (1M-node sphere, n = 31 / 50 / 70 / 101, and the held-out
// bumpy sphere, n = 50) the smallest ratio theta_j / theta_final was 0.44 at
// step 6, 0.74 at step 7, 0.93 at step 8 and 0.998 at step 9.  A guess is
// accepted at step j when k_j <= f_j accept_hi kappa_T with f_6..f_9 =
// 0.25, 0.45, 0.7, 0.85 (1.1-1.8x below the worst ratios seen); otherwise
// the same run continues to its full length and the usual test decides.
__host__ __device__ inline double early_accept_factor(int steps) {
    return steps == 6 ? 0.25 : steps == 7 ? 0.45 : steps == 8 ? 0.7 : steps == 9 ? 0.85 : 0.0;
}
constexpr double F_FAIL = 60.0;         // F value used when Phi is not numerically SPD

__host__ __device__ inline int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// ---------------------------------------------------------------------------
// kernels phi(eps r) and psi(r) = phi'(r)/r from eps^2 and r^2 (the FMA is
// written out so that every kernel rounds phi alike)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double phi_of(int kernel, double e2, double r2) {
    return kernel == RBFFD_GAUSSIAN ? exp(-(e2 * r2)) : rsqrt(fma(e2, r2, 1.0));
}
// psi in scaled units: Gaussian -2 eps^2 phi, IMQ -eps^2 phi^3
__device__ __forceinline__ double psi_from_phi(int kernel, double e2, double ph) {
    return kernel == RBFFD_GAUSSIAN ? -2.0 * e2 * ph : -e2 * ph * ph * ph;
}
// psi = psi_scale * psi_shape(phi): the pair pass of the weights sums
// psi_shape terms and applies the constant factor once per entry
__device__ __forceinline__ double psi_shape(int kernel, double ph) {
    return kernel == RBFFD_GAUSSIAN ? ph : ph * ph * ph;
}
__device__ __forceinline__ double psi_scale(int kernel, double e2) {
    return kernel == RBFFD_GAUSSIAN ? -2.0 * e2 : -e2;
}

struct Geo {
    double rs;        // stencil radius (max distance to the centre)
    double mean_d;    // mean scaled distance of the n-1 neighbours
};

// ---------------------------------------------------------------------------
// extreme eigenvalues of a symmetric tridiagonal (float32 Sturm bisection)
// ---------------------------------------------------------------------------
__device__ int sturm_below(const float* a, const float* b2, int k, float x) {
    int c = 0;
    float d = a[0] - x;
    if (d < 0.f) ++c;
#pragma unroll 1
    for (int i = 1; i < k; ++i) {
        if (d == 0.f) d = -1e-30f;
        d = (a[i] - x) - b2[i - 1] / d;
        if (d < 0.f) ++c;
    }
    return c;
}

// extreme eigenvalues of T (alpha[0..k-1], beta[0..k-2], scaled into
// [-1, 1]); returns the one of largest magnitude, signed, in double units
__device__ __noinline__ double tri_extreme(const float* a, const float* b2, int k, double scale) {
    float lo = -1.f, hi = 1.f;
    // top eigenvalue: count(x) < k  <=>  x <= lambda_max
#pragma unroll 1
    for (int it = 0; it < 26; ++it) {
        float mid = 0.5f * (lo + hi);
        if (sturm_below(a, b2, k, mid) < k) lo = mid; else hi = mid;
    }
    float top = 0.5f * (lo + hi);
    lo = -1.f; hi = 1.f;
    // bottom eigenvalue: count(x) >= 1  <=>  x > lambda_min
#pragma unroll 1
    for (int it = 0; it < 26; ++it) {
        float mid = 0.5f * (lo + hi);
        if (sturm_below(a, b2, k, mid) >= 1) hi = mid; else lo = mid;
    }
    float bot = 0.5f * (lo + hi);
    return scale * (double)(fabsf(top) >= fabsf(bot) ? top : bot);
}

__device__ double tri_max_abs(const float* a, const float* b2, int k, double scale) {
    return fabs(tri_extreme(a, b2, k, scale));
}

// Eigenvector y (unit) of the symmetric tridiagonal T for its eigenvalue
// theta: two steps of inverse iteration, each a solve with T - theta I by
// Gaussian elimination with partial pivoting (the factor has two
// superdiagonals after row exchanges).
__device__ __noinline__ void tri_eigvec(const double* al, const double* be, int k, double theta, double* y) {
    double d[LANCZOS_KMAX], du[LANCZOS_KMAX], du2[LANCZOS_KMAX], dl[LANCZOS_KMAX];
    bool sw[LANCZOS_KMAX];
    double tmax = 0.0;
#pragma unroll 1
    for (int i = 0; i < k; ++i) tmax = fmax(tmax, fabs(al[i] - theta) + (i < k - 1 ? fabs(be[i]) : 0.0));
    const double tiny = 1e-30 * (tmax > 0.0 ? tmax : 1.0);
#pragma unroll 1
    for (int i = 0; i < k; ++i) {
        d[i] = al[i] - theta;
        du[i] = i < k - 1 ? be[i] : 0.0;
        dl[i] = i < k - 1 ? be[i] : 0.0;
        du2[i] = 0.0;
        sw[i] = false;
    }
#pragma unroll 1
    for (int i = 0; i < k - 1; ++i) {
        if (fabs(d[i]) >= fabs(dl[i])) {
            if (d[i] == 0.0) d[i] = tiny;
            double f = dl[i] / d[i];
            dl[i] = f;
            d[i + 1] -= f * du[i];
        } else {   // exchange rows i and i + 1
            double f = d[i] / dl[i];
            d[i] = dl[i];
            dl[i] = f;
            double t = du[i];
            du[i] = d[i + 1];
            d[i + 1] = t - f * d[i + 1];
            if (i < k - 2) {
                du2[i] = du[i + 1];
                du[i + 1] = -f * du[i + 1];
            }
            sw[i] = true;
        }
    }
    if (d[k - 1] == 0.0) d[k - 1] = tiny;
#pragma unroll 1
    for (int i = 0; i < k; ++i) y[i] = 1.0;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int i = 0; i < k - 1; ++i) {
            if (sw[i]) {
                double t = y[i];
                y[i] = y[i + 1];
                y[i + 1] = t - dl[i] * y[i + 1];
            } else {
                y[i + 1] -= dl[i] * y[i];
            }
        }
        y[k - 1] /= d[k - 1];
        if (k > 1) y[k - 2] = (y[k - 2] - du[k - 2] * y[k - 1]) / d[k - 2];
#pragma unroll 1
        for (int i = k - 3; i >= 0; --i) y[i] = (y[i] - du[i] * y[i + 1] - du2[i] * y[i + 2]) / d[i];
        double nrm = 0.0;
#pragma unroll 1
        for (int i = 0; i < k; ++i) nrm = fmax(nrm, fabs(y[i]));
        double inv = nrm > 0.0 ? 1.0 / nrm : 1.0;
#pragma unroll 1
        for (int i = 0; i < k; ++i) y[i] *= inv;
    }
}

// splitmix64 (Steele, Lea, Flood 2014) mapped to [-1, 1): the pseudo-random
// start vector of the A^{-1} Lanczos run, seeded per stencil, so that no
// stencil's symmetry can leave it (nearly) orthogonal to the eigenvector of
// lambda_min, as a fixed smooth start vector can be.
__device__ inline double unit_hash(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    return (double)(x >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

// ---------------------------------------------------------------------------
// per-lane root finder: safeguarded Newton in x = ln eps_s
// ---------------------------------------------------------------------------
enum { PH_FIRST = 0, PH_NEWTON = 1, PH_DONE = 3 };

struct Search {
    double x_next;        // point to evaluate next
    double lo, hi;        // bracket of the root: F(lo) > 0 > F(hi) (F decreases)
    double x_ret, k_ret;  // result (eps_s = exp(x_ret)) and kappa reported for it
    double dx_prev;
    double f_prev;        // |F| at the previous iterate
    double ulo, uhi;      // caller's search range of x (+-inf when none)
    int phase, evals;
    int status;
};

__device__ inline double clampd(double v, double lo, double hi) { return fmin(fmax(v, lo), hi); }

// dF/dx near the root, about -(11 + n / 10) on quasi-uniform surface
// stencils (measured); used when the computed derivative is unusable.
__device__ inline double slope_model(int n) { return -(11.0 + 0.1 * n); }

// A learned guess predicts the root (kappa = kappa_T).  The search starts a
// slope model's step past it, at kappa ~0.85 kappa_T: early acceptance (see
// early_accept_factor) needs the estimate well below the band's upper edge,
// and the networks' errors leave more room below kappa_T than above it
// inside [0.5, 2] kappa_T.  On the 1M-node sphere this aim moves more first
// evaluations into the step-7 window than it pushes out of the band.
constexpr double LEARNED_AIM = 0.85;
__device__ inline double learned_start(float guess, int n) {
    return (double)guess + log(LEARNED_AIM) / slope_model(n);
}

__device__ inline void finish(Search& s, double x, double k, int status) {
    s.x_ret = x;
    s.k_ret = k;
    s.status = status;
    s.phase = PH_DONE;
}

// Consume F(x_next) = f with derivative d and kappa k.
//  * learned first guess: accepted when kappa is inside the band;
//  * Newton step dx = -f/d (slope model if d is unusable), clamped to +-3,
//    replaced by bisection of the bracket when it would leave it;
//  * stop when the distance to the root is below xtol/2, when the bracket
//    is narrower than xtol, or when the steps stop shrinking at the float64
//    noise floor of kappa (distance below xtol, step at least 0.9 of the
//    previous one); every stop returns the evaluated x, within xtol of the
//    root (the oracle's Brent guarantee).
__device__ __noinline__ void search_update(Search& s, double f, double d, double k, double tol_s, int max_evals,
                              double acc_lo, double acc_hi, bool learned, int n) {
    s.evals++;
    const double x = s.x_next;
    if (s.phase == PH_FIRST && learned && k >= acc_lo && k <= acc_hi) {
        finish(s, x, k, RBFFD_STENCIL_ACCEPTED_PREDICTION);
        return;
    }
    if (f == 0.0) {
        finish(s, x, k, RBFFD_STENCIL_OK);
        return;
    }
    if (f > 0.0) s.lo = fmax(s.lo, x); else s.hi = fmin(s.hi, x);
    // the root lies outside the caller's range: kappa is still above kappa_T
    // at its largest eps, or already below it at its smallest
    if ((f > 0.0 && x >= s.uhi) || (f < 0.0 && x <= s.ulo)) {
        finish(s, x, k, RBFFD_STENCIL_NO_BRACKET);
        return;
    }
    const double xtol = tol_s / exp(x);
    // the Hellmann-Feynman slope is trusted only within a factor 5 of the
    // slope model (a Ritz vector from a clustered pair can be poor)
    const double sm = slope_model(n);
    const bool usable = isfinite(d) && isfinite(f) && f != F_FAIL && d <= 0.2 * sm && d >= 5.0 * sm;
    const double sl = usable ? d : sm;
    double dx = clampd(-f / sl, -3.0, 3.0);
    double xn = x + dx;
    const bool bracketed = isfinite(s.lo) && isfinite(s.hi);
    // safeguard: bisect when the Newton point leaves the bracket, or when the
    // last Newton step did not halve |F| (the bracket then still shrinks
    // geometrically, whatever the quality of the slope)
    const bool slow = s.phase == PH_NEWTON && fabs(f) > 0.5 * s.f_prev;
    const bool bisect = bracketed && (!(xn > s.lo && xn < s.hi) || slow);
    if (bisect) xn = 0.5 * (s.lo + s.hi);
    xn = clampd(xn, s.ulo, s.uhi);
    dx = xn - x;
    // distance of x from the root: after a bisection x is an end of the
    // bracket, so at most 2|dx|; after a Newton step |F| over the flatter of
    // the computed slope and the model (a Ritz vector from a clustered pair
    // can give a slope several times too steep, and with it a step that
    // looks converged while x is still far from the root)
    const double dist = bisect ? fabs(dx) : fabs(f) / fmin(fabs(sl), fabs(sm));
    // every stop returns the evaluated x (its factorisation is still in
    // scratch for the weights)
    if (usable && dist < 0.5 * xtol) {
        finish(s, x, k, RBFFD_STENCIL_OK);
        return;
    }
    // without a usable slope: the same test with the flattest slope that
    // would have been trusted (0.2 |model|); it stops an iteration sitting
    // on the root (|F| at rounding level) whose Ritz vector gives no slope
    if (!usable && f != F_FAIL && fabs(f) < 0.1 * xtol * fabs(sm)) {
        finish(s, x, k, RBFFD_STENCIL_OK);
        return;
    }
    if (bracketed && s.hi - s.lo < xtol) {
        finish(s, x, k, RBFFD_STENCIL_OK);
        return;
    }
    // float64 noise floor of kappa: tiny steps that no longer shrink (a
    // linearly converging Newton, e.g. with a slope off by 2x, shrinks its
    // steps by a constant factor and does not stop here; when it is slow the
    // halving test above bisects instead)
    if (s.phase == PH_NEWTON && usable && dist < xtol && fabs(dx) >= 0.9 * fabs(s.dx_prev)) {
        finish(s, x, k, RBFFD_STENCIL_OK);
        return;
    }
    if (s.evals >= max_evals) {
        finish(s, x, k, bracketed ? RBFFD_STENCIL_NO_CONVERGENCE : RBFFD_STENCIL_NO_BRACKET);
        return;
    }
    s.dx_prev = dx;
    s.f_prev = fabs(f);
    s.x_next = xn;
    s.phase = PH_NEWTON;
}

__device__ inline double F_of(double k, double kT) {
    return isfinite(k) ? log(k / kT) : F_FAIL;
}

}  // namespace

// argument blocks of the build kernels (build.cu, team.cu)
struct SearchArgs {
    const double* X;
    const double* NR;
    double* w64;
    float* w32;
    const int32_t* idx;
    const int32_t* row_node;
    GroupInfo gi;
    double* scratch;
    int lane_size;
    int kernel;
    double kT, tol, acc_lo, acc_hi;
    double xlo, xhi;             // search range of ln(eps * r_s) (+-inf when none)
    int max_evals;
    const float* guess_rows;     // ln(eps_s) per internal row, or NULL
    unsigned long long* counters;  // per group
    double* eps;
    double* kappa;
    int32_t* evals;
    int32_t* status;
};

struct WeightArgs {
    const double* X;
    const double* NR;
    const int32_t* idx;
    const int32_t* row_node;
    GroupInfo gi;
    double* scratch;
    int lane_size;
    int kernel;
    const double* eps_node;
    double* w64;
    float* w32;
    int32_t* status;      // written only on failure
    int* nfail;
};

// weights at given shape parameters on teams: the operator's rows, or
// (stencils given) rows x n stencils of nodes in [0, N)
struct TeamWeightArgs {
    WeightArgs w;               // dense: X, NR, scratch, lane_size, kernel, eps_node (per row), w64, nfail
    const int32_t* stencils;    // dense: rows x n; NULL for an operator
    int64_t N, rows;
    int n;
};

// team.cu: lanes per stencil for a search over (weights of) rows stencils of
// padded size m, with learned guesses or without (0: the lane-per-stencil kernel is the faster one); the search
// and the weights on teams
int team_lanes(int m, int64_t rows, bool guesses);
int team_weight_lanes(int m, int64_t rows);
rbffd_status team_search(SearchArgs A, int m, int64_t rows, cudaStream_t st);
rbffd_status team_weights(TeamWeightArgs B, int64_t scratch_doubles, cudaStream_t st);

}  // namespace rbffd
