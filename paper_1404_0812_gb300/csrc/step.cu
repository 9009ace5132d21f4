// IMEX method-of-lines stepping (Section 4.2 method of lines; Section 7
// SBDF2 with the diffusion implicit; BiCGSTAB as Section 4.2 / Section 6 use).
//
//   d/dt u = delta_u L u + f(u, v),  d/dt v = delta_v L v + g(u, v)
//   SBDF2:  (3 I - 2 dt delta L) u^{n+1} = 4 u^n - u^{n-1} + 2 dt (2 f^n - f^{n-1})
//   first step without history: (I - dt delta L) u^1 = u^0 + dt f^0
//
// GPU design: both species are solved together, so each pass over the ELL
// matrix serves two products, and the solution is updated in place in u, v.
// Operators that fit the shared memory of the chip (up to about 30 MB) run all
// steps of a call in one launch with the matrix resident there
// (step_resident.cuh).  Larger ones run BiCGSTAB as a sequence of
// full-occupancy phase kernels under a device-side WHILE graph node (the
// phase-kernel section below says why and how).  A direct step is three
// launches: right-hand side, substitutions (lu.cu), report.
#include "common.cuh"
#include "step_plan.cuh"

#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>
#include <vector>

// Loop state of the phase-kernel BiCGSTAB (device memory).  Each phase
// kernel reads it as its previous kernel left it; only the last block of a
// phase (by ticket) writes it, after every other block of that phase has
// finished reading, a lane per species (the phase kernels' threads do no
// float64 scalar arithmetic).
struct SpeciesState {
    double bnorm, limit2;              // |b|; squared norm at which the residual has converged
    double rho, rho_prev, alpha, omega, res2;   // committed: (r-hat, r), ..., |r|^2
    double beta, alpha_n, omega_n;     // the current iteration's scalars
    int e0, e;                         // exponents of r-hat and of the iteration's vectors in the sums
    int active, fail, iters, zero;
    int actA, actB, early, actE;       //   and its decisions
};
struct PhaseCtl {
    SpeciesState s[2];
    int it;                      // iterations done in this step
    int more;                    // the loop continues (host-loop mode reads it)
    unsigned int ticket;
};

struct rbffd_step_ws {
    int dtype;
    int64_t N;
    size_t elem;
    void* vec;                     // 2 species x 7 vectors (b, r, rh, p, q, s, t), each padded to a multiple of 4
    unsigned long long* bar;       // barrier counter
    int* flags;                    // [0] error (timeout), [1] not converged, [2] has_history,
                                   // [3] report slot of the next step, [4] order of the last step
    int* rep;                      // per step: iters_u, iters_v, failed
    double* rep_res;               // per step: relres_u, relres_v
    double* tstart;                // time of u at the start of the call (device copy)
    int64_t rep_cap;
    cudaGraphExec_t graph;            // captured step
    cudaStream_t cap;                 // library-owned stream used only for capture
    unsigned char graph_args[1024];   // kernel arguments the graph holds
    size_t graph_args_size;
    int solver;                       // path the graph was captured with (1 LU, 2 phases)
    rbffd_lu* lu[4][2];               // banded LU factors by SBDF order and species
    rbffd_lu* graph_lu[4][2];         // the factors the captured graph's solve reads
    double* ywork;                    // the LU substitutions' work: per species 2 N + 16 float64
    PhaseCtl* ctl;                    // phase-kernel path: loop state
    double* pp;                       //   per-block partial sums
    int* more_host;                   //   host loop: pinned word in which a phase says whether the loop goes on
    int more_seq;                     //   and the number of the last phase that was launched to do so
    double* rpart;                    // resident kernel: per-block sums of two reductions
    rbffd::ResidentPlan plan[2];      //   and its shape by number of species
    bool planned[2];
};

namespace rbffd {

void step_ws_free(rbffd_step_ws* ws) {
    if (!ws) return;
    cudaFree(ws->vec);
    cudaFree(ws->bar);
    cudaFree(ws->flags);
    cudaFree(ws->rep);
    cudaFree(ws->rep_res);
    cudaFree(ws->tstart);
    if (ws->graph) cudaGraphExecDestroy(ws->graph);
    if (ws->cap) cudaStreamDestroy(ws->cap);
    for (auto& row : ws->lu)
        for (rbffd_lu* f : row) lu_free(f);
    cudaFree(ws->ywork);
    cudaFree(ws->ctl);
    cudaFree(ws->pp);
    if (ws->more_host) cudaFreeHost(ws->more_host);
    cudaFree(ws->rpart);
    delete ws;
}

namespace {

template <typename T>
struct Args {
    const int32_t* idx;
    const T* w;
    const int32_t* row_node;
    GroupInfo gi;
    int64_t N;
    T *u, *v, *up, *vp, *fp, *gp;
    T *up2, *vp2, *fp2, *gp2;   // levels n-2 and n-3 (SBDF3 / SBDF4 only)
    T *up3, *vp3, *fp3, *gp3;
    int order;         // SBDF order 1..4
    const T *su, *sv;  // source profiles h_u, h_v (or NULL): s(t) = exp(rate t) h
    double src_rate;
    const double* tstart;   // time of u when the call began
    T* vec;            // 2 x 7 vectors of ldv elements
    int64_t ldv;       // their stride: N rounded up to a multiple of 4 (16-byte aligned vectors)
    int vec4;          // the state u (and v) 16-byte aligned: the vector phases move 4 elements at a time
    int ns;
    int model;
    T c[8];
    T dt;
    T delta[2];
    double tol;
    int maxit;
    unsigned long long* bar;
    int* flags;
    int* rep;
    double* rep_res;
    PhaseCtl* ctl;                         // phase-kernel path: loop state and totals
    double* pp;                            //   per-block partial sums (blocks x 8)
    cudaGraphConditionalHandle cond;       //   WHILE handle of the step graph (0: host loop)
    int* more_host;                        //   host loop: where R and E say 2 more_seq + (the loop goes on)
    int more_seq;
};

enum { VB = 0, VR = 1, VRH = 2, VP = 3, VQ = 4, VS = 5, VT = 6 };

template <typename T>
__host__ __device__ __forceinline__ T* V(const Args<T>& a, int sp, int k) {
    return a.vec + ((int64_t)sp * 7 + k) * a.ldv;
}

template <typename T>
__device__ __forceinline__ void react(const Args<T>& a, T u, T v, T& f, T& g) {
    switch (a.model) {
        case RBFFD_MODEL_LINEAR: f = a.c[0] * u; g = a.c[1] * v; break;
        case RBFFD_MODEL_SCHNAKENBERG: {
            T uuv = u * u * v;
            f = a.c[2] * (a.c[0] - u + uuv);
            g = a.c[2] * (a.c[1] - uuv);
        } break;
        case RBFFD_MODEL_GRAY_SCOTT: {
            T uvv = u * v * v;
            f = -uvv + a.c[0] * (T(1) - u);
            g = uvv - (a.c[0] + a.c[1]) * v;
        } break;
        case RBFFD_MODEL_BARRIO: {   // Eqs. turing1, turing2
            T al = a.c[0], be = a.c[1], ga = a.c[2], t1 = a.c[3], t2 = a.c[4];
            f = al * u * (T(1) - t1 * v * v) + v * (T(1) - t2 * u);
            g = be * v * (T(1) + (al * t1 / be) * u * v) + u * (ga + t2 * v);
        } break;
        default: f = T(0); g = T(0);
    }
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ void load4s(const float* p, float (&w)[4]) {
    float4 v = __ldcs(reinterpret_cast<const float4*>(p));
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
__device__ __forceinline__ void load4s(const double* p, double (&w)[4]) {
    double2 a = __ldcs(reinterpret_cast<const double2*>(p));
    double2 b = __ldcs(reinterpret_cast<const double2*>(p + 2));
    w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
}

// the SBDF order, report slot and coefficients of the current step (from
// the flags a previous launch left; the same in every block)
template <typename T>
struct StepCoef {
    int nhist, ord, slot;
    T c0, cl, k0, k1, samp;
};

template <typename T>
__device__ __forceinline__ StepCoef<T> step_coef_at(const Args<T>& a, int nhist, int slot) {
    StepCoef<T> k;
    // past levels available -> the order of this step (SBDF1 .. SBDF4, the
    // first steps of a run without history climb one order per step)
    k.nhist = nhist;
    k.ord = min(a.order, nhist + 1);
    k.slot = slot;
    // the SBDFk system scaled to integer coefficients:
    //   c0 u^{n+1} - cl delta L u^{n+1} = sum_j A_j u^{n-j} + cl sum_j B_j f^{n-j}
    // k = 1: c0 1, cl dt;  k = 2: 3, 2 dt;  k = 3: 11, 6 dt;  k = 4: 25, 12 dt
    const int ord = k.ord;
    k.c0 = ord == 1 ? T(1) : ord == 2 ? T(3) : ord == 3 ? T(11) : T(25);
    k.cl = (ord == 1 ? T(1) : ord == 2 ? T(2) : ord == 3 ? T(6) : T(12)) * a.dt;
    k.k0 = k.cl * a.delta[0];
    k.k1 = k.cl * a.delta[1];
    // the source is taken at the new time level t^{n+1} (implicitly)
    k.samp = (a.su || a.sv) ? (T)exp(a.src_rate * (*a.tstart + (double)(k.slot + 1) * (double)a.dt)) : T(0);
    return k;
}

template <typename T>
__device__ __forceinline__ StepCoef<T> step_coef(const Args<T>& a) {
    return step_coef_at(a, *((volatile int*)(a.flags + 2)), *((volatile int*)(a.flags + 3)));
}

// Dot-product accumulators.  Float64 sums are float64.  Float32 sums are carried in
// three float32 values by the dot product DotK with K = 3 (Ogita, Rump & Oishi, "Accurate sum and dot
// product", SIAM J. Sci. Comput. 26 (2005), Algorithm 5.10, the last level a plain
// sum): each product a b split exactly into p + e by an FMA (TwoProduct), sums by
// Knuth's error-free TwoSum, the errors of the second level added at the end.  The
// rounding error is about 2^-72 of the sum of |a b|, below that of a float64 sum,
// with float32 instructions only: the float64 unit takes a warp 64 clocks for an
// FMA (two species, 1M rows: 5.28 ms a step with float64 sums, 5.06 with these;
// 500k rows of n = 17: 986 and 902 us; pairs of float32 values, about 2^-48 and not
// scaled, took 5.06 ms and 892 us).
// TwoProduct is exact, and the sum finite, while the terms stay within float32's
// range, so the factors are scaled to about one by powers of two (exactly).
struct Dot3 {
    float h, m, l;
};
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float x = __fadd_rn(a, b), z = __fsub_rn(x, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(x, z)), __fsub_rn(b, z));
    return x;
}
__device__ __forceinline__ void acc_zero(Dot3& s) { s.h = s.m = s.l = 0.f; }
__device__ __forceinline__ void acc_zero(double& s) { s = 0.0; }
__device__ __forceinline__ void acc_pair(Dot3& s, float p, float e) {
    float t, u, w;
    s.h = two_sum(s.h, p, t);
    s.m = two_sum(s.m, e, u);
    s.m = two_sum(s.m, t, w);
    s.l = __fadd_rn(s.l, __fadd_rn(u, w));
}
__device__ __forceinline__ void acc_add(Dot3& s, float a, float b) {
    const float p = __fmul_rn(a, b);
    acc_pair(s, p, __fmaf_rn(a, b, -p));   // a b = p + e exactly
}
__device__ __forceinline__ void acc_add(double& s, double a, double b) { s += a * b; }

// the exponent by which values of about 2^e are scaled: 2^-e and its inverse are
// normal float32 numbers
__device__ __forceinline__ int unit_exp(int e) { return min(max(e, -126), 126); }
__device__ __forceinline__ float unit_scale(int e) { return __int_as_float((127 - e) << 23); }   // 2^-e

// The sum of a warp's values, in fixed point: each value is cut into three integers
// of 20 bits (by adding and subtracting 1.5 2^23), relative to the largest of them
// all, and integers are summed exactly by warp reductions.  What is cut off is below
// 2^-55 of the largest value, a float64 rounding's share.  (With a shuffle tree of
// Dot3 values 40k rows of n = 50, two species, took 84.5 us a step, with this 81.)
struct Fixed {
    long long n;   // value n 2^e
    int e;
};
__device__ __forceinline__ Fixed warp_sum(const Dot3& s, int e) {
    const float x[3] = {s.h, s.m, s.l};
    unsigned m = 0;   // largest magnitude (the bits order like integers)
#pragma unroll
    for (int i = 0; i < 3; ++i) m = max(m, __float_as_uint(x[i]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    const int E = max((int)(m >> 23) - 127, -110);
    const float S = __int_as_float((127 + 15 - E) << 23), R = 12582912.f;   // to below 2^16; 1.5 2^23
    int n[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float y = x[i], f = S;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float t = __fmaf_rn(y, f, R);
            n[q] += __float_as_int(t) - __float_as_int(R);
            y = __fmaf_rn(y, f, -__fsub_rn(t, R));   // exactly what is left
            f = 1048576.f;
        }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) n[q] = __reduce_add_sync(0xffffffffu, n[q]);
    Fixed r;
    r.n = ((long long)n[0] << 40) + ((long long)n[1] << 20) + n[2];
    r.e = m < 0x7f800000u ? e + E - 55 : INT_MAX;   // infinite or NaN
    return r;
}
__device__ __forceinline__ double fixed_value(const Fixed& f) {
    if (f.e == INT_MAX) return NAN;
    // n as a float64 (its halves placed in the mantissas of 2^84 and 2^52)
    const double x = (__hiloint2double(0x45300000, (int)(f.n >> 32) ^ (int)0x80000000) - 19342822341709703277445120.0) +
                     __hiloint2double(0x43300000, (int)f.n);
    return f.n == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + (f.e << 20), __double2loint(x));
}

// Squared norms of two vectors whose scale is not known yet: float32 threads scale
// by their largest element so far, and a warp agrees on one exponent at the end.
struct Norms64 {
    double b = 0.0, r = 0.0;
    __device__ void add(double x, double y) {
        acc_add(b, x, x);
        acc_add(r, y, y);
    }
    __device__ int finish(double& sb, double& sr) const {
        sb = b;
        sr = r;
        return 0;
    }
};
struct Norms32 {
    Dot3 b{0.f, 0.f, 0.f}, r{0.f, 0.f, 0.f};
    int e = -126;
    // |g| <= 1: the sums at another exponent (what underflows is far below them)
    __device__ static void rescale(Dot3& s, float g) {
        s.h *= g;
        s.m *= g;
        s.l *= g;
    }
    __device__ void to(int en) {
        const float g = en - e < 63 ? unit_scale(2 * (en - e)) : 0.f;
        rescale(b, g);
        rescale(r, g);
        e = en;
    }
    __device__ void add(float x, float y) {
        const unsigned m = max(__float_as_uint(x) & 0x7fffffffu, __float_as_uint(y) & 0x7fffffffu);
        const int en = unit_exp((int)(m >> 23) - 127);
        if (en > e + 8) to(en);
        const float f = unit_scale(e), xs = x * f, ys = y * f;
        acc_add(b, xs, xs);
        acc_add(r, ys, ys);
    }
    __device__ int finish(Dot3& sb, Dot3& sr) {
        to(__reduce_max_sync(0xffffffffu, e));
        sb = b;
        sr = r;
        return e;
    }
};

// the steps' accumulators for state type T, and their factors' scaling
template <typename T>
struct PhaseAcc {
    using type = double;
    using norms = Norms64;
    __device__ static double scaled(double x, float) { return x; }
    __device__ static int exp_of(double) { return 0; }
};
template <>
struct PhaseAcc<float> {
    using type = Dot3;
    using norms = Norms32;
    __device__ static float scaled(float x, float f) { return x * f; }
    // the exponent of a vector by its squared norm
    __device__ static int exp_of(double norm2) {
        return unit_exp((((__double2hiint(norm2) >> 20) & 0x7ff) - 1023) >> 1);
    }
};

// kinetics and right-hand side b of the step's SBDF order at node i (values
// ui, vi), and the rotation of its history
template <typename T>
__device__ __forceinline__ void rhs_values(const Args<T>& a, const StepCoef<T>& kc, int64_t i, T ui, T vi, T& bu,
                                           T& bv) {
    const bool two = a.ns == 2;
    const int ord = kc.ord;
    const T cl = kc.cl, samp = kc.samp;
    T f, g;
    react(a, ui, vi, f, g);
    bv = T(0);
    if (ord == 2) {
        bu = T(4) * ui - a.up[i] + T(2) * a.dt * (T(2) * f - a.fp[i]);
        if (two) bv = T(4) * vi - a.vp[i] + T(2) * a.dt * (T(2) * g - a.gp[i]);
    } else if (ord == 1) {
        bu = ui + a.dt * f;
        if (two) bv = vi + a.dt * g;
    } else if (ord == 3) {
        bu = (T(18) * ui - T(9) * a.up[i] + T(2) * a.up2[i]) +
             cl * (T(3) * f - T(3) * a.fp[i] + a.fp2[i]);
        if (two)
            bv = (T(18) * vi - T(9) * a.vp[i] + T(2) * a.vp2[i]) +
                 cl * (T(3) * g - T(3) * a.gp[i] + a.gp2[i]);
    } else {
        bu = (T(48) * ui - T(36) * a.up[i] + T(16) * a.up2[i] - T(3) * a.up3[i]) +
             cl * (T(4) * f - T(6) * a.fp[i] + T(4) * a.fp2[i] - a.fp3[i]);
        if (two)
            bv = (T(48) * vi - T(36) * a.vp[i] + T(16) * a.vp2[i] - T(3) * a.vp3[i]) +
                 cl * (T(4) * g - T(6) * a.gp[i] + T(4) * a.gp2[i] - a.gp3[i]);
    }
    if (a.su) bu += cl * samp * a.su[i];
    if (two && a.sv) bv += cl * samp * a.sv[i];
    // shift the history by one level (only the levels the order keeps)
    if (a.order >= 4) {
        a.up3[i] = a.up2[i];
        a.fp3[i] = a.fp2[i];
    }
    if (a.order >= 3) {
        a.up2[i] = a.up[i];
        a.fp2[i] = a.fp[i];
    }
    a.up[i] = ui;
    a.fp[i] = f;
    if (two) {
        if (a.order >= 4) {
            a.vp3[i] = a.vp2[i];
            a.gp3[i] = a.gp2[i];
        }
        if (a.order >= 3) {
            a.vp2[i] = a.vp[i];
            a.gp2[i] = a.gp[i];
        }
        a.vp[i] = vi;
        a.gp[i] = g;
    }
}

// phase R of one row (node i, with (L u)_i = Lu, (L v)_i = Lv): the right-hand
// side, r0 = b - A u, r-hat = r0, p = q = 0; accumulates |b|^2, |r0|^2 per
// species into d[0..1], d[2..3]
template <typename T>
__device__ __forceinline__ void rhs_row(const Args<T>& a, const StepCoef<T>& kc, int64_t i, T Lu, T Lv,
                                        typename PhaseAcc<T>::norms (&d)[2]) {
    const bool two = a.ns == 2;
    const T ui = a.u[i], vi = two ? a.v[i] : T(0);
    T bu, bv;
    rhs_values(a, kc, i, ui, vi, bu, bv);
    const T ru = bu - (kc.c0 * ui - kc.k0 * Lu);
    V(a, 0, VB)[i] = bu;
    V(a, 0, VR)[i] = ru;
    V(a, 0, VRH)[i] = ru;
    V(a, 0, VP)[i] = T(0);
    V(a, 0, VQ)[i] = T(0);
    d[0].add(bu, ru);
    if (two) {
        const T rv = bv - (kc.c0 * vi - kc.k1 * Lv);
        V(a, 1, VB)[i] = bv;
        V(a, 1, VR)[i] = rv;
        V(a, 1, VRH)[i] = rv;
        V(a, 1, VP)[i] = T(0);
        V(a, 1, VQ)[i] = T(0);
        d[1].add(bv, rv);
    }
}

// right-hand side b of a step that a direct solve follows, and its SBDF order
// for the solve (flags[4])
template <typename T>
__global__ void __launch_bounds__(256) lu_rhs_kernel(Args<T> a) {
    const StepCoef<T> kc = step_coef(a);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * blockDim.x) {
        T bu, bv;
        rhs_values(a, kc, i, a.u[i], a.ns == 2 ? a.v[i] : T(0), bu, bv);
        V(a, 0, VB)[i] = bu;
        if (a.ns == 2) V(a, 1, VB)[i] = bv;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[4] = kc.ord;
}

// report of a direct step (no iterations) and the next step's history and slot
template <typename T>
__global__ void lu_commit_kernel(Args<T> a) {
    const int nhist = a.flags[2], slot = a.flags[3];
    int* rp = a.rep + (int64_t)slot * 3;
    rp[0] = rp[1] = rp[2] = 0;
    a.rep_res[(int64_t)slot * 2] = 0.0;
    a.rep_res[(int64_t)slot * 2 + 1] = 0.0;
    a.flags[2] = min(nhist + 1, max(a.order - 1, 1));
    a.flags[3] = slot + 1;
}

// ---------------------------------------------------------------------------
// Phase-kernel BiCGSTAB for large operators, replayed from a CUDA graph: the
// right-hand side (R), then a device-side WHILE loop whose body is one
// BiCGSTAB iteration as five kernels (A: p; B: q = A p; C: s; D: t = A s;
// E: x, r), then the report (F).  Kernel boundaries make the vectors
// coherent, so the SpMV gathers go through L1 (neighbouring rows share most
// of their stencil nodes) and no grid barrier is needed.  Operators just above
// what the resident kernel holds run here too: against one cooperative launch
// with grid barriers and gathers through L2, 60k rows of n = 101 in float32
// took 408 us a step instead of 674, 100k of n = 50 468 instead of 599, 60k of
// n = 50 in float64 979 instead of 1303.  Reductions: block partials, then the
// phase's last block (by ticket) sums them in block order (deterministic)
// and sets the scalars the next phase reads; the last block of E commits
// the iteration and sets the loop condition.
// ---------------------------------------------------------------------------
constexpr int PT = 256;     // threads per block of the SpMV phase kernels (R, B, D)
constexpr int PT_MINB = 4;  // their resident blocks per SM (<= 64 registers a thread: no spills)
constexpr int PV = 256;    // threads per block of the vector phase kernels (A, C, E)
constexpr int PV_BPS = 4;   //   and their blocks per SM
constexpr int VG = 2;       // four-element groups a thread of phases A and C loads together

// (L x0)_r and (L x1)_r through L1 (x is not written by this kernel); the
// next chunk's index and weight loads go out before this chunk's gathers,
// so that a thread has two chunks of the matrix in flight, and with
// ROW_PF > 0 an L2 prefetch ROW_PF chunks ahead runs on into the thread's
// next row (rnext)
constexpr int ROW_PF = 2;

template <typename T, bool two>
__device__ __forceinline__ void row_L1(const Args<T>& a, int64_t r, int64_t rnext, const T* __restrict__ x0,
                                       const T* __restrict__ x1, T& y0, T& y1) {
    const int g = group_of_row(a.gi, r);
    const int npad = a.gi.npad[g], nch = npad >> 2;
    const int64_t base = ell_elem(a.gi.ell_off[g], npad, r - a.gi.row_begin[g], 0);
    int64_t nbase = -1;
    int nnch = 0;
    if (ROW_PF > 0 && rnext < a.N) {
        const int gn = group_of_row(a.gi, rnext);
        nnch = a.gi.npad[gn] >> 2;
        nbase = ell_elem(a.gi.ell_off[gn], a.gi.npad[gn], rnext - a.gi.row_begin[gn], 0);
    }
    T s0 = T(0), s1 = T(0);
    int4 iv = __ldcs(reinterpret_cast<const int4*>(a.idx + base));
    T wv[4];
    load4s(a.w + base, wv);
    for (int c = 0; c < nch; ++c) {
        if (ROW_PF > 0) {
            const int k = c + ROW_PF;
            int64_t e = -1;
            if (k < nch) e = base + (int64_t)k * 128;
            else if (k - nch < nnch && nbase >= 0) e = nbase + (int64_t)(k - nch) * 128;
            if (e >= 0) {
                prefetch_l2(a.idx + e);
                prefetch_l2(a.w + e);
            }
        }
        int4 ivn = iv;
        T wn[4] = {wv[0], wv[1], wv[2], wv[3]};
        if (c + 1 < nch) {
            const int64_t en = base + (int64_t)(c + 1) * 128;
            ivn = __ldcs(reinterpret_cast<const int4*>(a.idx + en));
            load4s(a.w + en, wn);
        }
        const int ii[4] = {iv.x, iv.y, iv.z, iv.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s0 = fma(wv[q], __ldg(x0 + ii[q]), s0);
            if (two) s1 = fma(wv[q], __ldg(x1 + ii[q]), s1);
        }
        iv = ivn;
#pragma unroll
        for (int q = 0; q < 4; ++q) wv[q] = wn[q];
    }
    y0 = s0;
    y1 = two ? s1 : T(0);
}

// the product of the species that still run (L0, L1; the other stays unset): a
// second species' gathers, and the branch around them, only where both run
// (one species in float64, 300k rows, n = 50: 946 -> 692 us a step)
template <typename T>
__device__ __forceinline__ void row_species(const Args<T>& a, int64_t r, int64_t rnext, const T* x0, const T* x1, bool on0,
                                            bool on1, T& L0, T& L1) {
    if (on0 && on1) {
        row_L1<T, true>(a, r, rnext, x0, x1, L0, L1);
    } else {
        T y, none;
        const T* x = on0 ? x0 : x1;
        row_L1<T, false>(a, r, rnext, x, x, y, none);
        L0 = L1 = y;
    }
}

// K sums per block into pp[block][0..K-1]; the last block of the grid sums
// them in a fixed order and returns the totals (in shared memory; NULL in the
// other blocks).  Only one warp per sum does float64 arithmetic: one float64
// warp instruction takes the SM 16 clocks, and a float64 shuffle tree in every
// warp cost the vector phases more than their memory traffic (two species,
// float32, 1M rows: 5.63 -> 5.06 ms a step).  exp_of(k): the exponent of float32
// sum k (warp_sum).
template <int K, int NTB, typename A, typename F>
__device__ const double* phase_reduce(const A (&v)[K], double* pp, unsigned int* ticket, F exp_of) {
    using F32 = std::is_same<A, Dot3>;
    constexpr int NW = NTB / 32;
    using Shared = typename std::conditional<F32::value, Fixed, double>::type;
    __shared__ Shared sh[K][F32::value ? NW : NTB];
    __shared__ double tot[K];
    __shared__ int last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    static_assert(K <= NW && NW <= 32, "a warp per sum");
    double t = 0.0;
    if constexpr (F32::value) {   // a warp's sum in fixed point, then one warp per sum over the warps
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const Fixed x = warp_sum(v[k], exp_of(k));
            if (lane == 0) sh[k][wid] = x;
        }
        __syncthreads();
        if (wid < K) {
            if (lane < NW) t = fixed_value(sh[wid][lane]);
#pragma unroll
            for (int o = NW / 2; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        }
    } else {                      // float64: one warp per sum over the threads' values
#pragma unroll
        for (int k = 0; k < K; ++k) sh[k][threadIdx.x] = v[k];
        __syncthreads();
        if (wid < K) {
            t = sh[wid][lane];
#pragma unroll
            for (int w = 1; w < NW; ++w) t += sh[wid][w * 32 + lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        }
    }
    if (wid < K && lane == 0) {
        pp[(int64_t)blockIdx.x * 8 + wid] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return nullptr;
    __threadfence();
    // lane t of warp k sums blocks t, t + 32, ..., four loads in flight; then a fixed tree
    if (wid < K) {
        double s = 0.0;
        for (int64_t b0 = lane; b0 < gridDim.x; b0 += 128) {
            double x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = b0 + 32 * u < gridDim.x ? __ldcg(pp + (b0 + 32 * u) * 8 + wid) : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u) s += x[u];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) tot[wid] = s;
    }
    if (threadIdx.x == 0) *ticket = 0u;
    __syncthreads();
    return tot;
}

// the loop continues while a species runs
template <typename T>
__device__ __forceinline__ void set_more(const Args<T>& a, int more) {
    if (threadIdx.x == 0) {
        a.ctl->more = more;
        if (a.cond) cudaGraphSetConditional(a.cond, (unsigned)more);
        if (a.more_host) *(volatile int*)a.more_host = 2 * a.more_seq + more;
    }
}

// beta and the A-decision of the next iteration, from the committed state
__device__ __forceinline__ void next_iteration(SpeciesState& z) {
    z.beta = (z.rho / z.rho_prev) * (z.alpha / z.omega);
    z.actA = z.active && !(z.rho == 0.0 || !isfinite(z.beta));
    z.actB = z.early = z.actE = 0;
}

// R: right-hand side and r0
template <typename T>
__global__ void __launch_bounds__(PT, PT_MINB) phase_R(Args<T> a) {
    const StepCoef<T> kc = step_coef(a);
    const bool two = a.ns == 2;
    typename PhaseAcc<T>::norms d[2];
    for (int64_t r = blockIdx.x * (int64_t)PT + threadIdx.x; r < a.N; r += (int64_t)gridDim.x * PT) {
        const int64_t i = a.row_node[r];
        T Lu, Lv;
        row_species(a, r, r + (int64_t)gridDim.x * PT, (const T*)a.u, (const T*)a.v, true, two, Lu, Lv);
        rhs_row(a, kc, i, Lu, Lv, d);
    }
    PhaseCtl* c = a.ctl;
    typename PhaseAcc<T>::type v[4];
    int e[2];
    for (int k = 0; k < 2; ++k) e[k] = d[k].finish(v[2 * k], v[2 * k + 1]);
    const double* tot = phase_reduce<4, PT>(v, a.pp, &c->ticket, [&](int j) { return 2 * e[j >> 1]; });
    if (tot && threadIdx.x < 2) {
        const int k = threadIdx.x;
        const bool exists = k == 0 || two;
        SpeciesState z;
        z.bnorm = sqrt(tot[2 * k]);
        z.limit2 = (a.tol * z.bnorm) * (a.tol * z.bnorm);
        z.rho = z.res2 = tot[2 * k + 1];   // (r-hat, r0) = |r0|^2
        z.rho_prev = z.rho;   // beta = 1 (p = q = 0: any finite value)
        z.alpha = z.omega = 1.0;
        z.alpha_n = z.omega_n = 0.0;
        z.e0 = z.e = PhaseAcc<T>::exp_of(z.rho);
        z.active = exists && z.bnorm != 0.0 && !(sqrt(z.res2) / z.bnorm <= a.tol);
        z.fail = z.iters = 0;
        z.zero = exists && z.bnorm == 0.0;   // b = 0: x = 0
        next_iteration(z);
        c->s[k] = z;
        c->it = 0;
        const unsigned m = __ballot_sync(3u, z.active);
        set_more(a, m != 0 && a.maxit > 0);
    }
}

// The vector phases move groups of four consecutive elements with 16-byte
// loads and stores (every internal vector starts on a 16-byte boundary; the
// state u, v when the caller's are aligned, else a plain element loop): a
// quarter of the memory instructions and of the index arithmetic of an
// element loop, whose instruction count bounded them.  A thread visits
// groups g0, g0 + S, ... (S = the grid's threads), VG at a time with all
// their loads issued first; the last N mod 4 elements go element by
// element.  The dot products are summed per thread in that order.

__device__ __forceinline__ void ld4v(const float* p, float (&w)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
__device__ __forceinline__ void ld4v(const double* p, double (&w)[4]) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
}
__device__ __forceinline__ void st4v(float* p, const float (&w)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void st4v(double* p, const double (&w)[4]) {
    *reinterpret_cast<double2*>(p) = make_double2(w[0], w[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(w[2], w[3]);
}

// A: p = r + beta (p - omega q)
template <typename T>
__global__ void __launch_bounds__(PV, PV_BPS) phase_A(Args<T> a) {
    const PhaseCtl* c = a.ctl;
    if (!c->more) return;   // (an iteration the host loop launched ahead)
    const int64_t S = (int64_t)gridDim.x * PV, t0 = blockIdx.x * (int64_t)PV + threadIdx.x;
    for (int k = 0; k < a.ns; ++k) {
        if (!c->s[k].actA) continue;
        const T beta = (T)c->s[k].beta, omega = (T)c->s[k].omega;
        T* __restrict__ p = V(a, k, VP);
        const T* __restrict__ r = V(a, k, VR);
        const T* __restrict__ q = V(a, k, VQ);
        int64_t i = t0;
        if (a.vec4) {
            const int64_t G = a.N >> 2;
            for (int64_t g0 = t0; g0 < G; g0 += VG * S) {
                T rv[VG][4], pv[VG][4], qv[VG][4];
#pragma unroll
                for (int u = 0; u < VG; ++u)
                    if (g0 + u * S < G) {
                        const int64_t e = 4 * (g0 + u * S);
                        ld4v(r + e, rv[u]);
                        ld4v(p + e, pv[u]);
                        ld4v(q + e, qv[u]);
                    }
#pragma unroll
                for (int u = 0; u < VG; ++u)
                    if (g0 + u * S < G) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) pv[u][j] = rv[u][j] + beta * (pv[u][j] - omega * qv[u][j]);
                        st4v(p + 4 * (g0 + u * S), pv[u]);
                    }
            }
            i = 4 * G + t0;
        }
        for (; i < a.N; i += S) p[i] = r[i] + beta * (p[i] - omega * q[i]);
    }
}

// B: q = A p ; (r-hat, q).  With B_BACK it visits the rows from the last
// 32-row slice to the first (lanes keep their order within a slice): R and D
// run forward, so every pass over the matrix starts on the rows the pass
// before it ended on, which are still in L2.
constexpr bool B_BACK = true;

__device__ __forceinline__ int64_t back_row(int64_t k, int64_t Np) { return Np - 32 - (k & ~(int64_t)31) + (k & 31); }

template <typename T>
__global__ void __launch_bounds__(PT, PT_MINB) phase_B(Args<T> a) {
    PhaseCtl* c = a.ctl;
    if (!c->more) return;   // (an iteration the host loop launched ahead)
    const bool a0 = c->s[0].actA, a1 = a.ns == 2 && c->s[1].actA;
    const StepCoef<T> kc = step_coef(a);
    using PA = PhaseAcc<T>;
    typename PA::type d[2];
    for (auto& x : d) acc_zero(x);
    const int e0[2] = {c->s[0].e0, c->s[1].e0}, e[2] = {c->s[0].e, c->s[1].e};
    const float f0[2] = {unit_scale(e0[0]), unit_scale(e0[1])}, f[2] = {unit_scale(e[0]), unit_scale(e[1])};
    const int64_t S = (int64_t)gridDim.x * PT, Np = (a.N + 31) & ~(int64_t)31;
    for (int64_t k = blockIdx.x * (int64_t)PT + threadIdx.x; (a0 || a1) && k < Np; k += S) {
        const int64_t r = B_BACK ? back_row(k, Np) : k;
        if (r >= a.N) continue;
        const int64_t rn = k + S >= Np ? a.N : (B_BACK ? back_row(k + S, Np) : k + S);
        const int64_t i = a.row_node[r];
        T L0, L1;
        row_species(a, r, rn, (const T*)V(a, 0, VP), (const T*)V(a, 1, VP), a0, a1, L0, L1);
        if (a0) {
            const T q = kc.c0 * V(a, 0, VP)[i] - kc.k0 * L0;
            V(a, 0, VQ)[i] = q;
            acc_add(d[0], PA::scaled(V(a, 0, VRH)[i], f0[0]), PA::scaled(q, f[0]));
        }
        if (a1) {
            const T q = kc.c0 * V(a, 1, VP)[i] - kc.k1 * L1;
            V(a, 1, VQ)[i] = q;
            acc_add(d[1], PA::scaled(V(a, 1, VRH)[i], f0[1]), PA::scaled(q, f[1]));
        }
    }
    const double* tot = phase_reduce<2, PT>(d, a.pp, &c->ticket, [&](int k) { return e0[k] + e[k]; });
    if (tot && threadIdx.x < 2) {
        const int k = threadIdx.x;
        SpeciesState& z = c->s[k];
        const int act = z.actA;
        const double alpha = act ? z.rho / tot[k] : 0.0;
        z.alpha_n = alpha;
        z.actB = act && !(tot[k] == 0.0 || !isfinite(alpha));
    }
}

// C: s = r - alpha q ; |s|^2
template <typename T>
__global__ void __launch_bounds__(PV, PV_BPS) phase_C(Args<T> a) {
    PhaseCtl* c = a.ctl;
    if (!c->more) return;   // (an iteration the host loop launched ahead)
    using PA = PhaseAcc<T>;
    typename PA::type d[2];
    for (auto& x : d) acc_zero(x);
    const int64_t S = (int64_t)gridDim.x * PV, t0 = blockIdx.x * (int64_t)PV + threadIdx.x;
    const int e[2] = {c->s[0].e, c->s[1].e};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (k >= a.ns || !c->s[k].actB) continue;
        const T alpha = (T)c->s[k].alpha_n;
        const float f = unit_scale(e[k]);
        const T* __restrict__ r = V(a, k, VR);
        const T* __restrict__ q = V(a, k, VQ);
        T* __restrict__ sv = V(a, k, VS);
        int64_t i = t0;
        if (a.vec4) {
            const int64_t G = a.N >> 2;
            for (int64_t g0 = t0; g0 < G; g0 += VG * S) {
                T rv[VG][4], qv[VG][4];
#pragma unroll
                for (int u = 0; u < VG; ++u)
                    if (g0 + u * S < G) {
                        const int64_t i4 = 4 * (g0 + u * S);
                        ld4v(r + i4, rv[u]);
                        ld4v(q + i4, qv[u]);
                    }
#pragma unroll
                for (int u = 0; u < VG; ++u)
                    if (g0 + u * S < G) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            rv[u][j] = rv[u][j] - alpha * qv[u][j];
                            const T y = PA::scaled(rv[u][j], f);
                            acc_add(d[k], y, y);
                        }
                        st4v(sv + 4 * (g0 + u * S), rv[u]);
                    }
            }
            i = 4 * G + t0;
        }
        for (; i < a.N; i += S) {
            const T x = r[i] - alpha * q[i];
            sv[i] = x;
            acc_add(d[k], PA::scaled(x, f), PA::scaled(x, f));
        }
    }
    const double* tot = phase_reduce<2, PV>(d, a.pp, &c->ticket, [&](int k) { return 2 * e[k]; });
    if (tot && threadIdx.x < 2) {
        SpeciesState& z = c->s[threadIdx.x];
        const int early = z.actB && tot[threadIdx.x] <= z.limit2;
        z.early = early;
        if (early) z.res2 = tot[threadIdx.x];
    }
}

// D: t = A s ; (t, s), (t, t)   (x += alpha p where s already converged)
template <typename T>
__global__ void __launch_bounds__(PT, PT_MINB) phase_D(Args<T> a) {
    PhaseCtl* c = a.ctl;
    if (!c->more) return;   // (an iteration the host loop launched ahead)
    const StepCoef<T> kc = step_coef(a);
    const bool two = a.ns == 2;
    const bool e0 = c->s[0].early, e1 = two && c->s[1].early;
    const bool b0 = c->s[0].actB, b1 = two && c->s[1].actB;
    const bool need0 = b0 && !e0, need1 = b1 && !e1;
    using PA = PhaseAcc<T>;
    typename PA::type d[4];
    for (auto& x : d) acc_zero(x);
    const int e[2] = {c->s[0].e, c->s[1].e};
    const float f[2] = {unit_scale(e[0]), unit_scale(e[1])};
    for (int64_t r = blockIdx.x * (int64_t)PT + threadIdx.x; (b0 || b1) && r < a.N; r += (int64_t)gridDim.x * PT) {
        const int64_t i = a.row_node[r];
        T L0 = T(0), L1 = T(0);
        if (need0 || need1)
            row_species(a, r, r + (int64_t)gridDim.x * PT, (const T*)V(a, 0, VS), (const T*)V(a, 1, VS), need0, need1, L0,
                        L1);
#pragma unroll
        for (int k = 0; k < 2; ++k) {   // (e1 and b1 only with two species)
            T* x = k == 0 ? a.u : a.v;
            if (k == 0 ? e0 : e1) {
                x[i] += (T)c->s[k].alpha_n * V(a, k, VP)[i];
            } else if (k == 0 ? b0 : b1) {
                const T sv = V(a, k, VS)[i];
                const T t = kc.c0 * sv - (k == 0 ? kc.k0 * L0 : kc.k1 * L1);
                V(a, k, VT)[i] = t;
                const T ts = PA::scaled(t, f[k]);
                acc_add(d[2 * k], ts, PA::scaled(sv, f[k]));
                acc_add(d[2 * k + 1], ts, ts);
            }
        }
    }
    const double* tot = phase_reduce<4, PT>(d, a.pp, &c->ticket, [&](int j) { return 2 * e[j >> 1]; });
    if (tot && threadIdx.x < 2) {
        const int k = threadIdx.x;
        SpeciesState& z = c->s[k];
        const int act = z.actB && !z.early;
        const double omega = tot[2 * k] / tot[2 * k + 1];
        z.omega_n = omega;
        z.actE = act && !(tot[2 * k + 1] == 0.0 || !isfinite(omega));
    }
}

// E: x += alpha p + omega s ; r = s - omega t ; (r-hat, r), |r|^2; the last
// block commits the iteration and decides whether the loop continues
template <typename T>
__device__ __forceinline__ void e_update(T alpha, T omega, T& x, T p, T s, T t, T& r) {
    x = x + (alpha * p + omega * s);
    r = s - omega * t;
}

template <typename T>
__global__ void __launch_bounds__(PV, PV_BPS) phase_E(Args<T> a) {
    PhaseCtl* c = a.ctl;
    if (!c->more) return;   // (an iteration the host loop launched ahead)
    using PA = PhaseAcc<T>;
    typename PA::type d[4];
    for (auto& x : d) acc_zero(x);
    const int64_t S = (int64_t)gridDim.x * PV, t0 = blockIdx.x * (int64_t)PV + threadIdx.x;
    const int e0[2] = {c->s[0].e0, c->s[1].e0}, e[2] = {c->s[0].e, c->s[1].e};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (k >= a.ns || !c->s[k].actE) continue;
        const T alpha = (T)c->s[k].alpha_n, omega = (T)c->s[k].omega_n;
        const float f0 = unit_scale(e0[k]), f = unit_scale(e[k]);
        T* __restrict__ x = k == 0 ? a.u : a.v;
        const T* __restrict__ p = V(a, k, VP);
        const T* __restrict__ sv = V(a, k, VS);
        const T* __restrict__ t = V(a, k, VT);
        const T* __restrict__ rh = V(a, k, VRH);
        T* __restrict__ r = V(a, k, VR);
        int64_t i = t0;
        if (a.vec4) {
            const int64_t G = a.N >> 2;
            for (int64_t g = t0; g < G; g += S) {
                const int64_t i4 = 4 * g;
                T xv[4], pv[4], s_[4], tv[4], hv[4], rn[4];
                ld4v(x + i4, xv);
                ld4v(p + i4, pv);
                ld4v(sv + i4, s_);
                ld4v(t + i4, tv);
                ld4v(rh + i4, hv);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    e_update(alpha, omega, xv[j], pv[j], s_[j], tv[j], rn[j]);
                    const T y = PA::scaled(rn[j], f);
                    acc_add(d[2 * k], PA::scaled(hv[j], f0), y);
                    acc_add(d[2 * k + 1], y, y);
                }
                st4v(x + i4, xv);
                st4v(r + i4, rn);
            }
            i = 4 * G + t0;
        }
        for (; i < a.N; i += S) {
            T xi = x[i], rn;
            e_update(alpha, omega, xi, p[i], sv[i], t[i], rn);
            x[i] = xi;
            r[i] = rn;
            const T y = PA::scaled(rn, f);
            acc_add(d[2 * k], PA::scaled(rh[i], f0), y);
            acc_add(d[2 * k + 1], y, y);
        }
    }
    const double* tot =
        phase_reduce<4, PV>(d, a.pp, &c->ticket, [&](int j) { return (j & 1 ? e[j >> 1] : e0[j >> 1]) + e[j >> 1]; });
    if (tot && threadIdx.x < 2) {
        const int k = threadIdx.x, it = c->it + 1;
        SpeciesState z = c->s[k];
        if (z.active) {
            if (!z.actA || !z.actB || (!z.early && !z.actE)) {
                z.fail = 1;
                z.active = 0;
            } else if (z.early) {
                z.active = 0;
                z.iters = it;
            } else {
                z.rho_prev = z.rho;
                z.rho = tot[2 * k];
                z.alpha = z.alpha_n;
                z.omega = z.omega_n;
                z.res2 = tot[2 * k + 1];
                z.e = PA::exp_of(z.res2);
                if (z.res2 <= z.limit2) {
                    z.active = 0;
                    z.iters = it;
                } else if (z.omega_n == 0.0) {
                    z.fail = 1;
                    z.active = 0;
                }
            }
        }
        next_iteration(z);
        const unsigned m = __ballot_sync(3u, z.active);   // both lanes have read c->it
        c->s[k] = z;
        c->it = it;
        set_more(a, m != 0 && it < a.maxit);
    }
}

// F: report of the step, history flags, x = 0 where b = 0
template <typename T>
__global__ void __launch_bounds__(PT) phase_F(Args<T> a) {
    const PhaseCtl* c = a.ctl;
    for (int k = 0; k < a.ns; ++k) {
        if (!c->s[k].zero) continue;
        T* x = k == 0 ? a.u : a.v;
        for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * PT) x[i] = T(0);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const StepCoef<T> kc = step_coef(a);
        int* rp = a.rep + (int64_t)kc.slot * 3;
        bool bad = false;
        for (int k = 0; k < 2; ++k) {
            const SpeciesState& z = c->s[k];
            bad = bad || z.active || z.fail;   // still active: hit maxit
            rp[k] = z.active ? c->it : z.iters;
            a.rep_res[(int64_t)kc.slot * 2 + k] = z.bnorm > 0 ? sqrt(z.res2) / z.bnorm : 0.0;
        }
        rp[2] = bad ? 1 : 0;
        if (bad) atomicExch(a.flags + 1, 1);
        a.flags[2] = min(kc.nhist + 1, max(a.order - 1, 1));
        a.flags[3] = kc.slot + 1;
        a.flags[4] = kc.ord;
    }
}

#include "step_resident.cuh"

__global__ void lonely_barrier(unsigned long long* bar, int* err) {
    // a second arrival never comes: the bounded wait must give up
    grid_sync(bar, 2ull * gridDim.x, err);
}

template <typename T>
void fill_args(Args<T>& a, rbffd_op* op, rbffd_state* s, const rbffd_step_params* p, rbffd_step_ws* ws) {
    a.idx = op->idx;
    a.w = std::is_same<T, float>::value ? (const T*)op->w32 : (const T*)op->w64;
    a.row_node = op->row_node;
    a.gi = op->gi;
    a.N = op->N;
    a.u = (T*)s->u;
    a.v = (T*)s->v;
    a.up = (T*)s->u_prev;
    a.vp = (T*)s->v_prev;
    a.fp = (T*)s->f_prev;
    a.gp = (T*)s->g_prev;
    a.up2 = (T*)s->u_prev2;
    a.vp2 = (T*)s->v_prev2;
    a.fp2 = (T*)s->f_prev2;
    a.gp2 = (T*)s->g_prev2;
    a.up3 = (T*)s->u_prev3;
    a.vp3 = (T*)s->v_prev3;
    a.fp3 = (T*)s->f_prev3;
    a.gp3 = (T*)s->g_prev3;
    a.order = p->order == 0 ? 2 : p->order;
    a.su = (const T*)p->source_u;
    a.sv = p->nspecies == 2 ? (const T*)p->source_v : nullptr;
    a.src_rate = p->source_rate;
    a.tstart = ws->tstart;
    a.vec = (T*)ws->vec;
    a.ldv = (op->N + 3) & ~(int64_t)3;
    a.vec4 = ((uintptr_t)s->u % 16 == 0 && (p->nspecies == 1 || (uintptr_t)s->v % 16 == 0)) ? 1 : 0;
    a.ns = p->nspecies;
    a.model = p->model;
    for (int i = 0; i < 8; ++i) a.c[i] = (T)p->coef[i];
    a.dt = (T)p->dt;
    a.delta[0] = (T)p->delta_u;
    a.delta[1] = (T)p->delta_v;
    a.tol = p->tol;
    a.maxit = p->maxit;
    a.bar = ws->bar;
    a.flags = ws->flags;
    a.rep = ws->rep;
    a.rep_res = ws->rep_res;
    a.ctl = ws->ctl;
    a.pp = ws->pp;
    a.cond = 0;
}

// one step by the cached LU factors: (c0 I - cl delta L) x = b, the factors of
// the step's order (read on the device from flags[4]); x overwrites u, v
template <typename T>
rbffd_status launch_lu_step(Args<T>& a, rbffd_step_ws* ws, cudaStream_t st) {
    lu_rhs_kernel<T><<<(unsigned)std::min<int64_t>((a.N + 255) / 256, (int64_t)sm_count() * 8), 256, 0, st>>>(a);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    const void* b[2] = {V(a, 0, VB), a.ns == 2 ? V(a, 1, VB) : nullptr};
    void* x[2] = {a.u, a.ns == 2 ? a.v : nullptr};
    rbffd_status r = lu_solve_step(ws->lu, a.ns, b, x, std::is_same<T, float>::value ? RBFFD_F32 : RBFFD_F64,
                                   ws->flags + 4, ws->ywork, ws->flags, st);
    if (r != RBFFD_OK) return r;
    lu_commit_kernel<T><<<1, 1, 0, st>>>(a);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    return RBFFD_OK;
}

// resident-sized grids, grid-stride loops: the SpMV phases PT_MINB blocks
// of PT threads per SM (their register bound makes exactly that many fit:
// one wave, no partial second one), the vector phases one block of PV
// threads per SM.  (A grid of one thread per row or element ran slower:
// the per-block reduction and ticket then cost more than a block's work.)
// The per-block partials (pp) hold ceil(N / PT) blocks, more than either grid.
template <typename T>
void phase_grids(const Args<T>& a, unsigned* g_rows, unsigned* g_vec) {
    *g_rows = (unsigned)std::max<int64_t>(1, std::min<int64_t>((a.N + PT - 1) / PT, (int64_t)sm_count() * PT_MINB));
    *g_vec = (unsigned)std::max<int64_t>(1, std::min<int64_t>((a.N + PV - 1) / PV, (int64_t)sm_count() * PV_BPS));
}

// One step of the phase-kernel path from the host (no graph): R, then the
// iterations while the loop state says so, then F -- the same kernels and
// arithmetic as the graph.  R and E write into pinned host memory whether the loop
// goes on, and an iteration is launched before its predecessor has done so (it does
// nothing if the loop is over): with a copy and a wait between iterations the GPU
// idled for longer than the phases of thin rows take (one species in float64, n = 7,
// 120k rows: 331 us a step, so 283; replayed 226; one cooperative launch a step 313).
template <typename T>
rbffd_status phased_step_host(Args<T> a, rbffd_step_ws* ws, cudaStream_t st) {
    unsigned gr, gv;
    phase_grids(a, &gr, &gv);
    a.cond = 0;
    if (!ws->more_host) {
        RBFFD_CUDA_TRY(cudaMallocHost(&ws->more_host, sizeof(int)));
        *ws->more_host = 0;
    }
    a.more_host = ws->more_host;
    auto next = [&] { a.more_seq = ws->more_seq = (ws->more_seq + 1) & 0x3fffffff; };
    // what phase `seq` said; a later word means that it said yes
    auto goes_on = [&](int seq, bool* more) -> rbffd_status {
        for (int64_t polls = 1;; ++polls) {
            const int word = *(volatile int*)ws->more_host;
            if (((word >> 1) - seq & 0x3fffffff) < 0x20000000) {
                *more = (word >> 1) != seq || (word & 1);
                return RBFFD_OK;
            }
            if (polls % 4096 == 0) {   // the stream drained or failed without a word
                const cudaError_t e = cudaStreamQuery(st);
                if (e == cudaErrorNotReady) continue;
                RBFFD_CUDA_TRY(e);
                if (((*(volatile int*)ws->more_host >> 1) - seq & 0x3fffffff) < 0x20000000) continue;
                set_error("the steps' loop state did not arrive");
                return RBFFD_ECUDA;
            }
        }
    };
    next();
    phase_R<T><<<gr, PT, 0, st>>>(a);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    for (bool more = true; more;) {
        const int seq = a.more_seq;
        next();
        phase_A<T><<<gv, PV, 0, st>>>(a);
        phase_B<T><<<gr, PT, 0, st>>>(a);
        phase_C<T><<<gv, PV, 0, st>>>(a);
        phase_D<T><<<gr, PT, 0, st>>>(a);
        phase_E<T><<<gv, PV, 0, st>>>(a);
        note_launch(5);
        RBFFD_CUDA_TRY(cudaGetLastError());
        RBFFD_TRY(goes_on(seq, &more));
    }
    phase_F<T><<<gr, PT, 0, st>>>(a);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    return RBFFD_OK;
}

// The step as a graph: R -> WHILE (condition set on the device) { A B C D E } -> F
template <typename T>
rbffd_status build_phase_graph(Args<T> a, cudaGraphExec_t* out) {
    unsigned gr, gv;
    phase_grids(a, &gr, &gv);
    cudaGraph_t g = nullptr;
    RBFFD_CUDA_TRY(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h;
    cudaError_t e = cudaGraphConditionalHandleCreate(&h, g, 0, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g);
        RBFFD_CUDA_TRY(e);
    }
    a.cond = h;
    void* args[] = {&a};
    auto kernel = [&](cudaGraph_t graph, const void* fn, bool vec, cudaGraphNode_t* dep, cudaGraphNode_t* node) {
        cudaKernelNodeParams kp;
        memset(&kp, 0, sizeof(kp));
        kp.func = const_cast<void*>(fn);
        kp.gridDim = dim3(vec ? gv : gr);
        kp.blockDim = dim3(vec ? PV : PT);
        kp.kernelParams = args;
        return cudaGraphAddKernelNode(node, graph, dep, dep ? 1 : 0, &kp);
    };
    cudaGraphNode_t nR, nW, nF;
    e = kernel(g, (const void*)phase_R<T>, false, nullptr, &nR);
    // (the parameter union has no default constructor: zeroed raw storage)
    alignas(cudaGraphNodeParams) unsigned char cp_raw[sizeof(cudaGraphNodeParams)];
    memset(cp_raw, 0, sizeof(cp_raw));
    cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(cp_raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    if (e == cudaSuccess) e = cudaGraphAddNode(&nW, g, &nR, nullptr, 1, &cp);
    if (e == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        cudaGraphNode_t n1, n2, n3, n4, n5;
        e = kernel(body, (const void*)phase_A<T>, true, nullptr, &n1);
        if (e == cudaSuccess) e = kernel(body, (const void*)phase_B<T>, false, &n1, &n2);
        if (e == cudaSuccess) e = kernel(body, (const void*)phase_C<T>, true, &n2, &n3);
        if (e == cudaSuccess) e = kernel(body, (const void*)phase_D<T>, false, &n3, &n4);
        if (e == cudaSuccess) e = kernel(body, (const void*)phase_E<T>, true, &n4, &n5);
    }
    if (e == cudaSuccess) e = kernel(g, (const void*)phase_F<T>, false, &nW, &nF);
    if (e == cudaSuccess) e = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    RBFFD_CUDA_TRY(e);
    return RBFFD_OK;
}

// nsteps launches, directly or by replaying one captured graph of a step
template <typename T>
rbffd_status run_steps(Args<T>& a, rbffd_step_ws* ws, int64_t nsteps, bool use_graph, bool lu, int nhist,
                       bool* phased, cudaStream_t st) {
    static_assert(sizeof(Args<T>) <= sizeof(ws->graph_args), "graph key too small");
    if (!lu && nsteps > 0) {
        // operators that fit the chip's shared memory: one launch for all steps
        ResidentPlan& plan = ws->plan[a.ns - 1];
        if (!ws->planned[a.ns - 1]) {
            plan = resident_plan<T>(a.gi, a.N, a.ns, sm_count(),
                                    [&](const ResidentPlan& p) { return cluster_resides<T>(p, a.ns); });
            ws->planned[a.ns - 1] = true;
        }
        if (plan.blocks > 0)
            return resident_launch(a, plan, nhist, nsteps, ws->vec, ws->rpart, st);
    }
    if (!lu) {
        *phased = true;
        if (!use_graph) {
            for (int64_t k = 0; k < nsteps; ++k) {
                rbffd_status r = phased_step_host(a, ws, st);
                if (r != RBFFD_OK) return r;
            }
            return RBFFD_OK;
        }
        a.cond = 0;   // the graph key holds the arguments without the handle
        if (!ws->graph || ws->graph_args_size != sizeof(a) || memcmp(ws->graph_args, &a, sizeof(a)) != 0 ||
            ws->solver != 2) {
            if (ws->graph) {
                cudaGraphExecDestroy(ws->graph);
                ws->graph = nullptr;
            }
            rbffd_status r = build_phase_graph(a, &ws->graph);
            if (r != RBFFD_OK) return r;
            memcpy(ws->graph_args, &a, sizeof(a));
            ws->graph_args_size = sizeof(a);
            ws->solver = 2;
        }
        for (int64_t k = 0; k < nsteps; ++k) {
            RBFFD_CUDA_TRY(cudaGraphLaunch(ws->graph, st));
            note_launch(2);   // R and F; the loop body's five per iteration are counted from the report
        }
        return RBFFD_OK;
    }
    if (!use_graph) {
        for (int64_t k = 0; k < nsteps; ++k) {
            rbffd_status r = launch_lu_step(a, ws, st);
            if (r != RBFFD_OK) return r;
        }
        return RBFFD_OK;
    }
    // the graph holds the kernels' arguments, the LU solve's factor pointers
    // included: any change recaptures it
    if (!ws->graph || ws->graph_args_size != sizeof(a) || memcmp(ws->graph_args, &a, sizeof(a)) != 0 ||
        ws->solver != 1 || memcmp(ws->graph_lu, ws->lu, sizeof(ws->lu)) != 0) {
        if (ws->graph) {
            cudaGraphExecDestroy(ws->graph);
            ws->graph = nullptr;
        }
        // capture on a private stream (the caller's may be the legacy default
        // stream, which cannot be captured); replay on the caller's stream
        if (!ws->cap) RBFFD_CUDA_TRY(cudaStreamCreateWithFlags(&ws->cap, cudaStreamNonBlocking));
        cudaGraph_t g = nullptr;
        RBFFD_CUDA_TRY(cudaStreamBeginCapture(ws->cap, cudaStreamCaptureModeThreadLocal));
        rbffd_status r = launch_lu_step(a, ws, ws->cap);
        cudaError_t e = cudaStreamEndCapture(ws->cap, &g);
        if (r != RBFFD_OK) return r;
        RBFFD_CUDA_TRY(e);
        e = cudaGraphInstantiate(&ws->graph, g, 0);
        cudaGraphDestroy(g);
        RBFFD_CUDA_TRY(e);
        memcpy(ws->graph_args, &a, sizeof(a));
        ws->graph_args_size = sizeof(a);
        ws->solver = 1;
        memcpy(ws->graph_lu, ws->lu, sizeof(ws->lu));
    }
    for (int64_t k = 0; k < nsteps; ++k) {
        RBFFD_CUDA_TRY(cudaGraphLaunch(ws->graph, st));
        note_launch(3);   // right-hand side, solve, commit
    }
    return RBFFD_OK;
}

}  // namespace
}  // namespace rbffd

using namespace rbffd;

extern "C" rbffd_status rbffd_step_imex(rbffd_op* op, rbffd_state* s, const rbffd_step_params* p,
                                        int64_t nsteps, void* stream, rbffd_step_report* report) {
    RBFFD_CHECK_ARG(op && s && p, "NULL argument");
    RBFFD_CHECK_ARG(p->dtype == RBFFD_F32 || p->dtype == RBFFD_F64, "dtype");
    RBFFD_CHECK_ARG(p->nspecies == 1 || p->nspecies == 2, "nspecies must be 1 or 2");
    RBFFD_CHECK_ARG(s->u && s->u_prev && s->f_prev, "u / u_prev / f_prev are NULL");
    RBFFD_CHECK_ARG(p->nspecies == 1 || (s->v && s->v_prev && s->g_prev), "v state is NULL");
    RBFFD_CHECK_ARG(p->dt > 0 && p->tol > 0 && p->maxit > 0 && nsteps >= 0, "dt / tol / maxit / nsteps");
    RBFFD_CHECK_ARG(p->model >= RBFFD_MODEL_NONE && p->model <= RBFFD_MODEL_BARRIO, "model");
    RBFFD_CHECK_ARG(p->model != RBFFD_MODEL_BARRIO || p->coef[1] != 0.0, "Barrio model needs beta != 0");
    const int order = p->order == 0 ? 2 : p->order;
    RBFFD_CHECK_ARG(order >= 1 && order <= 4, "order must be 1..4 (0 = 2)");
    RBFFD_CHECK_ARG(order < 3 || (s->u_prev2 && s->f_prev2 &&
                                  (p->nspecies == 1 || (s->v_prev2 && s->g_prev2))),
                    "SBDF3/4 need u_prev2 / f_prev2 (and v_prev2 / g_prev2)");
    RBFFD_CHECK_ARG(order < 4 || (s->u_prev3 && s->f_prev3 &&
                                  (p->nspecies == 1 || (s->v_prev3 && s->g_prev3))),
                    "SBDF4 needs u_prev3 / f_prev3 (and v_prev3 / g_prev3)");
    RBFFD_CHECK_ARG(s->has_history >= 0, "has_history must be >= 0");
    RBFFD_CHECK_ARG(p->solver == RBFFD_SOLVER_BICGSTAB || p->solver == RBFFD_SOLVER_BANDED_LU, "solver");
    cudaStream_t st = as_stream(stream);
    const size_t elem = p->dtype == RBFFD_F32 ? 4 : 8;
    rbffd_step_ws* ws = op->step;
    if (ws && ws->elem != elem) {
        step_ws_free(ws);
        ws = op->step = nullptr;
    }
    if (!ws) {
        ws = new rbffd_step_ws();   // value-initialised: all zero
        op->step = ws;
        ws->elem = elem;
        ws->N = op->N;
        RBFFD_CUDA_TRY(cudaMalloc(&ws->vec, 2 * 7 * ((op->N + 3) & ~(int64_t)3) * elem));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->bar, sizeof(unsigned long long)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->flags, 5 * sizeof(int)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->tstart, sizeof(double)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->ctl, sizeof(PhaseCtl)));
        RBFFD_CUDA_TRY(cudaMemset(ws->ctl, 0, sizeof(PhaseCtl)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->pp, (size_t)std::max<int64_t>(1, (op->N + PT - 1) / PT) * 8 * sizeof(double)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->rpart, (size_t)2 * sm_count() * RES_SUMS * sizeof(double)));
        ws->rep_cap = 0;
    }
    if (ws->rep_cap < std::max<int64_t>(nsteps, 1)) {
        cudaFree(ws->rep);
        cudaFree(ws->rep_res);
        ws->rep_cap = std::max<int64_t>(nsteps, 1);
        RBFFD_CUDA_TRY(cudaMalloc(&ws->rep, ws->rep_cap * 3 * sizeof(int)));
        RBFFD_CUDA_TRY(cudaMalloc(&ws->rep_res, ws->rep_cap * 2 * sizeof(double)));
    }
    const int kept = std::max(order - 1, 1);   // past levels the order stores
    const int hist0 = std::min(s->has_history, kept);
    int hflags[5] = {0, 0, hist0, 0, 0};   // slot counter starts at 0
    if (p->solver == RBFFD_SOLVER_BANDED_LU) {
        // factor (c0 I - cl delta L) for every SBDF order this call steps
        // with (orders climb while history builds up) and species, once per
        // (order, dt, delta, dtype); factors live with the workspace
        int h = std::min(s->has_history, kept);
        bool need[4] = {false, false, false, false};
        for (int64_t k = 0; k < nsteps && k < 4; ++k) {
            need[std::min(order, h + 1) - 1] = true;
            h = std::min(h + 1, kept);
        }
        if (nsteps > 4) need[std::min(order, h + 1) - 1] = true;
        const double c0s[4] = {1.0, 3.0, 11.0, 25.0}, cls[4] = {1.0, 2.0, 6.0, 12.0};
        const double del[2] = {p->delta_u, p->delta_v};
        for (int o = 0; o < 4; ++o) {
            if (!need[o]) continue;
            for (int sp = 0; sp < p->nspecies; ++sp) {
                const double alpha = c0s[o], beta = cls[o] * p->dt * del[sp];
                rbffd_lu*& f = ws->lu[o][sp];
                // float64 factors whatever the step's dtype: a float32 band
                // LU loses several digits to its growth and rounding, while
                // the substitutions are latency-bound, not FP64-bound
                if (f && (f->alpha != alpha || f->beta != beta)) {
                    lu_free(f);
                    f = nullptr;
                }
                if (!f) {
                    rbffd_status fs = lu_factor(op, alpha, beta, RBFFD_F64, st, &f);
                    if (fs != RBFFD_OK) return fs;
                }
            }
        }
        if (!ws->ywork) RBFFD_CUDA_TRY(cudaMalloc(&ws->ywork, (2 * (2 * op->N + 16)) * sizeof(double) + 64));
    }
    RBFFD_CUDA_TRY(cudaMemcpyAsync(ws->flags, hflags, sizeof(hflags), cudaMemcpyHostToDevice, st));
    RBFFD_CUDA_TRY(cudaMemcpyAsync(ws->tstart, &s->t, sizeof(double), cudaMemcpyHostToDevice, st));
    RBFFD_CUDA_TRY(cudaMemsetAsync(ws->rep, 0, ws->rep_cap * 3 * sizeof(int), st));
    rbffd_status rs;
    const bool lu = p->solver == RBFFD_SOLVER_BANDED_LU;
    bool phased = false;   // BiCGSTAB ran as phase kernels (their launches are counted from the report)
    if (elem == 4) {
        Args<float> a;
        memset(&a, 0, sizeof(a));
        fill_args(a, op, s, p, ws);
        rs = run_steps(a, ws, nsteps, p->use_graph != 0, lu, hist0, &phased, st);
    } else {
        Args<double> a;
        memset(&a, 0, sizeof(a));
        fill_args(a, op, s, p, ws);
        rs = run_steps(a, ws, nsteps, p->use_graph != 0, lu, hist0, &phased, st);
    }
    if (rs != RBFFD_OK) return rs;
    std::vector<int> rep(std::max<int64_t>(nsteps, 1) * 3);
    std::vector<double> res(std::max<int64_t>(nsteps, 1) * 2);
    RBFFD_CUDA_TRY(cudaMemcpyAsync(hflags, ws->flags, 4 * sizeof(int), cudaMemcpyDeviceToHost, st));
    if (nsteps > 0) {
        RBFFD_CUDA_TRY(cudaMemcpyAsync(rep.data(), ws->rep, nsteps * 3 * sizeof(int), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(res.data(), ws->rep_res, nsteps * 2 * sizeof(double),
                                       cudaMemcpyDeviceToHost, st));
    }
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    rbffd_step_report r;
    memset(&r, 0, sizeof(r));
    r.failed_step = -1;
    for (int64_t k = 0; k < nsteps; ++k) {
        r.max_iters_u = std::max(r.max_iters_u, rep[3 * k]);
        r.max_iters_v = std::max(r.max_iters_v, rep[3 * k + 1]);
        r.total_iters += rep[3 * k] + rep[3 * k + 1];
        if (rep[3 * k + 2] && r.failed_step < 0) r.failed_step = s->step + k;
        r.last_relres_u = res[2 * k];
        r.last_relres_v = res[2 * k + 1];
    }
    if (phased && p->use_graph)
        for (int64_t k = 0; k < nsteps; ++k) note_launch(5 * std::max(rep[3 * k], rep[3 * k + 1]));
    r.steps_done = nsteps;
    s->has_history = (int)std::min<int64_t>((int64_t)std::min(s->has_history, kept) + nsteps, kept);
    s->step += nsteps;
    s->t += (double)nsteps * p->dt;
    if (report) *report = r;
    if (hflags[0]) {
        set_error("grid barrier timed out (blocks not co-resident?)");
        return RBFFD_TIMEOUT;
    }
    if (hflags[1]) {
        set_error("BiCGSTAB failed at step %lld", (long long)r.failed_step);
        return RBFFD_SOLVER_NOT_CONVERGED;
    }
    return RBFFD_OK;
}

extern "C" rbffd_status rbffd_selftest_barrier_timeout(void* stream) {
    cudaStream_t st = as_stream(stream);
    unsigned long long* bar = nullptr;
    int* err = nullptr;
    RBFFD_CUDA_TRY(cudaMalloc(&bar, sizeof(unsigned long long)));
    RBFFD_CUDA_TRY(cudaMalloc(&err, sizeof(int)));
    RBFFD_CUDA_TRY(cudaMemsetAsync(bar, 0, sizeof(unsigned long long), st));
    RBFFD_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
    lonely_barrier<<<1, 32, 0, st>>>(bar, err);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    int h = 0;
    RBFFD_CUDA_TRY(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFree(bar);
    cudaFree(err);
    if (h) {
        set_error("grid barrier wait gave up as designed");
        return RBFFD_TIMEOUT;
    }
    return RBFFD_OK;
}
