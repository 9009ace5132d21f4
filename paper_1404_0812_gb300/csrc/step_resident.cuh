// IMEX steps with the operator resident on the chip: one launch runs all the
// steps of a call, each block keeping its slices of the ELL matrix in shared
// memory and its rows' vectors in registers.
//
// What bounds it.  An operator of up to about 30 MB fits the shared memory of
// the chip, and then an iteration moves no matrix bytes: what is left are its
// synchronisations (one for each vector that neighbours read or sum that all
// blocks need, five per BiCGSTAB iteration) and the gathers.  Two forms:
//
//  * one thread-block cluster (up to 16 blocks) for small operators: the
//    gathered vector is copied to every block's shared memory, sums and copies
//    travel through distributed shared memory, and the barrier is the
//    cluster's (a few hundred nanoseconds);
//  * a cooperative grid of one block per SM: gathers through L1 / L2 and the
//    bounded grid barrier (about a microsecond).
//
// TPR lanes share a row: each reads every TPR-th chunk of four entries, a
// shuffle adds them up, and all of them hold the row's vector entries in
// registers.  Sums of products go through shared memory, one value per row,
// to one warp per sum (float64 arithmetic on all warps would cost more than
// the iteration; float32 products are scaled, exact and summed as Dot3, as in the
// phase kernels), and then from every block to all in a fixed order.
//
// Measured against one cooperative launch per step with the matrix streamed
// from L2 and three blocks for the small operator: 2,562 nodes, n = 31, heat
// equation in float64, 3.8 iterations per step: 314 -> 52 us per step; 40k
// torus, n = 50, two species in float32: 320 -> 92 us per step (its sums: a sphere of
// the same size 82 us with these, 78 with pairs of float32 values, which lost accuracy
// and the range of small and large fields, 85 with float64 ones).
//
// Included by step.cu inside its anonymous namespace.

struct ResidentInfo {
    int spb;             // slices of 32 rows per block
    int max_elems;       // matrix elements of a block, at most
    int64_t nsteps;
    int nhist;           // past levels valid when the call begins
    void* gather;        // grid form: ns x N gathered vector
    double* part;        // grid form: 2 x blocks x RES_SUMS
};

// A row's product as it goes to the summing warp.  Float64: the product itself.
// Float32: two factors scaled by the caller, as their exact product p + e; or, in
// the right-hand side's sums, whose scale is not known yet, the factors themselves,
// which the summing warp scales to the block's largest.
template <typename T>
struct Term {
    using type = double;
    __device__ static double of(double a, double b) { return a * b; }
    __device__ static double raw(double a, double b) { return a * b; }
    // the sum of the block's rows (times 2^e; RAW: of factors) by one warp, valid in lane 0
    template <bool RAW, int UN>
    __device__ static double sum(const double* t, int rows, int ln, int) {
        double s = t[ln];
#pragma unroll 4
        for (int r = ln + 32; r < rows; r += 32) s += t[r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        return s;
    }
};
template <>
struct Term<float> {
    using type = float2;
    __device__ static float2 of(float a, float b) {
        const float p = __fmul_rn(a, b);
        return make_float2(p, __fmaf_rn(a, b, -p));
    }
    __device__ static float2 raw(float a, float b) { return make_float2(a, b); }
    template <bool RAW, int UN>
    __device__ static double sum(const float2* t, int rows, int ln, int e) {
        float fa = 1.f, fb = 1.f;
        if (RAW) {
            unsigned ma = 0, mb = 0;   // largest magnitudes (their bits order like integers)
#pragma unroll 4
            for (int r = ln; r < rows; r += 32) {
                ma = max(ma, __float_as_uint(t[r].x) & 0x7fffffffu);
                mb = max(mb, __float_as_uint(t[r].y) & 0x7fffffffu);
            }
            const int ea = unit_exp((int)(__reduce_max_sync(0xffffffffu, ma) >> 23) - 127);
            const int eb = unit_exp((int)(__reduce_max_sync(0xffffffffu, mb) >> 23) - 127);
            fa = unit_scale(ea);
            fb = unit_scale(eb);
            e = ea + eb;
        }
        // (UN: blocks of few rows run faster with less code, two species on the
        // 60k sphere 95 -> 93 us a step, 150k rows with more, 166 -> 156)
        Dot3 s;
        acc_zero(s);
#pragma unroll UN
        for (int r = ln; r < rows; r += 32) {
            const float2 x = t[r];
            if (RAW) acc_add(s, x.x * fa, x.y * fb);
            else acc_pair(s, x.x, x.y);
        }
        return fixed_value(warp_sum(s, e));
    }
};

static_assert(sizeof(Term<float>::type) == RES_TERM && sizeof(Term<double>::type) == RES_TERM, "size of a term");

// one block's view of the synchronisations
template <typename T, int TPR, bool CL>
struct ResidentBlock {
    unsigned char* sm;
    ResidentSmem<T> L;
    const Args<T>& a;
    const ResidentInfo& ri;
    int rows;                        // rows of a block (padding included)
    int parity = 0;
    unsigned long long target = 0;   // grid form: barrier count

    // x (node i of species sp) to wherever blocks gather from: the TPR lanes
    // of the row share the peers
    __device__ void publish(int sp, int64_t i, int lane, T x) {
        if (CL) {
            const uint32_t at = smem_addr(sm + L.gather) + (uint32_t)((sp * a.N + i) * sizeof(T));
            for (int p = lane; p < (int)gridDim.x; p += TPR) st_cluster(peer_addr(at, p), x);
        } else if (lane == 0) {
            ((T*)ri.gather)[sp * a.N + i] = x;
        }
    }
    __device__ const T* gathered(int sp) const {
        return (CL ? (const T*)(sm + L.gather) : (const T*)ri.gather) + sp * a.N;
    }
    __device__ bool sync() {
        if (CL) {
            cluster_barrier();
            return true;
        }
        return grid_sync(a.bar, target += gridDim.x, a.flags);
    }
    // KS sums per species over all rows (terms v of each row, written by its
    // lane 0), and the barrier that makes them, and what was published,
    // visible; lane 0 of warp k then decides with the totals of species k.  exp_of:
    // exponent of sum j of species k (or RAW terms)
    template <int KS, int NS, bool RAW = false, typename E, typename F>
    __device__ bool reduce(const typename Term<T>::type (&v)[NS][KS], int row, bool writes, E exp_of, F decide) {
        using V = typename Term<T>::type;
        V* terms = (V*)(sm + L.terms);
        if (writes) {
#pragma unroll
            for (int k = 0; k < NS; ++k)
#pragma unroll
                for (int j = 0; j < KS; ++j) terms[(k * KS + j) * rows + row] = v[k][j];
        }
        __syncthreads();
        const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
        double* pp = CL ? (double*)(sm + L.part) + parity * RES_CLUSTER * RES_SUMS
                        : ri.part + (int64_t)parity * gridDim.x * RES_SUMS;
        for (int k = wid; k < NS * KS; k += nw) {
            const double s = Term<T>::template sum<RAW, TPR == 1 ? 4 : 2>(terms + k * rows, rows, ln, exp_of(k / KS, k % KS));
            if (CL) {
                const double t = __shfl_sync(0xffffffffu, s, 0);
                if (ln < (int)gridDim.x) st_cluster(peer_addr(smem_addr(pp + blockIdx.x * RES_SUMS + k), ln), t);
            } else if (ln == 0) {
                __stcg(pp + (int64_t)blockIdx.x * RES_SUMS + k, s);
            }
        }
        if (!sync()) return false;
        for (int k = wid; k < NS; k += nw) {
            double tot[KS];
#pragma unroll
            for (int j = 0; j < KS; ++j) tot[j] = 0.0;
            if (CL) {   // at most 16 blocks
#pragma unroll
                for (int j = 0; j < KS; ++j) tot[j] = ln < (int)gridDim.x ? pp[ln * RES_SUMS + k * KS + j] : 0.0;
            } else {
                for (int b0 = ln; b0 < (int)gridDim.x; b0 += 160) {   // five loads per lane in flight
                    double x[5][KS];
#pragma unroll
                    for (int u = 0; u < 5; ++u)
#pragma unroll
                        for (int j = 0; j < KS; ++j)
                            x[u][j] = b0 + 32 * u < (int)gridDim.x
                                          ? __ldcg(pp + (int64_t)(b0 + 32 * u) * RES_SUMS + k * KS + j) : 0.0;
#pragma unroll
                    for (int u = 0; u < 5; ++u)
#pragma unroll
                        for (int j = 0; j < KS; ++j) tot[j] += x[u][j];
                }
            }
#pragma unroll
            for (int o = CL ? RES_CLUSTER / 2 : 16; o > 0; o >>= 1)
#pragma unroll
                for (int j = 0; j < KS; ++j) tot[j] += __shfl_down_sync(0xffffffffu, tot[j], o);
            if (ln == 0) decide(k, tot);
        }
        __syncthreads();
        parity ^= 1;
        return true;
    }
};

template <typename T, int TPR, int NS, bool CL>
__global__ void __launch_bounds__(res_threads<T>(), 1) resident_kernel(Args<T> a, ResidentInfo ri) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    using TM = Term<T>;
    using PA = PhaseAcc<T>;
    const int rows = ri.spb * 32, RPW = 32 / TPR;
    ResidentBlock<T, TPR, CL> B{res_smem, ResidentSmem<T>(ri.max_elems, rows, a.N, NS, CL), a, ri, rows};
    T* sw = (T*)(res_smem + B.L.w);
    int32_t* si = (int32_t*)(res_smem + B.L.idx);

    // ---- this block's slices into shared memory; this thread's row
    const int64_t s0 = (int64_t)blockIdx.x * ri.spb;
    int64_t e0 = -1, e1 = 0;   // element range of the block
    const int tid = threadIdx.x, lane = (tid & 31) / RPW;            // lane of the row
    const int lrow = (tid >> 5) * RPW + (tid & 31) % RPW;            // row of the block
    bool own = false;
    int64_t node = 0, rbase = 0;
    int nch = 0;
    {
        int64_t sl = 0;   // slices before group g
        for (int g = 0; g < a.gi.ngroups; ++g) {
            const int64_t cnt = a.gi.row_begin[g + 1] - a.gi.row_begin[g], ns = (cnt + 31) / 32;
            const int64_t lo = max(s0, sl), hi = min(s0 + ri.spb, sl + ns);
            if (lo < hi) {
                const int64_t se = (int64_t)32 * a.gi.npad[g];
                if (e0 < 0) e0 = a.gi.ell_off[g] + (lo - sl) * se;
                e1 = a.gi.ell_off[g] + (hi - sl) * se;
            }
            const int64_t my = s0 + lrow / 32;
            if (lrow < rows && my >= sl && my < sl + ns) {
                const int64_t lr = (my - sl) * 32 + lrow % 32;
                own = lr < cnt;
                if (own) node = a.row_node[a.gi.row_begin[g] + lr];
                rbase = ell_elem(a.gi.ell_off[g], a.gi.npad[g], lr, 0);
                nch = a.gi.npad[g] >> 2;
            }
            sl += ns;
        }
    }
    if (e0 < 0) e0 = e1;
    for (int64_t e = e0 + 4 * tid; e < e1; e += 4 * (int64_t)blockDim.x) {
        *reinterpret_cast<int4*>(si + (e - e0)) = __ldcs(reinterpret_cast<const int4*>(a.idx + e));
        T w[4];
        load4s(a.w + e, w);
#pragma unroll
        for (int q = 0; q < 4; ++q) sw[e - e0 + q] = w[q];
    }
    const int sb = (int)(rbase - e0);

    // row sums of both species against the gathered vector
    auto product = [&](T (&y)[NS]) {
#pragma unroll
        for (int k = 0; k < NS; ++k) y[k] = T(0);
        if (own) {
            const T* g0 = B.gathered(0);
            const T* g1 = NS == 2 ? B.gathered(1) : g0;
#pragma unroll 2
            for (int c = lane; c < nch; c += TPR) {
                const int4 iv = *reinterpret_cast<const int4*>(si + sb + c * 128);
                T w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] = sw[sb + c * 128 + q];
                const int ii[4] = {iv.x, iv.y, iv.z, iv.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    y[0] = fma(w[q], g0[ii[q]], y[0]);
                    if (NS == 2) y[NS - 1] = fma(w[q], g1[ii[q]], y[NS - 1]);
                }
            }
        }
#pragma unroll
        for (int o = RPW; o < 32; o <<= 1)
#pragma unroll
            for (int k = 0; k < NS; ++k) y[k] += __shfl_xor_sync(0xffffffffu, y[k], o);
    };

    T x[NS], r[NS], rh[NS], p[NS], q[NS], s[NS], t[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        x[k] = own ? (k == 0 ? a.u : a.v)[node] : T(0);
        r[k] = rh[k] = p[k] = q[k] = s[k] = t[k] = T(0);
    }
    const bool lead = own && lane == 0, sums = lane == 0 && lrow < rows;
    volatile ResidentScalars<T>& sc = *(volatile ResidentScalars<T>*)(res_smem + B.L.scal);
    // state of the deciding lanes (lane 0 of warps 0 .. NS - 1); res2, limit2:
    // squared norms of the residual and of its tolerance
    double bnorm = 0.0, limit2 = 0.0, rho = 0.0, rho_prev = 1.0, alpha = 1.0, omega = 1.0, res2 = 0.0;
    bool active = false, fail = false;
    int iters = 0, it = 0, nhist = ri.nhist;
    if (CL) cluster_barrier();   // every block of the cluster runs before its shared memory is written

    for (int64_t step = 0; step < ri.nsteps; ++step) {
        const StepCoef<T> kc = step_coef_at(a, nhist, (int)step);
        const T kk[2] = {kc.k0, kc.k1};
#pragma unroll
        for (int k = 0; k < NS; ++k)
            if (own) B.publish(k, node, lane, x[k]);
        if (!B.sync()) return;
        // ---- right-hand side, r0 = b - A x
        T y[NS], b[2] = {T(0), T(0)};
        product(y);
        if (lead) rhs_values(a, kc, node, x[0], NS == 2 ? x[NS - 1] : T(0), b[0], b[1]);
        typename TM::type d1[NS][1], d2[NS][2];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            b[k] = __shfl_sync(0xffffffffu, b[k], (tid & 31) % RPW);
            r[k] = b[k] - (kc.c0 * x[k] - kk[k] * y[k]);
            rh[k] = r[k];
            p[k] = q[k] = T(0);
            d2[k][0] = TM::raw(b[k], b[k]);
            d2[k][1] = TM::raw(r[k], r[k]);
        }
        it = 0;
        if (!B.template reduce<2, NS, true>(d2, lrow, sums, [](int, int) { return 0; }, [&](int k, const double (&tot)[2]) {
                bnorm = sqrt(tot[0]);
                limit2 = (a.tol * bnorm) * (a.tol * bnorm);
                rho = tot[1];   // (r-hat, r0) = |r0|^2
                rho_prev = alpha = omega = 1.0;
                res2 = rho;
                active = !(bnorm == 0.0 || sqrt(rho) / bnorm <= a.tol);
                fail = active && !isfinite(rho);
                active = active && !fail;
                iters = 0;
                sc.beta[k] = T(0);
                sc.omega[k] = T(1);
                sc.act[k] = active;
                sc.zero[k] = bnorm == 0.0;
                sc.e0[k] = sc.e[k] = PhaseAcc<T>::exp_of(rho);
            }))
            return;
#pragma unroll
        for (int k = 0; k < NS; ++k)
            if (sc.zero[k]) x[k] = T(0);   // b = 0: x = 0
        // exponents of the sums' factors and their scales (float32 only)
        const auto e0 = [&](int k) { return sizeof(T) == 4 ? (int)sc.e0[k] : 0; };
        const auto e = [&](int k) { return sizeof(T) == 4 ? (int)sc.e[k] : 0; };
        while ((sc.act[0] || (NS == 2 && sc.act[NS - 1])) && it < a.maxit) {
            ++it;
            // ---- A: p = r + beta (p - omega q)
#pragma unroll
            for (int k = 0; k < NS; ++k)
                if (sc.act[k] && own) {
                    p[k] = r[k] + sc.beta[k] * (p[k] - sc.omega[k] * q[k]);
                    B.publish(k, node, lane, p[k]);
                }
            if (!B.sync()) return;
            // ---- B: q = A p ; (r-hat, q)
            product(y);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (sc.act[k]) q[k] = kc.c0 * p[k] - kk[k] * y[k];
                d1[k][0] = TM::of(PA::scaled(rh[k], unit_scale(e0(k))), PA::scaled(q[k], unit_scale(e(k))));
            }
            if (!B.template reduce<1, NS>(d1, lrow, sums, [&](int k, int) { return e0(k) + e(k); }, [&](int k, const double (&tot)[1]) {
                    if (active) {
                        alpha = rho / tot[0];
                        if (tot[0] == 0.0 || !isfinite(alpha)) {
                            fail = true;
                            active = false;
                        }
                        sc.alpha[k] = (T)alpha;
                    }
                    sc.act[k] = active;
                }))
                return;
            // ---- C: s = r - alpha q ; |s|^2
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (sc.act[k] && own) {
                    s[k] = r[k] - sc.alpha[k] * q[k];
                    B.publish(k, node, lane, s[k]);
                }
                d1[k][0] = TM::of(PA::scaled(s[k], unit_scale(e(k))), PA::scaled(s[k], unit_scale(e(k))));
            }
            if (!B.template reduce<1, NS>(d1, lrow, sums, [&](int k, int) { return 2 * e(k); }, [&](int k, const double (&tot)[1]) {
                    const bool early = active && tot[0] <= limit2;
                    if (early) {
                        res2 = tot[0];
                        iters = it;
                        active = false;
                    }
                    sc.early[k] = early;
                    sc.act[k] = active;
                }))
                return;
            // ---- D: t = A s ; (t, s), (t, t)   (x += alpha p where s converged)
#pragma unroll
            for (int k = 0; k < NS; ++k)
                if (sc.early[k]) x[k] += sc.alpha[k] * p[k];
            if (!(sc.act[0] || (NS == 2 && sc.act[NS - 1]))) break;
            product(y);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (sc.act[k]) t[k] = kc.c0 * s[k] - kk[k] * y[k];
                const T ts = PA::scaled(t[k], unit_scale(e(k)));
                d2[k][0] = TM::of(ts, PA::scaled(s[k], unit_scale(e(k))));
                d2[k][1] = TM::of(ts, ts);
            }
            if (!B.template reduce<2, NS>(d2, lrow, sums, [&](int k, int) { return 2 * e(k); }, [&](int k, const double (&tot)[2]) {
                    if (active) {
                        omega = tot[0] / tot[1];
                        if (tot[1] == 0.0 || !isfinite(omega)) {
                            fail = true;
                            active = false;
                        }
                        sc.omega[k] = (T)omega;
                    }
                    sc.act[k] = active;
                }))
                return;
            // ---- E: x += alpha p + omega s ; r = s - omega t ; (r-hat, r), |r|^2
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (sc.act[k]) {
                    x[k] += sc.alpha[k] * p[k] + sc.omega[k] * s[k];
                    r[k] = s[k] - sc.omega[k] * t[k];
                }
                const T rs = PA::scaled(r[k], unit_scale(e(k)));
                d2[k][0] = TM::of(PA::scaled(rh[k], unit_scale(e0(k))), rs);
                d2[k][1] = TM::of(rs, rs);
            }
            if (!B.template reduce<2, NS>(d2, lrow, sums, [&](int k, int j) { return (j ? e(k) : e0(k)) + e(k); }, [&](int k, const double (&tot)[2]) {
                    if (active) {
                        rho_prev = rho;
                        rho = tot[0];
                        if (tot[1] <= limit2) {
                            iters = it;
                            active = false;
                        } else {
                            // beta of the next iteration, if there is one
                            const double beta = (rho / rho_prev) * (alpha / omega);
                            if (omega == 0.0 || (it < a.maxit && (rho == 0.0 || !isfinite(beta)))) {
                                fail = true;
                                active = false;
                            }
                            sc.beta[k] = (T)beta;
                        }
                        res2 = tot[1];
                        sc.e[k] = PhaseAcc<T>::exp_of(res2);
                    }
                    sc.act[k] = active;
                }))
                return;
        }
        // ---- report of the step
        if (blockIdx.x == 0 && (tid & 31) == 0 && (tid >> 5) < NS) {
            const int k = tid >> 5;
            if (active) iters = it;   // hit maxit
            a.rep[step * 3 + k] = iters;
            a.rep_res[step * 2 + k] = bnorm > 0 ? sqrt(res2) / bnorm : 0.0;
            if (active || fail) {
                atomicExch(a.rep + step * 3 + 2, 1);
                atomicExch(a.flags + 1, 1);
            }
            if (NS == 1) {
                a.rep[step * 3 + 1] = 0;
                a.rep_res[step * 2 + 1] = 0.0;
            }
        }
        nhist = min(nhist + 1, max(a.order - 1, 1));
    }
#pragma unroll
    for (int k = 0; k < NS; ++k)
        if (lead) (k == 0 ? a.u : a.v)[node] = x[k];
}

// the kernel of a form; float64 rows have one lane each
template <typename T, int NS, bool CL>
const void* resident_fn(int tpr) {
    if constexpr (sizeof(T) == 4) {
        if (tpr == 4) return (const void*)resident_kernel<T, 4, NS, CL>;
        if (tpr == 2) return (const void*)resident_kernel<T, 2, NS, CL>;
    }
    return (const void*)resident_kernel<T, 1, NS, CL>;
}
template <typename T>
const void* resident_fn(const ResidentPlan& p, int ns) {
    if (p.cluster) return ns == 1 ? resident_fn<T, 1, true>(p.tpr) : resident_fn<T, 2, true>(p.tpr);
    return ns == 1 ? resident_fn<T, 1, false>(p.tpr) : resident_fn<T, 2, false>(p.tpr);
}

// a launch of the plan's kernel, and whether the device can hold its cluster (the
// launch of a cluster that no partition of the device has room for fails)
template <typename T>
rbffd_status resident_config(const ResidentPlan& p, const void* fn, cudaLaunchConfig_t* cfg,
                             cudaLaunchAttribute* at) {
    RBFFD_TRY(allow_shared(fn, RES_STATIC));
    memset(cfg, 0, sizeof(*cfg));
    cfg->gridDim = dim3(p.blocks);
    cfg->blockDim = dim3(std::max(64, p.spb * 32 * p.tpr));   // at least a warp per species
    cfg->dynamicSmemBytes = p.smem;
    if (p.cluster) {
        RBFFD_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = p.blocks;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
    } else {
        at->id = cudaLaunchAttributeCooperative;
        at->val.cooperative = 1;
    }
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return RBFFD_OK;
}
template <typename T>
bool cluster_resides(const ResidentPlan& p, int ns) {
    const void* fn = resident_fn<T>(p, ns);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    int n = 0;
    if (resident_config<T>(p, fn, &cfg, &at) != RBFFD_OK) return false;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return n >= 1;
}

template <typename T>
rbffd_status resident_launch(Args<T>& a, const ResidentPlan& p, int nhist, int64_t nsteps, void* gather, double* part,
                             cudaStream_t st) {
    ResidentInfo ri;
    memset(&ri, 0, sizeof(ri));
    ri.spb = p.spb;
    ri.max_elems = p.max_elems;
    ri.nsteps = nsteps;
    ri.nhist = nhist;
    ri.gather = gather;
    ri.part = part;
    const void* fn = resident_fn<T>(p, a.ns);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    RBFFD_TRY(resident_config<T>(p, fn, &cfg, &at));
    cfg.stream = st;
    if (!p.cluster) RBFFD_CUDA_TRY(cudaMemsetAsync(a.bar, 0, sizeof(unsigned long long), st));
    void* args[] = {&a, &ri};
    RBFFD_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
    note_launch();
    return RBFFD_OK;
}
