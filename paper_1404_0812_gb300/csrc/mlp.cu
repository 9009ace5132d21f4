// Learned shape-parameter warm start (not in the paper; it feeds the
// Section 5 search a first guess, and the search stays the arbiter).
//
// Features (float64 geometry, stored float32): tangent-frame offsets
// (t1.d, t2.d, nh.d) / r_s of every stencil node, with nh oriented so that
// sum nh.d <= 0, t1 = unit tangent part of the nearest neighbour's offset,
// t2 = nh x t1.  Network 3n -> 64 -> 64 -> 1 with GELU (erf form), float32.
//
// GPU design: one CTA of 256 threads owns a tile of 64 samples and runs the
// whole forward and backward pass in shared memory (4x4 register tiles for
// the three dense products); each CTA writes its gradient contribution to
// its own row of a partial buffer, and a second kernel sums the rows in a
// fixed order (deterministic) and applies Adam.  A mini-batch is too few tiles
// for the chip (1,024 samples: 16); mlp_tile_cluster then spreads each tile
// over a cluster of CTAs, with the same sums in the same order.  The products are far too
// small (64 x 64 x <=303 per tile) for tensor-core tiles to pay, and the
// network is specified in float32, so they run on the FP32 pipes.
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

namespace rbffd {
namespace {

constexpr int H = 64;      // hidden width
constexpr int TS = 64;     // samples per CTA tile
constexpr int NT = 256;    // threads per CTA

__host__ __device__ inline int64_t param_count(int D) {
    return (int64_t)D * H + H + H * H + H + H + 1;
}

struct View {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
};
__device__ inline View view(const float* p, int D) {
    View v;
    v.W1 = p;
    v.b1 = v.W1 + (int64_t)D * H;
    v.W2 = v.b1 + H;
    v.b2 = v.W2 + H * H;
    v.W3 = v.b2 + H;
    v.b3 = v.W3 + H;
    return v;
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ---------------------------------------------------------------------------
// features of the rows [0, count) of group g (internal row order = node order
// within the group)
// ---------------------------------------------------------------------------
__global__ void features_kernel(const double* __restrict__ X, const double* __restrict__ NR,
                                const int32_t* __restrict__ idx, const int32_t* __restrict__ row_node,
                                GroupInfo gi, int g, const double* __restrict__ eps,
                                float* __restrict__ feats, float* __restrict__ target) {
    const int64_t count = gi.row_begin[g + 1] - gi.row_begin[g];
    int64_t lr = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (lr >= count) return;
    const int n = gi.n[g], npad = gi.npad[g];
    const int64_t off = gi.ell_off[g];
    int c = idx[ell_elem(off, npad, lr, 0)];
    double cx = X[3 * (int64_t)c], cy = X[3 * (int64_t)c + 1], cz = X[3 * (int64_t)c + 2];
    double nx = NR[3 * (int64_t)c], ny = NR[3 * (int64_t)c + 1], nz = NR[3 * (int64_t)c + 2];
    double inv = rsqrt(nx * nx + ny * ny + nz * nz);
    nx *= inv; ny *= inv; nz *= inv;
    double rs2 = 0.0, sn = 0.0;
    for (int j = 1; j < n; ++j) {
        int k = idx[ell_elem(off, npad, lr, j)];
        double dx = X[3 * (int64_t)k] - cx, dy = X[3 * (int64_t)k + 1] - cy, dz = X[3 * (int64_t)k + 2] - cz;
        rs2 = fmax(rs2, dx * dx + dy * dy + dz * dz);
        sn += nx * dx + ny * dy + nz * dz;
    }
    if (sn > 0.0) { nx = -nx; ny = -ny; nz = -nz; }
    double rs = sqrt(rs2), irs = 1.0 / rs;
    int k1 = idx[ell_elem(off, npad, lr, 1)];
    double ax = X[3 * (int64_t)k1] - cx, ay = X[3 * (int64_t)k1 + 1] - cy, az = X[3 * (int64_t)k1 + 2] - cz;
    double an = nx * ax + ny * ay + nz * az;
    double t1x = ax - an * nx, t1y = ay - an * ny, t1z = az - an * nz;
    double it = rsqrt(t1x * t1x + t1y * t1y + t1z * t1z);
    t1x *= it; t1y *= it; t1z *= it;
    double t2x = ny * t1z - nz * t1y, t2y = nz * t1x - nx * t1z, t2z = nx * t1y - ny * t1x;
    // the projections in float32: each offset is formed in float64 (no
    // cancellation) and rounded once, the frame vectors carry the 1 / r_s
    // scale; the float32 features then differ from float64 projections by
    // a few float32 roundings (~1e-7 of their size), and the float64 pipe
    // (a small fraction of the float32 one here) does only the subtractions
    const float f1x = (float)(t1x * irs), f1y = (float)(t1y * irs), f1z = (float)(t1z * irs);
    const float f2x = (float)(t2x * irs), f2y = (float)(t2y * irs), f2z = (float)(t2z * irs);
    const float f3x = (float)(nx * irs), f3y = (float)(ny * irs), f3z = (float)(nz * irs);
    float* f = feats + lr * (int64_t)(3 * n);
    for (int j = 0; j < n; ++j) {
        int k = idx[ell_elem(off, npad, lr, j)];
        const float dx = (float)(X[3 * (int64_t)k] - cx), dy = (float)(X[3 * (int64_t)k + 1] - cy),
                    dz = (float)(X[3 * (int64_t)k + 2] - cz);
        f[3 * j] = fmaf(f1x, dx, fmaf(f1y, dy, f1z * dz));
        f[3 * j + 1] = fmaf(f2x, dx, fmaf(f2y, dy, f2z * dz));
        f[3 * j + 2] = fmaf(f3x, dx, fmaf(f3y, dy, f3z * dz));
    }
    if (target) target[lr] = (float)log(eps[row_node[gi.row_begin[g] + lr]] * rs);
}

// ---------------------------------------------------------------------------
// one tile: forward (mode 0: write predictions) or forward + backward
// (mode 1: per-CTA gradient partial and loss partial)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(NT)
mlp_tile(const float* __restrict__ params, int D, const float* __restrict__ feats,
         const float* __restrict__ target, const int32_t* __restrict__ sel, int64_t count,
         float inv_B, int mode, float* __restrict__ pred, float* __restrict__ partial,
         float* __restrict__ loss_part) {
    extern __shared__ float sm[];
    float* Xs = sm;                     // TS x D
    float* Z1 = Xs + TS * D;            // TS x H
    float* H1 = Z1 + TS * H;
    float* Z2 = H1 + TS * H;
    float* H2 = Z2 + TS * H;
    float* ys = H2 + TS * H;            // TS
    float* dys = ys + TS;               // TS
    const View P = view(params, D);
    const int t = threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.x * TS;
    const int ns = (int)((count - s0) < TS ? (count - s0) : TS);

    for (int e = t; e < TS * D; e += NT) {
        int s = e / D, d = e - s * D;
        float v = 0.f;
        if (s < ns) {
            int64_t row = sel ? sel[s0 + s] : s0 + s;
            v = feats[row * D + d];
        }
        Xs[e] = v;
    }
    __syncthreads();
    const int sa = (t >> 4) * 4;    // 4 samples
    const int ha = (t & 15) * 4;    // 4 hidden units
    {   // Z1 = X W1 + b1
        float acc[4][4];
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) acc[a][b] = P.b1[ha + b];
        for (int d = 0; d < D; ++d) {
            float4 w = __ldg(reinterpret_cast<const float4*>(P.W1 + (int64_t)d * H + ha));
            for (int a = 0; a < 4; ++a) {
                float x = Xs[(sa + a) * D + d];
                acc[a][0] = fmaf(x, w.x, acc[a][0]);
                acc[a][1] = fmaf(x, w.y, acc[a][1]);
                acc[a][2] = fmaf(x, w.z, acc[a][2]);
                acc[a][3] = fmaf(x, w.w, acc[a][3]);
            }
        }
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) {
                Z1[(sa + a) * H + ha + b] = acc[a][b];
                H1[(sa + a) * H + ha + b] = gelu(acc[a][b]);
            }
    }
    __syncthreads();
    {   // Z2 = H1 W2 + b2
        float acc[4][4];
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) acc[a][b] = P.b2[ha + b];
        for (int k = 0; k < H; ++k) {
            float4 w = __ldg(reinterpret_cast<const float4*>(P.W2 + k * H + ha));
            for (int a = 0; a < 4; ++a) {
                float x = H1[(sa + a) * H + k];
                acc[a][0] = fmaf(x, w.x, acc[a][0]);
                acc[a][1] = fmaf(x, w.y, acc[a][1]);
                acc[a][2] = fmaf(x, w.z, acc[a][2]);
                acc[a][3] = fmaf(x, w.w, acc[a][3]);
            }
        }
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) {
                Z2[(sa + a) * H + ha + b] = acc[a][b];
                H2[(sa + a) * H + ha + b] = gelu(acc[a][b]);
            }
    }
    __syncthreads();
    if (t < TS) {
        float y = P.b3[0];
        for (int h = 0; h < H; ++h) y = fmaf(H2[t * H + h], P.W3[h], y);
        ys[t] = y;
        if (mode == 0 && t < ns) pred[s0 + t] = y;
    }
    if (mode == 0) return;
    __syncthreads();
    if (t < TS) {
        float r = 0.f;
        if (t < ns) {
            int64_t row = sel ? sel[s0 + t] : s0 + t;
            r = ys[t] - target[row];
        }
        dys[t] = 2.f * r * inv_B;
        ys[t] = r * r;   // reuse for the loss
    }
    __syncthreads();
    const int64_t Pc = param_count(D);
    float* G = partial + (int64_t)blockIdx.x * Pc;
    float* gW1 = G;
    float* gb1 = gW1 + (int64_t)D * H;
    float* gW2 = gb1 + H;
    float* gb2 = gW2 + H * H;
    float* gW3 = gb2 + H;
    float* gb3 = gW3 + H;
    if (t < H) {            // dW3, loss
        float g = 0.f;
        for (int s = 0; s < TS; ++s) g = fmaf(H2[s * H + t], dys[s], g);
        gW3[t] = g;
    } else if (t == H) {
        float g = 0.f, l = 0.f;
        for (int s = 0; s < TS; ++s) {
            g += dys[s];
            l += ys[s];
        }
        gb3[0] = g;
        loss_part[blockIdx.x] = l;
    }
    __syncthreads();
    // dZ2 = dy W3^T * gelu'(Z2)  (in place in Z2)
    for (int e = t; e < TS * H; e += NT) {
        int s = e / H, h = e - s * H;
        Z2[e] = dys[s] * P.W3[h] * gelu_grad(Z2[e]);
    }
    __syncthreads();
    {   // dW2 = H1^T dZ2 ; dZ1 = (dZ2 W2^T) * gelu'(Z1) into H2
        const int ka = (t >> 4) * 4;
        float acc[4][4] = {};
        for (int s = 0; s < TS; ++s) {
            float4 dz = *reinterpret_cast<const float4*>(Z2 + s * H + ha);
            for (int a = 0; a < 4; ++a) {
                float x = H1[s * H + ka + a];
                acc[a][0] = fmaf(x, dz.x, acc[a][0]);
                acc[a][1] = fmaf(x, dz.y, acc[a][1]);
                acc[a][2] = fmaf(x, dz.z, acc[a][2]);
                acc[a][3] = fmaf(x, dz.w, acc[a][3]);
            }
        }
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) gW2[(ka + a) * H + ha + b] = acc[a][b];
        // dH1[s][k] = sum_h dZ2[s][h] W2[k][h]; thread: samples sa..+3, k = ha..+3
        float dh[4][4] = {};
        for (int h = 0; h < H; ++h) {
            float w0 = P.W2[(ha + 0) * H + h], w1 = P.W2[(ha + 1) * H + h];
            float w2 = P.W2[(ha + 2) * H + h], w3 = P.W2[(ha + 3) * H + h];
            for (int a = 0; a < 4; ++a) {
                float dz = Z2[(sa + a) * H + h];
                dh[a][0] = fmaf(dz, w0, dh[a][0]);
                dh[a][1] = fmaf(dz, w1, dh[a][1]);
                dh[a][2] = fmaf(dz, w2, dh[a][2]);
                dh[a][3] = fmaf(dz, w3, dh[a][3]);
            }
        }
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
                H2[(sa + a) * H + ha + b] = dh[a][b] * gelu_grad(Z1[(sa + a) * H + ha + b]);
    }
    __syncthreads();
    if (t < H) {            // db2, db1
        float g2 = 0.f, g1 = 0.f;
        for (int s = 0; s < TS; ++s) {
            g2 += Z2[s * H + t];
            g1 += H2[s * H + t];
        }
        gb2[t] = g2;
        gb1[t] = g1;
    }
    // dW1 = X^T dZ1
    for (int d = t >> 4; d < D; d += NT / 16) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int s = 0; s < TS; ++s) {
            float x = Xs[s * D + d];
            float4 dz = *reinterpret_cast<const float4*>(H2 + s * H + ha);
            acc[0] = fmaf(x, dz.x, acc[0]);
            acc[1] = fmaf(x, dz.y, acc[1]);
            acc[2] = fmaf(x, dz.z, acc[2]);
            acc[3] = fmaf(x, dz.w, acc[3]);
        }
        for (int b = 0; b < 4; ++b) gW1[(int64_t)d * H + ha + b] = acc[b];
    }
}

// ---------------------------------------------------------------------------
// forward + backward of one tile on a cluster of C CTAs (mode 1 of mlp_tile
// for mini-batches).  A step is bound by latency: 16 tiles of 1,024 samples
// keep 16 of 152 SMs busy for 85 us.  Here a CTA runs TS / C samples forward
// and back to dZ1, copies its samples' H1, H2, dZ2 and dZ1 to its peers through
// distributed shared memory, and after one cluster barrier forms 1 / C of the
// gradient's rows over all samples of the tile.  Every element keeps its sum in
// sample order, so the gradient has the bits of mlp_tile's.  n = 50, batches of
// 1,024: 85 -> 13 us for the gradient of a step.
// ---------------------------------------------------------------------------
constexpr int W2S = H + 1;   // row stride of W2 in shared memory (rows and columns are read)

struct ClusterTile {         // float offsets in shared memory
    int X, XS, XC, W1, W2, W3, Z1, Z2, H1, H2, D2, D1, dy, sq, total;
    __host__ __device__ ClusterTile(int D, int C) {
        const int own = TS / C, slice = (D + C - 1) / C;
        XS = (D + 3) / 4 * 4;         // row stride of X (read four features at a time)
        int o = 0;
        W1 = o; o += D * H;
        W3 = o; o += H;
        X = o; o += own * XS;         // own samples' features
        XC = o; o += TS * slice;      // all samples' features of this CTA's gradient rows
        W2 = o; o += H * W2S;
        Z1 = o; o += own * H;
        Z2 = o; o += own * H;
        o = (o + 3) / 4 * 4;
        // all samples, filled by the cluster (H1: the columns of this CTA's rows
        // of dW2 beside its own samples; H2: complete on the last CTA)
        H1 = o; o += TS * H;
        H2 = o; o += TS * H;
        D2 = o; o += TS * H;
        D1 = o; o += TS * H;
        dy = o; o += TS;
        sq = o; o += TS;
        total = o;
    }
};

// acc + a[0] w[0] + ... + a[3] w[3], in this order (a: 16-byte aligned, shared memory)
__device__ __forceinline__ float dot4(const float* a, const float (&w)[4], float acc) {
    const float4 x = *reinterpret_cast<const float4*>(a);
    return fmaf(x.w, w[3], fmaf(x.z, w[2], fmaf(x.y, w[1], fmaf(x.x, w[0], acc))));
}

__device__ __forceinline__ void st_peer4(uint32_t a, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ void cp4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// rows and features of the tile's samples, by asynchronous copies (loads in the
// products' loops cost 15 us of L2 latency); they need no weights, so a step's
// are on their way while the step before it (and nothing else) updates those
template <int C>
__device__ __forceinline__ void load_samples(float* smc, const ClusterTile& L, int64_t* row, int D,
                                             const float* feats, const int32_t* sel, int64_t s0, int ns, int rank) {
    constexpr int OWN = TS / C;
    const int t = threadIdx.x, first = rank * OWN, slice = (D + C - 1) / C, d0 = rank * slice;
    if (t < TS) row[t] = t < ns ? (sel ? (int64_t)sel[s0 + t] : s0 + t) : -1;
    __syncthreads();
    for (int s = t >> 5; s < TS; s += NT / 32) {        // a warp per sample
        const float* f = feats + row[s] * D;
        const bool real = row[s] >= 0;
        for (int d = d0 + (t & 31); d < d0 + slice; d += 32) {
            float* to = smc + L.XC + s * slice + d - d0;
            if (real && d < D) cp4(to, f + d); else *to = 0.f;
        }
        if (s >= first && s < first + OWN)
            for (int d = t & 31; d < D; d += 32) {
                float* to = smc + L.X + (s - first) * L.XS + d;
                if (real) cp4(to, f + d); else *to = 0.f;
            }
    }
}

// weights, forward and backward pass, and the tile's gradient partial; start:
// the peers' first barrier phase is still to be waited for
template <int C>
__device__ __forceinline__ void cluster_gradient(float* smc, const ClusterTile& L, const int64_t* row, const View& P,
                                                 int D, const float* target, int ns, float inv_B, int rank,
                                                 bool start, float* G, float* loss_part) {
    constexpr int OWN = TS / C, PER = OWN / 4;   // samples of this CTA; outputs per thread of a layer
    const int t = threadIdx.x;
    const int first = rank * OWN;                // tile sample of this CTA's sample 0
    const int slice = (D + C - 1) / C, d0 = rank * slice, d1 = min(D, d0 + slice);
    for (int e = 4 * t; e < D * H; e += 4 * NT) cp16(smc + L.W1 + e, P.W1 + e);
    for (int e = t; e < H; e += NT) cp4(smc + L.W3 + e, P.W3 + e);
    for (int e = t; e < H * H; e += NT) cp4(smc + L.W2 + (e / H) * W2S + e % H, P.W2 + e);
    const int h = t & 63, sb = t >> 6;           // this thread's unit; samples sb + 4 i
    const float bias1 = __ldcg(P.b1 + h), bias2 = __ldcg(P.b2 + h), bias3 = __ldcg(P.b3);
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const float tgt = t < OWN && first + t < ns ? target[row[first + t]] : 0.f;
    float* const H1 = smc + L.H1 + first * H;    // own samples' rows of the shared arrays
    float* const H2 = smc + L.H2 + first * H;
    float* const D2 = smc + L.D2 + first * H;
    float* const D1 = smc + L.D1 + first * H;
    float acc[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = bias1;
    // four features of a sample per load: one word of shared memory per FMA
    // and load cost the layers twice the reads
    int d = 0;
#pragma unroll 4
    for (; d + 4 <= D; d += 4) {
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = smc[L.W1 + (d + q) * H + h];
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] = dot4(smc + L.X + (sb + 4 * i) * L.XS + d, w, acc[i]);
    }
    for (; d < D; ++d) {
        const float w = smc[L.W1 + d * H + h];
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] = fmaf(smc[L.X + (sb + 4 * i) * L.XS + d], w, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        smc[L.Z1 + (sb + 4 * i) * H + h] = acc[i];
        H1[(sb + 4 * i) * H + h] = gelu(acc[i]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = bias2;
#pragma unroll 4
    for (int k = 0; k < H; k += 4) {
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = smc[L.W2 + (k + q) * W2S + h];
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] = dot4(H1 + (sb + 4 * i) * H + k, w, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        smc[L.Z2 + (sb + 4 * i) * H + h] = acc[i];
        H2[(sb + 4 * i) * H + h] = gelu(acc[i]);
    }
    __syncthreads();
    if (t < OWN) {
        float y = bias3;
#pragma unroll 16
        for (int k = 0; k < H; ++k) y = fmaf(H2[t * H + k], smc[L.W3 + k], y);
        float r = 0.f;
        if (first + t < ns) r = y - tgt;
        smc[L.dy + first + t] = 2.f * r * inv_B;
        smc[L.sq + first + t] = r * r;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int s = sb + 4 * i;
        D2[s * H + h] = smc[L.dy + first + s] * smc[L.W3 + h] * gelu_grad(smc[L.Z2 + s * H + h]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = 0.f;
#pragma unroll 4
    for (int k = 0; k < H; k += 4) {
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = smc[L.W2 + h * W2S + k + q];   // unit h of layer 1
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] = dot4(D2 + (sb + 4 * i) * H + k, w, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) D1[(sb + 4 * i) * H + h] = acc[i] * gelu_grad(smc[L.Z1 + (sb + 4 * i) * H + h]);
    __syncthreads();
    // ---- own samples to the peers
    if (start) asm volatile("barrier.cluster.wait;" ::: "memory");
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smc);
    for (int e = t; e < C * OWN * (H / 4); e += NT) {
        const int p = e / (OWN * (H / 4)), q = e - p * (OWN * (H / 4));
        if (p == rank) continue;
        const uint32_t pb = peer_addr(base, p);
        const int off = first * H + 4 * q;
        const int col = (4 * q) % H;
        if (col >= p * (H / C) && col < (p + 1) * (H / C))
            st_peer4(pb + 4 * (L.H1 + off), *reinterpret_cast<const float4*>(smc + L.H1 + off));
        if (p == C - 1) st_peer4(pb + 4 * (L.H2 + off), *reinterpret_cast<const float4*>(smc + L.H2 + off));
        st_peer4(pb + 4 * (L.D2 + off), *reinterpret_cast<const float4*>(smc + L.D2 + off));
        st_peer4(pb + 4 * (L.D1 + off), *reinterpret_cast<const float4*>(smc + L.D1 + off));
        if (q < 2 * OWN / 4) {   // dy and sq of the own samples
            const int o1 = (q < OWN / 4 ? L.dy : L.sq) + first + 4 * (q % (OWN / 4));
            st_peer4(pb + 4 * o1, *reinterpret_cast<const float4*>(smc + o1));
        }
    }
    cluster_barrier();
    // ---- this CTA's rows of the tile's gradient
    float* gW1 = G;
    float* gb1 = gW1 + (int64_t)D * H;
    float* gW2 = gb1 + H;
    float* gb2 = gW2 + H * H;
    float* gW3 = gb2 + H;
    float* gb3 = gW3 + H;
    const int ha = (t & 15) * 4, rg = t >> 4;
    for (int d = d0 + rg; d < d1; d += NT / 16) {
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
        for (int s = 0; s < TS; ++s) {
            const float x = smc[L.XC + s * slice + (d - d0)];
            const float4 dz = *reinterpret_cast<const float4*>(smc + L.D1 + s * H + ha);
            a[0] = fmaf(x, dz.x, a[0]);
            a[1] = fmaf(x, dz.y, a[1]);
            a[2] = fmaf(x, dz.z, a[2]);
            a[3] = fmaf(x, dz.w, a[3]);
        }
        for (int b = 0; b < 4; ++b) gW1[(int64_t)d * H + ha + b] = a[b];   // a tile's partial starts at any float
    }
    for (int k = rank * (H / C) + rg; k < (rank + 1) * (H / C); k += NT / 16) {
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
        for (int s = 0; s < TS; ++s) {
            const float x = smc[L.H1 + s * H + k];
            const float4 dz = *reinterpret_cast<const float4*>(smc + L.D2 + s * H + ha);
            a[0] = fmaf(x, dz.x, a[0]);
            a[1] = fmaf(x, dz.y, a[1]);
            a[2] = fmaf(x, dz.z, a[2]);
            a[3] = fmaf(x, dz.w, a[3]);
        }
        for (int b = 0; b < 4; ++b) gW2[k * H + ha + b] = a[b];
    }
    if (rank == 0 && t < H) {
        float g2 = 0.f, g1 = 0.f;
#pragma unroll 8
        for (int s = 0; s < TS; ++s) {
            g2 += smc[L.D2 + s * H + t];
            g1 += smc[L.D1 + s * H + t];
        }
        gb2[t] = g2;
        gb1[t] = g1;
    } else if (rank == C - 1 && t < H) {
        float g = 0.f;
#pragma unroll 8
        for (int s = 0; s < TS; ++s) g = fmaf(smc[L.H2 + s * H + t], smc[L.dy + s], g);
        gW3[t] = g;
    } else if (rank == C - 1 && t == H) {
        float g = 0.f, l = 0.f;
        for (int s = 0; s < TS; ++s) {
            g += smc[L.dy + s];
            l += smc[L.sq + s];
        }
        gb3[0] = g;
        *loss_part = l;
    }
}

template <int C>
__global__ void __launch_bounds__(NT)
mlp_tile_cluster(const float* __restrict__ params, int D, const float* __restrict__ feats,
                 const float* __restrict__ target, const int32_t* __restrict__ sel, int64_t count, float inv_B,
                 float* __restrict__ partial, float* __restrict__ loss_part) {
    extern __shared__ __align__(16) float smc[];
    __shared__ int64_t row[TS];
    const ClusterTile L(D, C);
    const int rank = blockIdx.x % C;
    const int64_t tile = blockIdx.x / C, s0 = tile * TS;
    const int ns = (int)((count - s0) < TS ? (count - s0) : TS);
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // peers have started (waited for below)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load_samples<C>(smc, L, row, D, feats, sel, s0, ns, rank);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    cluster_gradient<C>(smc, L, row, view(params, D), D, target, ns, inv_B, rank, true,
                        partial + tile * param_count(D), loss_part + tile);
}

// p's gradient: the sum over tiles in a fixed order
__device__ __forceinline__ float sum_tiles(const float* partial, int ntiles, int64_t P, int64_t p) {
    float g = 0.f;
#pragma unroll 16
    for (int c = 0; c < ntiles; ++c) g += __ldcg(partial + (int64_t)c * P + p);
    return g;
}

__device__ __forceinline__ void adam_update(float* params, float* m, float* v, int64_t p, float g, int adam_t,
                                            float lr) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    float mm = b1 * m[p] + (1.f - b1) * g;
    float vv = b2 * v[p] + (1.f - b2) * g * g;
    m[p] = mm;
    v[p] = vv;
    float mh = mm / (1.f - powf(b1, (float)adam_t));
    float vh = vv / (1.f - powf(b2, (float)adam_t));
    params[p] -= lr * mh / (sqrtf(vh) + eps);
}

// grad[p] = sum over tiles of partial[c][p] (fixed order); optionally Adam.
__global__ void reduce_grad(const float* __restrict__ partial, int ntiles, int64_t P,
                            const float* __restrict__ loss_part, float* __restrict__ grad,
                            float* __restrict__ loss_out, float* __restrict__ params,
                            float* __restrict__ m, float* __restrict__ v, int adam_t, float lr,
                            int loss_slot) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < P;
         p += (int64_t)gridDim.x * blockDim.x) {
        const float g = sum_tiles(partial, ntiles, P, p);
        if (grad) grad[p] = g;
        if (params) adam_update(params, m, v, p, g, adam_t, lr);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && loss_out) {
        float l = 0.f;
        for (int c = 0; c < ntiles; ++c) l += loss_part[c];
        loss_out[loss_slot] = l;
    }
}

// ---------------------------------------------------------------------------
// a whole epoch of mini-batch steps in one cooperative launch of clusters: the
// CTAs stay on their SMs, a step's two kernels become two halves between grid
// barriers (each parameter's sum and Adam update by one thread of the grid),
// and the next step's features are fetched under the barrier.  With a pair of
// launches per step the host's launch calls were the bound (n = 50, batches of
// 1,024: 29 us a step, 18 of them the kernels; 20 us in this kernel).
// The barriers are bounded: a CTA that gives up leaves its loop, and a last
// cluster barrier keeps its shared memory in place until a peer that passed the
// same grid barrier has stored to it.
// ---------------------------------------------------------------------------
struct EpochArgs {
    float *params, *adam_m, *adam_v, *partial, *loss_part, *loss_out;
    const float *feats, *target;
    const int32_t* sel;
    int64_t count, P;
    int D, batch, adam_t;   // adam_t: steps taken before this epoch
    float lr;
    unsigned long long* bar;
    int* err;
};

template <int C>
__global__ void __launch_bounds__(NT) mlp_epoch_cluster(EpochArgs a) {
    extern __shared__ __align__(16) float smc[];
    __shared__ int64_t row[TS];
    const ClusterTile L(a.D, C);
    const int rank = blockIdx.x % C, tile = blockIdx.x / C;
    const View P = view(a.params, a.D);
    const int64_t s0 = (int64_t)tile * TS;
    unsigned long long target = 0;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    int step = 0;
    for (int64_t b0 = 0; b0 < a.count; b0 += a.batch, ++step) {
        const int64_t nb = min((int64_t)a.batch, a.count - b0);
        const int tiles = (int)((nb + TS - 1) / TS);
        const bool mine = tile < tiles;             // (a last, smaller batch leaves clusters idle)
        const int ns = (int)min((int64_t)TS, nb - s0);
        if (mine) load_samples<C>(smc, L, row, a.D, a.feats, a.sel + b0, s0, ns, rank);
        if (step > 0 && !grid_sync(a.bar, target += gridDim.x, a.err)) break;   // the weights are updated
        if (mine)
            cluster_gradient<C>(smc, L, row, P, a.D, a.target, ns, __fdiv_rn(1.f, (float)nb), rank, step == 0,
                                a.partial + tile * a.P, a.loss_part + tile);
        if (!grid_sync(a.bar, target += gridDim.x, a.err)) break;               // the partials are complete
        for (int64_t p = blockIdx.x * (int64_t)NT + threadIdx.x; p < a.P; p += (int64_t)gridDim.x * NT)
            adam_update(a.params, a.adam_m, a.adam_v, p, sum_tiles(a.partial, tiles, a.P, p), a.adam_t + step + 1,
                        a.lr);
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == NT - 1) {
            float l = 0.f;
#pragma unroll 16
            for (int c = 0; c < tiles; ++c) l += __ldcg(a.loss_part + c);
            a.loss_out[step] = l;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    cluster_barrier();
}

size_t tile_smem(int D) { return (size_t)(TS * D + 4 * TS * H + 2 * TS) * sizeof(float); }

template <int C>
rbffd_status launch_cluster_tiles(const rbffd_mlp* m, const float* feats, const float* target, const int32_t* sel,
                                  int64_t count, int tiles, float* loss_part, bool after_reduce, cudaStream_t st) {
    const size_t smem = (size_t)ClusterTile(m->D, C).total * sizeof(float);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * C));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see launch_reduce
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = after_reduce ? 2 : 1;
    RBFFD_CUDA_TRY(cudaLaunchKernelEx(&cfg, mlp_tile_cluster<C>, (const float*)m->params, m->D, feats, target, sel,
                                      count, 1.f / (float)count, m->partial, loss_part));
    note_launch();
    return RBFFD_OK;
}

// Gradient partials of `count` samples (sel: their rows, or NULL): clusters of
// eight or four CTAs per tile while those stay within one wave of the chip, a
// CTA per tile beyond (its register tiles move fewer shared-memory bytes per
// FMA, and there are tiles enough), or where the weights of a large network
// leave no room for a cluster's arrays.  after_reduce: the kernel ahead on the
// stream is this network's reduce_grad, which writes no samples; only then may the
// tiles start while it drains, because they fetch their samples before they wait
// for it.  Behind any other kernel, which may be the one that makes the samples and
// may let its dependents start early, they are launched in plain stream order.
constexpr size_t CLUSTER_SMEM_MAX = 227 * 1024;
template <int C>
bool cluster_fits(int D) { return ClusterTile(D, C).total * sizeof(float) + 1024 <= CLUSTER_SMEM_MAX; }

rbffd_status gradient_tiles(const rbffd_mlp* m, const float* feats, const float* target, const int32_t* sel,
                            int64_t count, float* loss_part, bool after_reduce, cudaStream_t st) {
    const int64_t tiles = (count + TS - 1) / TS;
    if (tiles * 8 <= sm_count() && cluster_fits<8>(m->D))
        return launch_cluster_tiles<8>(m, feats, target, sel, count, (int)tiles, loss_part, after_reduce, st);
    if (tiles * 4 <= sm_count() && cluster_fits<4>(m->D))
        return launch_cluster_tiles<4>(m, feats, target, sel, count, (int)tiles, loss_part, after_reduce, st);
    mlp_tile<<<(unsigned)tiles, NT, tile_smem(m->D), st>>>(m->params, m->D, feats, target, sel, count,
                                                           1.f / (float)count, 1, nullptr, m->partial, loss_part);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    return RBFFD_OK;
}

// The sum over tiles (and Adam).  Launched, like the cluster tiles, as a
// programmatic dependent: the kernel starts while the one before it drains, and
// waits for its results (griddepcontrol.wait) only before it reads them, which
// takes the launch latencies of a step's two kernels off its path.
rbffd_status launch_reduce(const rbffd_mlp* m, int tiles, float* grad, float* params, float* am, float* av, int adam_t,
                           float lr, int slot, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((m->P + 127) / 128));
    cfg.blockDim = dim3(128);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    RBFFD_CUDA_TRY(cudaLaunchKernelEx(&cfg, reduce_grad, (const float*)m->partial, tiles, m->P,
                                      (const float*)(m->loss + 4096), grad, m->loss, params, am, av, adam_t, lr, slot));
    note_launch();
    return RBFFD_OK;
}

// The grid barrier's words, behind the losses.
unsigned long long* barrier_words(const rbffd_mlp* m) {
    return reinterpret_cast<unsigned long long*>(m->loss + 4096 + (m->partial_rows + 1) / 2 * 2);
}

template <int C>
rbffd_status launch_epoch(const rbffd_mlp* m, EpochArgs a, int tiles, cudaStream_t st, bool* done) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * C));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = (size_t)ClusterTile(m->D, C).total * sizeof(float);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    RBFFD_TRY(allow_shared((const void*)mlp_epoch_cluster<C>));
    int resident = 0;
    RBFFD_CUDA_TRY(cudaOccupancyMaxActiveClusters(&resident, mlp_epoch_cluster<C>, &cfg));
    if (resident < tiles) return RBFFD_OK;
    a.bar = barrier_words(m);
    a.err = reinterpret_cast<int*>(a.bar + 1);
    RBFFD_CUDA_TRY(cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned long long), st));
    RBFFD_CUDA_TRY(cudaLaunchKernelEx(&cfg, mlp_epoch_cluster<C>, a));
    note_launch();
    *done = true;
    return RBFFD_OK;
}

// One epoch (the samples in the order sel) in one launch where its clusters are
// all resident at once: of eight CTAs per tile, else of four (batches of more
// tiles than 1,024 samples have).  Otherwise *done stays false.
rbffd_status epoch_launch(const rbffd_mlp* m, const float* feats, const float* target, const int32_t* sel,
                          int64_t count, int batch, float lr, cudaStream_t st, bool* done) {
    EpochArgs a = {};
    a.params = m->params;
    a.adam_m = m->adam_m;
    a.adam_v = m->adam_v;
    a.partial = m->partial;
    a.loss_part = m->loss + 4096;
    a.loss_out = m->loss;
    a.feats = feats;
    a.target = target;
    a.sel = sel;
    a.count = count;
    a.P = m->P;
    a.D = m->D;
    a.batch = batch;
    a.adam_t = m->adam_t;
    a.lr = lr;
    const int64_t tiles = (std::min<int64_t>(batch, count) + TS - 1) / TS;
    *done = false;
    rbffd_status s = RBFFD_OK;
    if (tiles * 8 <= sm_count() && cluster_fits<8>(m->D)) s = launch_epoch<8>(m, a, (int)tiles, st, done);
    if (s == RBFFD_OK && !*done && tiles * 4 <= sm_count() && cluster_fits<4>(m->D))
        s = launch_epoch<4>(m, a, (int)tiles, st, done);
    return s;
}

rbffd_status ensure_smem() {
    RBFFD_TRY(allow_shared((const void*)mlp_tile));
    RBFFD_TRY(allow_shared((const void*)mlp_tile_cluster<8>));
    RBFFD_TRY(allow_shared((const void*)mlp_tile_cluster<4>));
    return RBFFD_OK;
}

rbffd_status ensure_train_ws(rbffd_mlp* m, int64_t tiles) {
    if (!m->adam_m) {
        RBFFD_CUDA_TRY(cudaMalloc(&m->adam_m, m->P * sizeof(float)));
        RBFFD_CUDA_TRY(cudaMalloc(&m->adam_v, m->P * sizeof(float)));
        RBFFD_CUDA_TRY(cudaMemset(m->adam_m, 0, m->P * sizeof(float)));
        RBFFD_CUDA_TRY(cudaMemset(m->adam_v, 0, m->P * sizeof(float)));
    }
    if (m->partial_rows < tiles) {
        cudaFree(m->partial);
        cudaFree(m->loss);
        m->partial = nullptr;
        RBFFD_CUDA_TRY(cudaMalloc(&m->partial, tiles * m->P * sizeof(float)));
        RBFFD_CUDA_TRY(cudaMalloc(&m->loss, (tiles + 4096 + 6) * sizeof(float))   /* and barrier words */);
        m->partial_rows = tiles;
    }
    return RBFFD_OK;
}

rbffd_status predict_launch(const rbffd_mlp* m, const float* feats, int64_t count, float* out,
                            cudaStream_t st) {
    if (count <= 0) return RBFFD_OK;
    rbffd_status s = ensure_smem();
    if (s != RBFFD_OK) return s;
    unsigned tiles = (unsigned)((count + TS - 1) / TS);
    mlp_tile<<<tiles, NT, tile_smem(m->D), st>>>(m->params, m->D, feats, nullptr, nullptr, count, 0.f,
                                                 0, out, nullptr, nullptr);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    return RBFFD_OK;
}

__global__ void scatter_guess(const float* __restrict__ pred, int64_t count, int64_t row0,
                              float* __restrict__ guess) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < count) guess[row0 + i] = pred[i];
}

__global__ void fill_nan(float* a, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) a[i] = NAN;
}

}  // namespace

rbffd_status mlp_guess(const rbffd_op* op, const double* nodes, const double* normals,
                       const rbffd_build_opts& o, float* guess_rows, cudaStream_t st) {
    fill_nan<<<(unsigned)((op->N + 255) / 256), 256, 0, st>>>(guess_rows, op->N);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    for (int g = 0; g < op->gi.ngroups; ++g) {
        const rbffd_mlp* net = nullptr;
        for (int i = 0; i < RBFFD_MAX_GROUPS; ++i)
            if (o.mlp[i] && o.mlp[i]->n == op->gi.n[g]) net = o.mlp[i];
        if (!net) continue;
        int64_t count = op->gi.row_begin[g + 1] - op->gi.row_begin[g];
        float *feats = nullptr, *pred = nullptr;
        RBFFD_CUDA_TRY(pool_alloc(&feats, count * net->D * sizeof(float), st));
        RBFFD_CUDA_TRY(pool_alloc(&pred, count * sizeof(float), st));
        features_kernel<<<(unsigned)((count + 127) / 128), 128, 0, st>>>(
            nodes, normals, op->idx, op->row_node, op->gi, g, nullptr, feats, nullptr);
        note_launch();
        RBFFD_CUDA_TRY(cudaGetLastError());
        rbffd_status s = predict_launch(net, feats, count, pred, st);
        if (s != RBFFD_OK) return s;
        scatter_guess<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(pred, count, op->gi.row_begin[g],
                                                                       guess_rows);
        note_launch();
        RBFFD_CUDA_TRY(cudaGetLastError());
        cudaFreeAsync(feats, st);
        cudaFreeAsync(pred, st);
    }
    return RBFFD_OK;
}

}  // namespace rbffd

using namespace rbffd;

extern "C" {

int64_t rbffd_mlp_param_count(int n) { return param_count(3 * n); }

rbffd_status rbffd_mlp_create(int n, const float* params_host, rbffd_mlp** out) {
    RBFFD_CHECK_ARG(out, "out is NULL");
    *out = nullptr;
    RBFFD_CHECK_ARG(n >= 2 && n <= RBFFD_MAX_N, "n must be in [2, 128]");
    rbffd_mlp* m = new rbffd_mlp();
    memset(m, 0, sizeof(*m));
    m->n = n;
    m->D = 3 * n;
    m->P = param_count(m->D);
    cudaError_t e = cudaMalloc(&m->params, m->P * sizeof(float));
    if (e == cudaSuccess)
        e = params_host ? cudaMemcpy(m->params, params_host, m->P * sizeof(float), cudaMemcpyHostToDevice)
                        : cudaMemset(m->params, 0, m->P * sizeof(float));
    if (e != cudaSuccess) {
        set_error("rbffd_mlp_create: %s", cudaGetErrorString(e));
        cudaFree(m->params);
        delete m;
        return RBFFD_ECUDA;
    }
    *out = m;
    return RBFFD_OK;
}

rbffd_status rbffd_mlp_get_params(const rbffd_mlp* m, float* params_host) {
    RBFFD_CHECK_ARG(m && params_host, "NULL argument");
    RBFFD_CUDA_TRY(cudaMemcpy(params_host, m->params, m->P * sizeof(float), cudaMemcpyDeviceToHost));
    return RBFFD_OK;
}

rbffd_status rbffd_mlp_load(rbffd_mlp* m, const float* params_host) {
    RBFFD_CHECK_ARG(m && params_host, "NULL argument");
    RBFFD_CUDA_TRY(cudaMemcpy(m->params, params_host, m->P * sizeof(float), cudaMemcpyHostToDevice));
    // new parameters start a new optimisation: Adam's moments and step count reset
    if (m->adam_m) RBFFD_CUDA_TRY(cudaMemset(m->adam_m, 0, m->P * sizeof(float)));
    if (m->adam_v) RBFFD_CUDA_TRY(cudaMemset(m->adam_v, 0, m->P * sizeof(float)));
    m->adam_t = 0;
    return RBFFD_OK;
}

void rbffd_mlp_destroy(rbffd_mlp* m) {
    if (!m) return;
    cudaFree(m->params);
    cudaFree(m->adam_m);
    cudaFree(m->adam_v);
    cudaFree(m->partial);
    cudaFree(m->grad);
    cudaFree(m->loss);
    delete m;
}

rbffd_status rbffd_features(const rbffd_op* op, const double* nodes, const double* normals, int n,
                            float* feats, float* target, int64_t* count_host, void* stream) {
    RBFFD_CHECK_ARG(op && nodes && normals && feats, "NULL argument");
    cudaStream_t st = as_stream(stream);
    int g = -1;
    for (int i = 0; i < op->gi.ngroups; ++i)
        if (op->gi.n[i] == n) g = i;
    RBFFD_CHECK_ARG(g >= 0, "no stencil of that size in the operator");
    int64_t count = op->gi.row_begin[g + 1] - op->gi.row_begin[g];
    if (count_host) *count_host = count;
    features_kernel<<<(unsigned)((count + 127) / 128), 128, 0, st>>>(nodes, normals, op->idx, op->row_node,
                                                                     op->gi, g, op->eps, feats, target);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    return RBFFD_OK;
}

rbffd_status rbffd_mlp_loss_grad(const rbffd_mlp* mc, const float* feats, const float* target,
                                 int64_t count, float* grad, float* loss, void* stream) {
    RBFFD_CHECK_ARG(mc && feats && target && grad && count > 0, "NULL argument");
    rbffd_mlp* m = const_cast<rbffd_mlp*>(mc);
    cudaStream_t st = as_stream(stream);
    int64_t tiles = (count + TS - 1) / TS;
    rbffd_status s = ensure_train_ws(m, tiles);
    if (s != RBFFD_OK) return s;
    s = ensure_smem();
    if (s != RBFFD_OK) return s;
    s = gradient_tiles(m, feats, target, nullptr, count, m->loss + 4096, false, st);
    if (s != RBFFD_OK) return s;
    s = launch_reduce(m, (int)tiles, grad, nullptr, nullptr, nullptr, 0, 0.f, 0, st);
    if (s != RBFFD_OK) return s;
    if (loss) {
        // mean squared error = sum of squares / count
        float hl = 0.f;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(&hl, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
        hl /= (float)count;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(loss, &hl, sizeof(float), cudaMemcpyHostToDevice, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return RBFFD_OK;
}

rbffd_status rbffd_mlp_train(rbffd_mlp* m, const float* feats, const float* target, int64_t count,
                             int epochs, int batch, float lr, uint64_t seed, void* stream,
                             float* loss_host) {
    RBFFD_CHECK_ARG(m && feats && target && count > 0 && epochs > 0 && batch > 0, "bad argument");
    RBFFD_CHECK_ARG(count < (int64_t)1 << 31, "too many samples");
    cudaStream_t st = as_stream(stream);
    int64_t tiles_per_batch = (batch + TS - 1) / TS;
    rbffd_status s = ensure_train_ws(m, tiles_per_batch);
    if (s != RBFFD_OK) return s;
    s = ensure_smem();
    if (s != RBFFD_OK) return s;
    int32_t* perm_d = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&perm_d, count * sizeof(int32_t), st));
    struct Freed {   // whichever way the call ends
        int32_t* p;
        cudaStream_t st;
        ~Freed() { cudaFreeAsync(p, st); }
    } freed{perm_d, st};
    std::vector<int32_t> perm(count), next;
    for (int64_t i = 0; i < count; ++i) perm[i] = (int32_t)i;
    std::mt19937_64 rng(seed);
    int64_t steps_per_epoch = (count + batch - 1) / batch;
    RBFFD_CHECK_ARG(steps_per_epoch <= 4096, "count / batch must be <= 4096");
    std::vector<float> lossv(steps_per_epoch);
    auto shuffle = [&](std::vector<int32_t>& p) {
        for (int64_t i = count - 1; i > 0; --i) {
            int64_t j = (int64_t)(rng() % (uint64_t)(i + 1));
            std::swap(p[i], p[j]);
        }
    };
    shuffle(perm);
    for (int ep = 0; ep < epochs; ++ep) {
        RBFFD_CUDA_TRY(cudaMemcpyAsync(perm_d, perm.data(), count * sizeof(int32_t), cudaMemcpyHostToDevice, st));
        bool whole;
        s = epoch_launch(m, feats, target, perm_d, count, batch, lr, st, &whole);
        if (s != RBFFD_OK) return s;
        if (whole) m->adam_t += (int)steps_per_epoch;
        for (int64_t b = 0; !whole && b < steps_per_epoch; ++b) {
            int64_t b0 = b * batch;
            int64_t nb = std::min<int64_t>(batch, count - b0);
            unsigned tiles = (unsigned)((nb + TS - 1) / TS);
            ++m->adam_t;   // the step counter lives with the network's moments
            s = gradient_tiles(m, feats, target, perm_d + b0, nb, m->loss + 4096, b > 0, st);
            if (s != RBFFD_OK) return s;
            s = launch_reduce(m, (int)tiles, nullptr, m->params, m->adam_m, m->adam_v, m->adam_t, lr, (int)b, st);
            if (s != RBFFD_OK) return s;
        }
        RBFFD_CUDA_TRY(cudaGetLastError());
        if (ep + 1 < epochs) {   // the next epoch's order while the device works on this one
            next = perm;
            shuffle(next);
        }
        int gave_up = 0;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(lossv.data(), m->loss, steps_per_epoch * sizeof(float),
                                       cudaMemcpyDeviceToHost, st));
        if (whole)
            RBFFD_CUDA_TRY(cudaMemcpyAsync(&gave_up, barrier_words(m) + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
        if (gave_up) {
            set_error("rbffd_mlp_train: a grid barrier of the training kernel gave up");
            return RBFFD_TIMEOUT;
        }
        perm.swap(next);
        if (loss_host) {
            double tot = 0.0;
            for (float l : lossv) tot += l;
            loss_host[ep] = (float)(tot / (double)count);
        }
    }
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    return RBFFD_OK;
}

rbffd_status rbffd_mlp_predict(const rbffd_mlp* m, const float* feats, int64_t count, float* out,
                               void* stream) {
    RBFFD_CHECK_ARG(m && feats && out, "NULL argument");
    return predict_launch(m, feats, count, out, as_stream(stream));
}

}  // extern "C"
