// Locality orderings of the nodes.  Section 4.1 reorders L_X by reverse
// Cuthill-McKee (George and Liu) for faster iterative solves; a Morton
// (Z-order) key of the coordinates is the geometric alternative, available
// before any stencil exists.  Both return a permutation perm with perm[k] =
// the original index of the node placed k-th; the caller applies it to its
// node, normal and field arrays (x_new[k] = x[perm[k]]) and builds on the
// reordered set.  The Morton keys are sorted on the device (a stable radix
// sort); the breadth-first searches of the Cuthill-McKee order run on the host.
#include "common.cuh"

#include <algorithm>
#include <cstring>
#include <numeric>
#include <thread>
#include <vector>

namespace rbffd {
namespace {

constexpr int BOX_THREADS = 256;

// bounding box of n boxes (in: 6 doubles each, lo then hi) or, with X, of
// nodes: one box per block into out (min and max are exact: any order); a node that
// is not finite makes the box infinite
__global__ void __launch_bounds__(BOX_THREADS) bbox_blocks(const double* __restrict__ X, const double* __restrict__ in,
                                                          int64_t n, double* __restrict__ out) {
    __shared__ double w[6][BOX_THREADS / 32];
    double v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = blockIdx.x * (int64_t)BOX_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * BOX_THREADS)
        for (int a = 0; a < 3; ++a) {
            double lo = X ? X[3 * i + a] : in[6 * i + a], hi = X ? lo : in[6 * i + 3 + a];
            if (X && (__double2hiint(lo) & 0x7ff00000) == 0x7ff00000) {   // (fmin and fmax would drop a NaN)
                lo = -INFINITY;
                hi = INFINITY;
            }
            v[a] = fmin(v[a], lo);
            v[3 + a] = fmax(v[3 + a], hi);
        }
    for (int o = 16; o > 0; o >>= 1)
        for (int a = 0; a < 3; ++a) {
            v[a] = fmin(v[a], __shfl_xor_sync(0xffffffffu, v[a], o));
            v[3 + a] = fmax(v[3 + a], __shfl_xor_sync(0xffffffffu, v[3 + a], o));
        }
    if ((threadIdx.x & 31) == 0)
        for (int a = 0; a < 6; ++a) w[a][threadIdx.x >> 5] = v[a];
    __syncthreads();
    if (threadIdx.x < 6) {
        double x = w[threadIdx.x][0];
        for (int k = 1; k < BOX_THREADS / 32; ++k)
            x = threadIdx.x < 3 ? fmin(x, w[threadIdx.x][k]) : fmax(x, w[threadIdx.x][k]);
        out[6 * blockIdx.x + threadIdx.x] = x;
    }
}

// spread the low 21 bits of v to every third bit
__device__ __forceinline__ uint64_t spread3(uint64_t v) {
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__global__ void morton_keys(const double* __restrict__ X, int64_t N, double x0, double y0, double z0,
                            double scale, uint64_t* __restrict__ key) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double c[3] = {X[3 * i] - x0, X[3 * i + 1] - y0, X[3 * i + 2] - z0};
    uint64_t q[3];
    for (int a = 0; a < 3; ++a) {
        double t = c[a] * scale;   // in [0, 2^21 - 1]
        q[a] = (uint64_t)fmin(fmax(t, 0.0), 2097151.0);
    }
    key[i] = spread3(q[0]) | (spread3(q[1]) << 1) | (spread3(q[2]) << 2);
}

// ---------------------------------------------------------------------------
// Stable radix sort of (key, index) pairs, least significant byte first.
//
// A pass reads and writes 12 bytes per node; at a million nodes these stay in
// L2 and the sort is bound by its launches (three per pass: digit counts of
// every tile, their prefix sums digit by digit, scatter).  A tile's ranks come
// from warp matches, in element order, so equal keys keep the index order; the
// tile is put in order in shared memory first, which makes the scatter runs of
// neighbours.  Up to one tile of nodes, one block does all passes.  Against
// keys copied to the host and sorted there: 1M nodes 74 -> 0.39 ms a call.
// ---------------------------------------------------------------------------
constexpr int SORT_THREADS = 256, SORT_ITEMS = 16, SORT_WARPS = SORT_THREADS / 32;
constexpr int TILE = SORT_THREADS * SORT_ITEMS, BINS = 256, PASSES = 8;   // 63-bit keys

struct TileShared {
    uint64_t key[TILE];
    int32_t val[TILE];
    int32_t wcount[SORT_WARPS][BINS];   // per warp: counts, then the offset among equal digits
    int32_t first[BINS];                // tile position of each digit's first element
    int32_t gbase[BINS];                // global position of the same
    int32_t wsum[SORT_WARPS];
};

// exclusive prefix sum of one value per thread over the block
__device__ int32_t block_exclusive(int32_t v, int32_t* wsum) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int32_t base = 0;
    for (int k = 0; k < w; ++k) base += wsum[k];
    __syncthreads();
    return base + x - v;
}

// Sorts a tile of n elements by the digit at `shift` into S.key / S.val;
// element warp * 512 + i * 32 + lane is item i of a thread.  S.first holds the
// digits' first positions.
__device__ void sort_tile(TileShared& S, const uint64_t (&key)[SORT_ITEMS], const int32_t (&val)[SORT_ITEMS], int n,
                          int shift) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int b = threadIdx.x; b < SORT_WARPS * BINS; b += SORT_THREADS) (&S.wcount[0][0])[b] = 0;
    __syncthreads();
    int32_t rank[SORT_ITEMS];
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int e = w * (32 * SORT_ITEMS) + i * 32 + lane;
        const int d = e < n ? (int)(key[i] >> shift) & (BINS - 1) : BINS;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int32_t old = d < BINS ? S.wcount[w][d] : 0;
        rank[i] = old + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (d < BINS && (peers >> lane) == 1u) S.wcount[w][d] = old + __popc(peers);   // the last of its peers
        __syncwarp();
    }
    __syncthreads();
    int32_t total = 0;
    for (int k = 0; k < SORT_WARPS; ++k) {
        const int32_t c = S.wcount[k][threadIdx.x];
        S.wcount[k][threadIdx.x] = total;
        total += c;
    }
    S.first[threadIdx.x] = block_exclusive(total, S.wsum);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int e = w * (32 * SORT_ITEMS) + i * 32 + lane;
        if (e < n) {
            const int d = (int)(key[i] >> shift) & (BINS - 1);
            const int at = S.first[d] + S.wcount[w][d] + rank[i];
            S.key[at] = key[i];
            S.val[at] = val[i];
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(SORT_THREADS) sort_counts(const uint64_t* __restrict__ key, int64_t N, int shift,
                                                           int ntiles, int32_t* __restrict__ counts) {
    __shared__ int32_t h[BINS];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * TILE;
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int64_t e = base + i * SORT_THREADS + threadIdx.x;
        const int d = e < N ? (int)(key[e] >> shift) & (BINS - 1) : BINS;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (d < BINS && (peers >> (threadIdx.x & 31)) == 1u) atomicAdd(&h[d], __popc(peers));
    }
    __syncthreads();
    counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// counts of digit blockIdx.x over the tiles -> exclusive prefix sums, and the
// digit's total
__global__ void __launch_bounds__(SORT_THREADS) sort_prefix(int32_t* __restrict__ counts, int ntiles,
                                                           int32_t* __restrict__ totals) {
    __shared__ int32_t wsum[SORT_WARPS], last;
    int32_t* c = counts + (int64_t)blockIdx.x * ntiles;
    int32_t run = 0;
    for (int t0 = 0; t0 < ntiles; t0 += SORT_THREADS) {
        const int t = t0 + threadIdx.x;
        const int32_t v = t < ntiles ? c[t] : 0;
        const int32_t x = block_exclusive(v, wsum);
        if (t < ntiles) c[t] = run + x;
        if (threadIdx.x == SORT_THREADS - 1) last = x + v;
        __syncthreads();
        run += last;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

// one pass: keys in -> out; in_val NULL: the element's own index (first
// pass); out_key NULL: only the indices are written (last pass)
__global__ void __launch_bounds__(SORT_THREADS) sort_scatter(const uint64_t* __restrict__ in_key,
                                                            const int32_t* __restrict__ in_val, int64_t N, int shift,
                                                            int ntiles, const int32_t* __restrict__ prefix,
                                                            const int32_t* __restrict__ totals,
                                                            uint64_t* __restrict__ out_key,
                                                            int32_t* __restrict__ out_val) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    TileShared& S = *reinterpret_cast<TileShared*>(sort_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    const int n = (int)(N - base < TILE ? N - base : TILE);
    uint64_t key[SORT_ITEMS];
    int32_t val[SORT_ITEMS];
#pragma unroll
    for (int i = 0; i < SORT_ITEMS; ++i) {
        const int e = w * (32 * SORT_ITEMS) + i * 32 + lane;
        key[i] = e < n ? in_key[base + e] : 0;
        val[i] = e < n ? (in_val ? in_val[base + e] : (int32_t)(base + e)) : 0;
    }
    S.gbase[threadIdx.x] = block_exclusive(totals[threadIdx.x], S.wsum) + prefix[(int64_t)threadIdx.x * ntiles + blockIdx.x];
    sort_tile(S, key, val, n, shift);
    for (int j = threadIdx.x; j < n; j += SORT_THREADS) {
        const uint64_t k = S.key[j];
        const int d = (int)(k >> shift) & (BINS - 1);
        const int64_t at = (int64_t)S.gbase[d] + (j - S.first[d]);
        if (out_key) out_key[at] = k;
        out_val[at] = S.val[j];
    }
}

// all passes of up to one tile
__global__ void __launch_bounds__(SORT_THREADS) sort_one_tile(const uint64_t* __restrict__ in_key, int n,
                                                             int32_t* __restrict__ out_val) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    TileShared& S = *reinterpret_cast<TileShared*>(sort_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < n; j += SORT_THREADS) {
        S.key[j] = in_key[j];
        S.val[j] = j;
    }
    __syncthreads();
    for (int p = 0; p < PASSES; ++p) {
        uint64_t key[SORT_ITEMS];
        int32_t val[SORT_ITEMS];
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            const int e = w * (32 * SORT_ITEMS) + i * 32 + lane;
            key[i] = e < n ? S.key[e] : 0;
            val[i] = e < n ? S.val[e] : 0;
        }
        __syncthreads();
        sort_tile(S, key, val, n, 8 * p);
    }
    for (int j = threadIdx.x; j < n; j += SORT_THREADS) out_val[j] = S.val[j];
}

// perm = the indices of key[0..N-1] in (key, index) order; key is scratch
rbffd_status sort_keys_device(uint64_t* key, int64_t N, int32_t* perm, cudaStream_t st) {
    const size_t smem = sizeof(TileShared);
    if (N <= TILE) {
        RBFFD_TRY(allow_shared((const void*)sort_one_tile));
        sort_one_tile<<<1, SORT_THREADS, smem, st>>>(key, (int)N, perm);
        note_launch();
        RBFFD_CUDA_TRY(cudaGetLastError());
        return RBFFD_OK;
    }
    RBFFD_TRY(allow_shared((const void*)sort_scatter));
    const int ntiles = (int)((N + TILE - 1) / TILE);
    // one allocation: nothing is left behind where it fails
    uint64_t* key2 = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&key2, (size_t)N * (sizeof(uint64_t) + 2 * sizeof(int32_t)) +
                                         (size_t)BINS * (ntiles + 1) * sizeof(int32_t), st));
    int32_t *val = reinterpret_cast<int32_t*>(key2 + N), *val2 = val + N, *counts = val2 + N;
    int32_t* totals = counts + (size_t)BINS * ntiles;
    const uint64_t* k_in = key;
    uint64_t* k_out = key2;
    const int32_t* v_in = nullptr;
    int32_t* v_out = val;
    for (int p = 0; p < PASSES; ++p) {
        const bool final_pass = p == PASSES - 1;
        sort_counts<<<ntiles, SORT_THREADS, 0, st>>>(k_in, N, 8 * p, ntiles, counts);
        sort_prefix<<<BINS, SORT_THREADS, 0, st>>>(counts, ntiles, totals);
        sort_scatter<<<ntiles, SORT_THREADS, smem, st>>>(k_in, v_in, N, 8 * p, ntiles, counts, totals,
                                                        final_pass ? nullptr : k_out, final_pass ? perm : v_out);
        note_launch(3);
        k_in = k_out;
        k_out = k_out == key ? key2 : key;
        v_in = v_out;
        v_out = v_out == val ? val2 : val;
    }
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(key2, st);
    RBFFD_CUDA_TRY(e);
    return RBFFD_OK;
}

__global__ void stencil_rows(const int32_t* __restrict__ idx, const int32_t* __restrict__ row_node, GroupInfo gi,
                             int64_t R, int nmax, int32_t* __restrict__ out, int32_t* __restrict__ deg) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= R) return;
    int g = group_of_row(gi, r);
    int n = gi.n[g], npad = gi.npad[g];
    int64_t lr = r - gi.row_begin[g];
    int node = row_node[r];
    for (int j = 0; j < nmax; ++j)
        out[(int64_t)node * nmax + j] = j < n ? idx[ell_elem(gi.ell_off[g], npad, lr, j)] : -1;
    deg[node] = n;
}

}  // namespace
}  // namespace rbffd

using namespace rbffd;

extern "C" rbffd_status rbffd_morton_order(const double* nodes, int64_t N, int32_t* perm, void* stream) {
    RBFFD_CHECK_ARG(nodes && perm, "NULL argument");
    RBFFD_CHECK_ARG(N >= 1 && N < (int64_t)1 << 31, "N must be in [1, 2^31)");
    cudaStream_t st = as_stream(stream);
    const int nb = (int)std::min<int64_t>((int64_t)sm_count() * 4, (N + BOX_THREADS - 1) / BOX_THREADS);
    double* part = nullptr;
    uint64_t* key = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&part, (size_t)(nb + 1) * 6 * sizeof(double), st));
    bbox_blocks<<<nb, BOX_THREADS, 0, st>>>(nodes, nullptr, N, part + 6);
    bbox_blocks<<<1, BOX_THREADS, 0, st>>>(nullptr, part + 6, nb, part);
    note_launch(2);
    RBFFD_CUDA_TRY(cudaGetLastError());
    double box[6];
    RBFFD_CUDA_TRY(cudaMemcpyAsync(box, part, sizeof(box), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFreeAsync(part, st);
    const double *lo = box, *hi = box + 3;
    double ext = std::max(hi[0] - lo[0], std::max(hi[1] - lo[1], hi[2] - lo[2]));
    RBFFD_CHECK_ARG(std::isfinite(ext), "non-finite node coordinates");
    const double scale = ext > 0.0 ? 2097151.0 / ext : 0.0;   // one cube: the Z-order keeps proportions
    RBFFD_CUDA_TRY(pool_alloc(&key, (size_t)N * sizeof(uint64_t), st));
    morton_keys<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(nodes, N, lo[0], lo[1], lo[2], scale, key);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    const rbffd_status s = sort_keys_device(key, N, perm, st);
    cudaFreeAsync(key, st);
    if (s != RBFFD_OK) return s;
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    return RBFFD_OK;
}

extern "C" rbffd_status rbffd_rcm_order_host(const int64_t* rowptr, const int32_t* cols, int64_t N, int32_t* perm) {
    RBFFD_CHECK_ARG(rowptr && perm && (cols || N == 0), "NULL argument");
    RBFFD_CHECK_ARG(N >= 0 && N < (int64_t)1 << 31, "N must be in [0, 2^31)");
    for (int64_t i = 0; i < N; ++i)
        for (int64_t e = rowptr[i]; e < rowptr[i + 1]; ++e)
            RBFFD_CHECK_ARG(cols[e] >= 0 && cols[e] < N, "column index out of range");
    // passes over disjoint ranges of nodes, on the host's cores
    auto for_nodes = [&](auto&& body) {
        const int64_t nt = std::max<int64_t>(1, std::min<int64_t>(std::thread::hardware_concurrency(), N / 4096));
        std::vector<std::thread> pool;
        for (int64_t t = 1; t < nt; ++t) pool.emplace_back([&, t] { body(N * t / nt, N * (t + 1) / nt); });
        body(0, N / nt);
        for (auto& th : pool) th.join();
    };
    // symmetrised adjacency in one flat array: node i's slots are
    // nb[off[i] .. off[i + 1]) (its out- and in-edges, self loops dropped);
    // after the repeats are removed its neighbours are the first deg[i].
    // Each thread scans every edge and fills only the slots of its own
    // nodes, so no two threads write the same place.
    std::vector<int64_t> off((size_t)N + 1, 0);
    for_nodes([&](int64_t lo, int64_t hi) {
        for (int64_t i = 0; i < N; ++i)
            for (int64_t e = rowptr[i]; e < rowptr[i + 1]; ++e) {
                const int64_t j = cols[e];
                if (j == i) continue;
                if (i >= lo && i < hi) off[(size_t)i + 1]++;
                if (j >= lo && j < hi) off[(size_t)j + 1]++;
            }
    });
    for (int64_t i = 0; i < N; ++i) off[(size_t)i + 1] += off[(size_t)i];
    std::vector<int32_t> nb((size_t)off[(size_t)N]);
    for_nodes([&](int64_t lo, int64_t hi) {
        std::vector<int64_t> fill(off.begin() + lo, off.begin() + hi);
        for (int64_t i = 0; i < N; ++i)
            for (int64_t e = rowptr[i]; e < rowptr[i + 1]; ++e) {
                const int64_t j = cols[e];
                if (j == i) continue;
                if (i >= lo && i < hi) nb[(size_t)fill[(size_t)(i - lo)]++] = (int32_t)j;
                if (j >= lo && j < hi) nb[(size_t)fill[(size_t)(j - lo)]++] = (int32_t)i;
            }
    });
    std::vector<int32_t> deg((size_t)N);
    for_nodes([&](int64_t lo, int64_t hi) {
        for (int64_t i = lo; i < hi; ++i) {
            int32_t* a = nb.data() + off[(size_t)i];
            int32_t* b = nb.data() + off[(size_t)i + 1];
            std::sort(a, b);
            deg[(size_t)i] = (int32_t)(std::unique(a, b) - a);
        }
    });
    // neighbours in increasing degree (ties by index), the Cuthill-McKee
    // visiting order: sorted as 64-bit keys (degree, index)
    for_nodes([&](int64_t lo, int64_t hi) {
        std::vector<uint64_t> key;
        for (int64_t i = lo; i < hi; ++i) {
            int32_t* a = nb.data() + off[(size_t)i];
            const int32_t d = deg[(size_t)i];
            key.resize((size_t)d);
            for (int32_t k = 0; k < d; ++k) key[(size_t)k] = ((uint64_t)(uint32_t)deg[(size_t)a[k]] << 32) | (uint32_t)a[k];
            std::sort(key.begin(), key.end());
            for (int32_t k = 0; k < d; ++k) a[k] = (int32_t)(key[(size_t)k] & 0xffffffffu);
        }
    });
    auto adj_begin = [&](int32_t v) { return nb.data() + off[(size_t)v]; };
    auto adj_end = [&](int32_t v) { return nb.data() + off[(size_t)v] + deg[(size_t)v]; };
    std::vector<int32_t> level((size_t)N, -1), order;
    order.reserve((size_t)N);
    std::vector<char> done((size_t)N, 0);
    std::vector<int32_t> queue;
    queue.reserve((size_t)N);
    // BFS from s over the unvisited component: levels and the last level.
    // Level-synchronous: each frontier (comp[fb, fe), all at level depth) is
    // expanded by the host's threads, a node joining the next frontier through
    // an atomic claim of its level.  Levels, depth and the component's node
    // set are those of a sequential BFS; only the order of comp differs, and
    // nothing below depends on it (every choice is by (degree, index)).
    const int64_t hw = std::max<int64_t>(1, (int64_t)std::thread::hardware_concurrency());
    auto bfs_levels = [&](int32_t s, std::vector<int32_t>& comp, int& depth) {
        comp.clear();
        comp.push_back(s);
        level[s] = 0;
        depth = 0;
        size_t fb = 0, fe = 1;
        std::vector<std::vector<int32_t>> part;
        while (fb < fe) {
            const int32_t next = depth + 1;
            const int64_t F = (int64_t)(fe - fb);
            const int64_t nt = std::max<int64_t>(1, std::min<int64_t>(hw, F / 512));
            part.assign((size_t)nt, {});
            auto expand = [&](int64_t t) {
                std::vector<int32_t>& out = part[(size_t)t];
                for (size_t h = fb + (size_t)(F * t / nt); h < fb + (size_t)(F * (t + 1) / nt); ++h) {
                    const int32_t v = comp[h];
                    for (const int32_t* pw = adj_begin(v); pw != adj_end(v); ++pw) {
                        int32_t* lw = &level[(size_t)*pw];
                        int32_t expect = -1;
                        if (__atomic_load_n(lw, __ATOMIC_RELAXED) < 0 &&
                            __atomic_compare_exchange_n(lw, &expect, next, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED))
                            out.push_back(*pw);
                    }
                }
            };
            std::vector<std::thread> pool;
            for (int64_t t = 1; t < nt; ++t) pool.emplace_back(expand, t);
            expand(0);
            for (auto& th : pool) th.join();
            fb = fe;
            for (const auto& p : part) comp.insert(comp.end(), p.begin(), p.end());
            fe = comp.size();
            if (fe > fb) depth = next;
        }
    };
    std::vector<int32_t> comp;
    for (int64_t seed = 0; seed < N; ++seed) {
        if (done[(size_t)seed]) continue;
        // pseudo-peripheral start (George-Liu): from a minimum-degree node of
        // the component, move to a minimum-degree node of the deepest BFS
        // level while the eccentricity grows
        int depth;
        bfs_levels((int32_t)seed, comp, depth);
        int32_t start = (int32_t)seed;
        for (int32_t v : comp)
            if (deg[v] < deg[start] || (deg[v] == deg[start] && v < start)) start = v;
        for (int32_t v : comp) level[v] = -1;
        int d0 = -1;
        for (int it = 0; it < 8; ++it) {
            bfs_levels(start, comp, depth);
            int32_t best = -1;
            for (int32_t v : comp)
                if (level[v] == depth && (best < 0 || deg[v] < deg[best] || (deg[v] == deg[best] && v < best))) best = v;
            for (int32_t v : comp) level[v] = -1;
            if (depth <= d0) break;
            d0 = depth;
            if (best == start) break;
            start = best;
        }
        // Cuthill-McKee BFS from the start
        queue.clear();
        queue.push_back(start);
        done[(size_t)start] = 1;
        for (size_t h = 0; h < queue.size(); ++h) {
            int32_t v = queue[h];
            order.push_back(v);
            for (const int32_t* pw = adj_begin(v); pw != adj_end(v); ++pw)
                if (!done[(size_t)*pw]) {
                    done[(size_t)*pw] = 1;
                    queue.push_back(*pw);
                }
        }
    }
    // reversed
    for (int64_t k = 0; k < N; ++k) perm[k] = order[(size_t)(N - 1 - k)];
    return RBFFD_OK;
}

extern "C" rbffd_status rbffd_rcm_order(const rbffd_op* op, int32_t* perm, void* stream) {
    RBFFD_CHECK_ARG(op && perm, "NULL argument");
    cudaStream_t st = as_stream(stream);
    const int64_t N = op->N;
    const int nmax = op->n_max;
    int32_t *rows = nullptr, *deg = nullptr;
    RBFFD_CUDA_TRY(pool_alloc(&rows, (size_t)N * nmax * sizeof(int32_t), st));
    RBFFD_CUDA_TRY(pool_alloc(&deg, (size_t)N * sizeof(int32_t), st));
    stencil_rows<<<(unsigned)((N + 127) / 128), 128, 0, st>>>(op->idx, op->row_node, op->gi, N, nmax, rows, deg);
    note_launch();
    RBFFD_CUDA_TRY(cudaGetLastError());
    std::vector<int32_t> hr((size_t)N * nmax), hd((size_t)N);
    RBFFD_CUDA_TRY(cudaMemcpyAsync(hr.data(), rows, hr.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaMemcpyAsync(hd.data(), deg, hd.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFreeAsync(rows, st);
    cudaFreeAsync(deg, st);
    // CSR of the stencil graph: node k -> its n_k - 1 neighbours
    std::vector<int64_t> rp((size_t)N + 1, 0);
    for (int64_t k = 0; k < N; ++k) rp[(size_t)k + 1] = rp[(size_t)k] + std::max(0, hd[(size_t)k] - 1);
    std::vector<int32_t> cols((size_t)rp[(size_t)N]);
    for (int64_t k = 0; k < N; ++k)
        for (int j = 1; j < hd[(size_t)k]; ++j) cols[(size_t)(rp[(size_t)k] + j - 1)] = hr[(size_t)k * nmax + j];
    std::vector<int32_t> hp((size_t)N);
    rbffd_status s = rbffd_rcm_order_host(rp.data(), cols.data(), N, hp.data());
    if (s != RBFFD_OK) return s;
    RBFFD_CUDA_TRY(cudaMemcpyAsync(perm, hp.data(), (size_t)N * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    return RBFFD_OK;
}
