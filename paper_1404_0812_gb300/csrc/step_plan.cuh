// The shape of the resident step kernel (step_resident.cuh) for an operator: host
// arithmetic only, no CUDA calls.
#pragma once

#include "common.cuh"

#include <algorithm>

namespace rbffd {

constexpr int RES_SUMS = 6;        // sums of one reduction, at most
constexpr int RES_CLUSTER = 16;    // blocks of a cluster

// threads per block, at most (float64 rows hold twice the registers)
template <typename T>
constexpr int res_threads() { return sizeof(T) == 8 ? 512 : 1024; }
constexpr size_t RES_TERM = 8;     // bytes of a row's product on its way to the summing warp

// what one lane per species decides and every thread of the block reads (the
// scalar arithmetic is float64: on all warps it would cost more than the
// products)
template <typename T>
struct ResidentScalars {
    T beta[2], alpha[2], omega[2];
    int act[2], early[2], zero[2];
    int e0[2], e[2];   // exponents of r-hat and of the iteration's vectors in the sums
};

// shared memory of a block, in this order (all offsets multiples of 16 bytes)
template <typename T>
struct ResidentSmem {
    size_t w, idx, gather, terms, part, scal, total;
    __host__ __device__ ResidentSmem(int max_elems, int rows, int64_t N, int ns, bool cluster) {
        auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
        w = 0;
        idx = up(w + (size_t)max_elems * sizeof(T));
        gather = up(idx + (size_t)max_elems * sizeof(int32_t));
        terms = up(gather + (cluster ? (size_t)ns * N * sizeof(T) : 0));
        part = up(terms + (size_t)RES_SUMS * rows * RES_TERM);
        scal = up(part + (cluster ? 2 * RES_CLUSTER * RES_SUMS * sizeof(double) : 0));
        total = up(scal + sizeof(ResidentScalars<T>));
    }
};

// TPR lanes per row, slices of 32 rows per block, blocks and form; blocks = 0 when
// the operator does not fit
struct ResidentPlan {
    int blocks = 0, tpr = 1, spb = 0, max_elems = 0;
    bool cluster = false;
    size_t smem = 0;
};

inline int64_t slices_of(const GroupInfo& gi, int g) { return (gi.row_begin[g + 1] - gi.row_begin[g] + 31) / 32; }

// elements of the largest of the runs of spb consecutive slices that the blocks take
inline int64_t largest_block(const GroupInfo& gi, int64_t slices, int spb) {
    int64_t most = 0;
    for (int64_t b = 0; b < slices; b += spb) {
        int64_t elems = 0, s0 = 0;
        for (int g = 0; g < gi.ngroups; ++g) {
            const int64_t ns = slices_of(gi, g);
            elems += std::max<int64_t>(0, std::min(b + spb, s0 + ns) - std::max(b, s0)) * 32 * gi.npad[g];
            s0 += ns;
        }
        most = std::max(most, elems);
    }
    return most;
}

constexpr int RES_STATIC = 16;     // the grid barrier's own bytes
constexpr size_t RES_SMEM_MAX = 227 * 1024 - RES_STATIC;

// resides(plan): the device has room for the cluster of a plan.  Where it has not (a
// partition of a GPU may have fewer SMs side by side), the cooperative grid takes the
// operator.  The cluster comes first wherever its shared memory holds the operator (us
// a step, n = 31, cluster / grid: heat equation in float64, 642 rows 45/69, 2,562
// 54/71, 3,500 58/75, 5,000 70/72, 6,300 84/74; two species in float32, 642 rows 15/25,
// 2,562 26/29, 5,000 28/30, 6,300 34/32: its last fifth, above 5k rows, would be as
// fast or up to a fifth faster on the grid).
template <typename T, typename F>
ResidentPlan resident_plan(const GroupInfo& gi, int64_t N, int ns, int sms, F resides) {
    int64_t slices = 0;
    for (int g = 0; g < gi.ngroups; ++g) slices += slices_of(gi, g);
    for (int form = 0; form < 2; ++form) {
        ResidentPlan p;
        p.cluster = form == 0;
        const int64_t blocks = std::min<int64_t>(slices, p.cluster ? RES_CLUSTER : sms);
        const int64_t spb = (slices + blocks - 1) / blocks;
        if (spb * 32 > res_threads<T>()) continue;
        p.spb = (int)spb;
        p.blocks = (int)((slices + p.spb - 1) / p.spb);
        if (p.cluster)   // a power of two; the last blocks may have no rows
            for (int c = 1;; c *= 2)
                if (c >= p.blocks) {
                    p.blocks = c;
                    break;
                }
        const int64_t elems = largest_block(gi, slices, p.spb);
        if (elems * (int64_t)(sizeof(T) + 4) > (int64_t)RES_SMEM_MAX) continue;
        p.max_elems = (int)elems;
        p.smem = ResidentSmem<T>(p.max_elems, p.spb * 32, N, ns, p.cluster).total;
        if (p.smem > RES_SMEM_MAX) continue;
        // float32 rows take up to four lanes, float64 ones have one (us a step, n = 31,
        // one / two lanes: one species, 642 rows 45/39, 1,280 48/44, 2,562 54/57, 3,500
        // 58/63, 20k 78/76; two species, 2,562 63/71, 6,300 95/80, 20k 137/140: the
        // float64 unit is the bound unless a block has few rows)
        while (sizeof(T) == 4 && p.tpr < 4 && p.spb * 32 * p.tpr * 2 <= res_threads<T>()) p.tpr *= 2;
        if (p.cluster && !resides(p)) continue;
        return p;
    }
    return ResidentPlan();
}

}  // namespace rbffd
