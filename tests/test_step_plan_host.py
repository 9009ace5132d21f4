"""The resident step kernel's shape for an operator, on the host: a cluster where
the device has room for it, the cooperative grid where it has not (as on a
partition of a GPU with fewer SMs side by side), and the blocks' shares of operators
of one and of several stencil sizes against a list of their slices."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include "step_plan.cuh"
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
using namespace rbffd;

static GroupInfo groups(const std::vector<std::pair<int64_t, int>>& sizes, int64_t* N) {
    GroupInfo gi;
    memset(&gi, 0, sizeof(gi));
    *N = 0;
    for (auto& s : sizes) {
        gi.n[gi.ngroups] = s.second;
        gi.npad[gi.ngroups] = (s.second + 3) / 4 * 4;
        gi.row_begin[++gi.ngroups] = *N += s.first;
    }
    return gi;
}
static int64_t largest_by_list(const GroupInfo& gi, int spb) {
    std::vector<int64_t> start(1, 0);
    for (int g = 0; g < gi.ngroups; ++g)
        for (int64_t k = 0; k < (gi.row_begin[g + 1] - gi.row_begin[g] + 31) / 32; ++k)
            start.push_back(start.back() + 32 * gi.npad[g]);
    const int64_t n = (int64_t)start.size() - 1;
    int64_t most = 0;
    for (int64_t b = 0; b < n; b += spb) most = std::max(most, start[std::min(n, b + spb)] - start[b]);
    return most;
}
template <typename T>
static int check(const GroupInfo& gi, int64_t N, int ns, int limit) {
    int asked = 0;
    const ResidentPlan p = resident_plan<T>(gi, N, ns, 152, [&](const ResidentPlan& q) {
        ++asked;
        return q.blocks <= limit;
    });
    if (p.blocks == 0) return 0;
    int64_t slices = 0;
    for (int g = 0; g < gi.ngroups; ++g) slices += slices_of(gi, g);
    const bool sound = (int64_t)p.blocks * p.spb >= slices && p.spb * 32 * p.tpr <= res_threads<T>() &&
                       p.max_elems == largest_by_list(gi, p.spb) && p.smem <= RES_SMEM_MAX &&
                       p.blocks <= (p.cluster ? std::min(limit, RES_CLUSTER) : 152) && (!p.cluster || asked > 0);
    if (!sound) printf("unsound plan: N %lld blocks %d spb %d\n", (long long)N, p.blocks, p.spb);
    return !sound ? -1 : p.cluster ? 2 : 1;
}
int main() {
    int bad = 0;
    int64_t N;
    GroupInfo gi = groups({{2562, 31}}, &N);
    bad += check<double>(gi, N, 1, 16) != 2;    // a cluster of 16
    bad += check<double>(gi, N, 1, 8) != 1;     // no room for it: the grid
    bad += check<float>(gi, N, 2, 0) != 1;
    gi = groups({{40344, 50}}, &N);
    bad += check<float>(gi, N, 2, 16) != 1;
    gi = groups({{1000000, 31}}, &N);
    bad += check<float>(gi, N, 2, 16) != 0;     // too large for the chip
    std::mt19937 rng(1);
    for (int k = 0; k < 2000; ++k) {
        std::vector<std::pair<int64_t, int>> s;
        for (int g = 0; g < 1 + (int)(rng() % 4); ++g)
            s.push_back({1 + rng() % (k % 2 ? 3000 : 40000), 2 + (int)(rng() % 127)});
        gi = groups(s, &N);
        for (int limit : {0, 4, 16}) {
            bad += check<float>(gi, N, 1 + k % 2, limit) < 0;
            bad += check<double>(gi, N, 1 + k % 2, limit) < 0;
        }
    }
    printf("failed checks: %d\n", bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_plans_on_the_host(tmp_path):
    src = tmp_path / "plan.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "plan"
    csrc = os.path.join(ROOT, "paper_1404_0812_gb300", "csrc")
    build = subprocess.run([NVCC, "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-gencode",
                            "arch=compute_103a,code=sm_103a", "-o", str(exe), str(src)], capture_output=True, text=True)
    assert build.returncode == 0, build.stderr[-2000:]
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout[-2000:]
