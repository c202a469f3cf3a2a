"""Length of the FP32 addition chains in the Gram-Schmidt dot products, for single right-hand sides and batches.

All products are 1 + 29 x 2^-23, whose excess over 1 is lost in every addition to a sum of 64 and more, so that a long
chain shows as a relative error of 2e-6 and more. Bar: 22 x 2^-24 relative: where four sums share a wave of two blocks of
384 threads per SM a thread has at most 38 points of a 1041 x 1041 field, added in groups of two or four (at
most 19 additions of groups, one level in a group of two), and the warp's first two steps are in FP32; everything above is in 64
bits.
"""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "helm_common.cuh"
#include "helm_internal.h"
using namespace helm;

template <typename E> E* dev(size_t n) {
    void* p = nullptr;
    if (cudaMalloc(&p, n * sizeof(E)) != cudaSuccess || cudaMemset(p, 0, n * sizeof(E)) != cudaSuccess) std::exit(9);
    return static_cast<E*>(p);
}

int main(int, char** argv) {
    const size_t n = 1041 * 1041;
    const int nrhs = std::atoi(argv[1]), j = std::atoi(argv[2]), m = kMaxRestart;
    const size_t vs = n * nrhs, nb = nrhs;
    const float c = 1.0f + 29.0f / 8388608.0f;
    std::vector<float2> slot(vs, make_float2(c, 0.0f));
    float2* V = dev<float2>(vs * (j + 2));
    for (int k = 0; k <= j; ++k) cudaMemcpy(V + vs * k, slot.data(), sizeof(float2) * vs, cudaMemcpyHostToDevice);
    for (auto& v : slot) v = make_float2(1.0f, 0.0f);
    cudaMemcpy(V + vs * (j + 1), slot.data(), sizeof(float2) * vs, cudaMemcpyHostToDevice);
    FgDev fg = {};
    fg.m = m;
    fg.H = dev<double2>(nb * (m + 1) * m);
    fg.tmp = dev<double2>(nb * (m + 1));
    fg.sinv = dev<double>(nb * (m + 1));
    fg.wn2 = dev<double>(nb);
    std::vector<double> ones(nb * (m + 1), 1.0);
    cudaMemcpy(fg.sinv, ones.data(), sizeof(double) * ones.size(), cudaMemcpyHostToDevice);
    std::vector<RhsState> st(nrhs, RhsState{});
    for (auto& s : st) s.active = 1;
    RhsState* dst = dev<RhsState>(nb);
    cudaMemcpy(dst, st.data(), sizeof(RhsState) * nb, cudaMemcpyHostToDevice);
    const int ps = fg_partials(n);
    double* part = dev<double>((size_t)ps * nb);
    launch_fg_dots<float>((float*)V, vs, (float*)(V + vs * (j + 1)), j, 0, 0, 0, part, ps, dst, fg, n, nrhs, 0);
    std::vector<double2> d(nb * (m + 1));
    if (cudaMemcpy(d.data(), fg.tmp, sizeof(double2) * d.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    double worst = 0.0;
    for (int b = 0; b < nrhs; ++b)
        for (int i = 0; i <= j; ++i) {
            const double e = std::fabs(d[b * (m + 1) + i].x / ((double)n * c) - 1.0);
            if (!(e <= worst)) worst = e;
        }
    std::printf("nrhs %d, j %d: %.3g\n", nrhs, j, worst);
    return worst <= 22.0 / 16777216.0 ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def exe(lib, tmp_path_factory):
    from paper_1712_08743_gb300 import build

    d = tmp_path_factory.mktemp("dots")
    src, out = d / "dots.cu", str(d / "dots")
    src.write_text(PROGRAM)
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", f"-I{build.CSRC}",
                        f"-I{build.INCLUDE}", str(src), "-o", out, f"-L{build.BUILD}", "-l:libhelm.so", "-Xlinker",
                        f"-rpath={build.BUILD}"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("nrhs", [1, 2, 20])
@pytest.mark.parametrize("j", [0, 1, 3, 7, 9, 15])
def test_chains(exe, nrhs, j):
    r = subprocess.run([exe, str(nrhs), str(j)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
