"""The pivoted inverse of the tail's coarsest level behind an elimination that reported a pivot.

400 slots (more than the GPU holds at once, so late blocks start while early ones are done) of an 11 x 9
level with random weights, row-wise diagonally dominant by a quarter. With a weight of 1e90 everywhere
but in the first nodes the elimination's squared determinants overflow and every slot takes the
pivoted kernel; with a weight of 1 none does. Bar: max |M X - I| <= 1e-12. M is row-scaled in the
product; diagonal dominance by a quarter bounds the scaled condition number by (1 + 0.8) / (1 - 0.8) = 9, and
99 nodes x 9 x 2^-53 = 1e-13 with a factor of ten for complex products.
"""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "helm_internal.h"
using namespace helm;
using C = std::complex<double>;

int main(int, char** argv) {
    const double big = std::atof(argv[1]);
    const int nx = 11, nz = 9, n = nx * nz, ns = 400;
    std::vector<double> gk(kGalerkinCoefs * n, 0.0), w(n), w2(ns);
    std::vector<int> mods(ns, 0);
    srand(5);
    auto u = [] { return 0.5 + 0.5 * rand() / RAND_MAX; };
    for (int p = 0; p < n; ++p) w[p] = (p % nx < 3 && p / nx < 3 ? 1.0 : big) * u();
    auto edge = [&](int e, int p) -> int {   // the other node of stored entry e of node p, or -1
        const int dx[5] = {0, 1, 0, 1, -1}, dz[5] = {0, 0, 1, 1, 1};
        const int x = p % nx + dx[e], z = p / nx + dz[e];
        return x < 0 || x >= nx || z >= nz ? -1 : z * nx + x;
    };
    std::vector<double> sum(n, 0.0);
    for (int p = 0; p < n; ++p)
        for (int e = 1; e < 5; ++e)
            if (int q = edge(e, p); q >= 0) {
                const double g = std::fmin(w[p], w[q]) * u();
                gk[e * n + p] = -g;
                sum[p] += g;
                sum[q] += g;
            }
    for (int p = 0; p < n; ++p) { gk[p] = 1.25 * sum[p]; gk[5 * n + p] = u(); }
    for (int k = 0; k < ns; ++k) w2[k] = 1e-5 * (k + 1);
    const size_t nn = (size_t)n * n * ns;
    double *dgk, *dw2;
    double2 *work, *md;
    float2* mf;
    int *dmod, *err;
    if (cudaMalloc(&dgk, sizeof(double) * gk.size()) || cudaMalloc(&dw2, sizeof(double) * ns) ||
        cudaMalloc(&dmod, sizeof(int) * ns) || cudaMalloc(&err, sizeof(int)) || cudaMalloc(&work, sizeof(double2) * 2 * nn) ||
        cudaMalloc(&md, sizeof(double2) * nn) || cudaMalloc(&mf, sizeof(float2) * nn)) return 1;
    cudaMemcpy(dgk, gk.data(), sizeof(double) * gk.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dw2, w2.data(), sizeof(double) * ns, cudaMemcpyHostToDevice);
    cudaMemcpy(dmod, mods.data(), sizeof(int) * ns, cudaMemcpyHostToDevice);
    LevelDev L = {};
    L.nx = nx;
    L.nz = nz;
    L.gk = dgk;
    const double b1 = 1.0, b2 = 0.5;
    launch_coarse_invert(L, dw2, dmod, ns, b1, b2, work, err, mf, md, 0);
    int flag = -1;
    std::vector<C> X(nn);
    std::vector<std::complex<float>> Xf(nn);
    if (cudaMemcpy(X.data(), md, sizeof(double2) * nn, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(Xf.data(), mf, sizeof(float2) * nn, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(&flag, err, sizeof(int), cudaMemcpyDeviceToHost)) return 2;
    if ((flag != 0) != (big > 1.0)) { std::printf("flag %d\n", flag); return 3; }
    double worst = 0.0;
    int at = -1;
    for (int k = 0; k < ns; ++k) {
        std::vector<std::vector<std::pair<int, C>>> M(n);
        std::vector<double> D(n);
        for (int p = 0; p < n; ++p)
            for (int e = 0; e < 5; ++e) {
                const int q = edge(e, p);
                if (q < 0) continue;
                const C m(gk[e * n + p] - w2[k] * b1 * gk[(5 + e) * n + p], w2[k] * b2 * gk[(5 + e) * n + p]);
                M[p].push_back({q, m});
                if (e == 0) D[p] = std::abs(m);
                else M[q].push_back({p, m});
            }
        const C* Xk = X.data() + (size_t)k * n * n;
        for (int p = 0; p < n; ++p)
            for (int c = 0; c < n; ++c) {
                C r(p == c ? -1.0 : 0.0, 0.0);
                for (auto& t : M[p]) r += t.second * Xk[t.first * n + c];
                // column c of X carries 1 / M_cc, the row M_pp
                const double v = std::abs(r) * D[c] / D[p];
                if (!(v <= worst)) { worst = v; at = k; }
                const C x = Xk[p * n + c];
                if (!(Xf[(size_t)k * n * n + p * n + c] == std::complex<float>((float)x.real(), (float)x.imag()))) return 4;
            }
    }
    std::printf("weight %g: worst %.3g (slot %d)\n", big, worst, at);
    return worst <= 1e-12 ? 0 : 5;
}
"""


@pytest.mark.parametrize("weight", ["1", "1e90"])
def test_every_slot_is_inverted(lib, tmp_path, weight):
    from paper_1712_08743_gb300 import build

    src = tmp_path / "pivoted.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "pivoted")
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", f"-I{build.CSRC}", f"-I{build.INCLUDE}", str(src),
                        "-o", exe, f"-L{build.BUILD}", "-l:libhelm.so", "-Xlinker", f"-rpath={build.BUILD}"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe, weight], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
