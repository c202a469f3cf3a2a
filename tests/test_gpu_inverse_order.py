"""What orders the loads that the coarse solves issue ahead of their programmatic wait.

A kernel launched early behind an inversion may start its own successor before the inversion's writes
are visible, so an inversion has to end with an ordinary edge to a launch that carries no data
(launch_order). The launchers are captured into a graph, followed by an early launch, and the graph's edges
are read: no programmatic edge leaves a kernel that writes the inverse. Nothing is executed.
"""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cuda.h>
#include <cstdio>
#include <string>
#include <vector>
#include "helm_internal.h"
using namespace helm;

static int edges(const char* what, cudaStream_t s, bool tail) {
    LevelDev L = {};
    L.nx = tail ? 11 : 31;
    L.nz = tail ? 9 : 30;
    const int n = L.nx * L.nz;
    char* d = nullptr;
    cudaMalloc(&d, 1 << 12);   // stands for every array: nothing is executed
    double* w2 = (double*)d;
    int* i = (int*)(d + 2048);
    cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    TAIL_OR_DENSE
    launch_coarse_dense<float>(n, (float*)d, i, i, 1, 1, (float*)d, (float*)d, 0, nullptr, s);
    cudaGraph_t g = nullptr;
    if (cudaStreamEndCapture(s, &g) != cudaSuccess || !g) return 1;
    size_t ne = 0;
    if (cuGraphGetEdges(g, nullptr, nullptr, nullptr, &ne) != CUDA_SUCCESS) return 2;
    std::vector<CUgraphNode> from(ne), to(ne);
    std::vector<CUgraphEdgeData> ed(ne);
    if (cuGraphGetEdges(g, from.data(), to.data(), ed.data(), &ne) != CUDA_SUCCESS) return 3;
    int early = 0, bad = 0;
    for (size_t k = 0; k < ne; ++k) {
        if (ed[k].type != CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC) continue;
        ++early;
        CUDA_KERNEL_NODE_PARAMS p;
        const char* name = nullptr;
        if (cuGraphKernelNodeGetParams(from[k], &p) != CUDA_SUCCESS || cuFuncGetName(&name, p.func) != CUDA_SUCCESS)
            return 4;
        if (std::string(name).find("k_order") == std::string::npos) { ++bad; std::printf("%s: early edge from %s\n", what, name); }
    }
    std::printf("%s: %zu edges, %d early, %d bad\n", what, ne, early, bad);
    cudaGraphDestroy(g);
    cudaFree(d);
    return bad || early != 1 ? 5 : 0;
}

int main() {
    cudaFree(nullptr);
    cudaStream_t s;
    cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    const int a = edges("dense level", s, false), b = edges("tail", s, true);
    return a ? 10 + a : b ? 20 + b : 0;
}
""".replace("TAIL_OR_DENSE", """if (tail)
        launch_coarse_invert(L, w2, i, 1, 1.0, 0.5, (double2*)d, i, (float2*)d, (double2*)d, s);
    else
        launch_dense_invert<float>(L, w2, i, 1, 1.0, 0.5, (float*)d, i, s);""")


def test_early_launches_behind_an_inversion(lib, tmp_path):
    from paper_1712_08743_gb300 import build

    src = tmp_path / "edges.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "edges")
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", f"-I{build.CSRC}", f"-I{build.INCLUDE}", str(src), "-o", exe,
                        f"-L{build.BUILD}", "-l:libhelm.so", "-L/usr/local/cuda/lib64/stubs", "-lcuda", "-Xlinker", f"-rpath={build.BUILD}"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300, cwd=os.path.dirname(exe))
    assert r.returncode == 0, r.stdout + r.stderr
