"""A dense inversion whose launch is refused: cycle and solve take the multigrid tail.

The launcher is replaced, in a child process, by one that returns an error code and launches nothing (a shared
object loaded ahead of the library, whose symbol the library's calls then resolve to). Bar: the cycle is
that of the tail bit for bit; the solve converges on the tail (dense_level 0).
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

FAKE = r"""
#include "helm_internal.h"
namespace helm {
template <typename T>
cudaError_t launch_dense_invert(const LevelDev&, const double*, const int*, int, double, double, T*, int*,
                                cudaStream_t, bool) {
    return cudaErrorInvalidConfiguration;
}
template cudaError_t launch_dense_invert<float>(const LevelDev&, const double*, const int*, int, double, double, float*,
                                                int*, cudaStream_t, bool);
}
"""

CHILD = r"""
import ctypes, sys
ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL)
import numpy as np
import paper_1712_08743_gb300 as hg
from synth import models
mdl = models.c1_model()
ctx = hg.Context(0)
model = hg.helm_create_model(ctx, mdl.slowness, mdl.h, mdl.npml, mdl.alpha_max)
r = models.random_complex(np.random.default_rng(1), (1, model.nz, model.nx), np.complex64)
z = [hg.helm_vcycle(model, mdl.omegas, r, (1.0, 0.5), 0.5, coarse=c) for c in (hg.HELM_COARSE_DENSE, hg.HELM_COARSE_TAIL)]
assert np.all(np.isfinite(z[1])) and np.array_equal(z[0], z[1])
u, st, rc = hg.helm_solve(model, mdl.omegas, mdl.sources, opts=dict(tol=1e-8))
assert rc == hg.HELM_OK and st[0]["converged"] and st[0]["dense_level"] == 0, (rc, st)
model.close()
ctx.close()
print("took the tail")
"""


def test_tail_behind_a_refused_launch(lib, tmp_path):
    from paper_1712_08743_gb300 import build

    src, so = tmp_path / "fake.cu", str(tmp_path / "fake.so")
    src.write_text(FAKE)
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{build.CSRC}",
                        f"-I{build.INCLUDE}", str(src), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([sys.executable, "-c", CHILD, so], capture_output=True, text=True, timeout=300, cwd=build.ROOT,
                       env=dict(os.environ, PYTHONPATH=build.ROOT))
    assert r.returncode == 0 and "took the tail" in r.stdout, r.stdout + r.stderr
