"""The finest level's marching kernels, whose warps (column strips of 30 coarse or 60 fine columns by row
segments) fill the blocks without gaps: sides around a strip's width and a segment's length, and
batches that give blocks of one, of some and of the most warps, against the CPU cycle
(complex64) and through whole FP64 solves.

Bars. Cycle: 2e-5 relative, that of the cycle's other tests. Solve: the solver's own,
||f - B u|| <= tol ||f|| with the CPU operator in FP64 (1e-3 of it left for that rounding).
"""
import numpy as np
import pytest

import oracle
import oracle.helmholtz as hz
import oracle.multigrid as mg
from synth import models

pytestmark = pytest.mark.gpu

NPML = 6
SIDES = [(59, 61), (60, 64), (61, 127), (120, 37), (121, 66), (241, 45)]


@pytest.fixture(scope="module")
def hg(lib):
    import paper_1712_08743_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(hg):
    c = hg.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("nx,nz", SIDES)
@pytest.mark.parametrize("nrhs", [1, 5, 48])
def test_cycle_against_cpu(hg, ctx, nx, nz, nrhs):
    rng = np.random.default_rng(nx + 7 * nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 4, 1500.0, 3500.0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)
    om = np.sort(2 * np.pi * rng.uniform(3.0, 7.0, nrhs))
    r = models.random_complex(rng, (nrhs, nz, nx), np.complex64)
    z = hg.helm_vcycle(model, om, r, (1.0, 0.5), 0.5, coarse=hg.HELM_COARSE_DENSE)
    m2 = oracle.pad_slowness(1.0 / c, NPML) ** 2
    lf = mg.fcycle_level(mg.level_shapes(nx, nz), (10.0 * om[0]) ** 2, float(np.sqrt(m2.max())))
    for k in {0, nrhs // 2, nrhs - 1}:
        V = mg.VCycle(m2, (10.0 * om[k]) ** 2, (1.0, 0.5), 0.5, None, coarse="dense")
        V.lt = lf
        ref = V.apply(r[k].astype(np.complex128).ravel()).reshape(nz, nx)
        assert np.linalg.norm(z[k] - ref) <= 2e-5 * np.linalg.norm(ref), k
    model.close()


@pytest.mark.parametrize("nx,nz", SIDES)
@pytest.mark.parametrize("nrhs", [1, 9])
@pytest.mark.parametrize("krylov", ["BICGSTAB", "FGMRES"])
def test_fp64_solve(hg, ctx, nx, nz, nrhs, krylov):
    rng = np.random.default_rng(nx + 5 * nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 4, 1500.0, 3500.0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)
    om = 2 * np.pi * np.linspace(3.0, 7.0, nrhs)
    f = models.random_complex(rng, (nrhs, nz, nx), np.complex64).astype(np.complex128)
    opts = dict(tol=1e-10, precision=hg.HELM_PREC_FP64, krylov=getattr(hg, "HELM_KRYLOV_" + krylov))
    u, st, rc = hg.helm_solve(model, om, f=f, opts=opts)
    assert rc == hg.HELM_OK and all(s["converged"] for s in st)
    alpha = hz.damping_profile(nx - 2 * NPML, nz - 2 * NPML, NPML, 0.5)
    for k in {0, nrhs - 1}:
        B = hz.operator(oracle.pad_slowness(1.0 / c, NPML), 10.0, om[k], alpha)
        res = f[k].ravel() - B @ u[k].ravel()
        assert np.linalg.norm(res) <= 1e-10 * (1 + 1e-3) * np.linalg.norm(f[k]), k
    model.close()
