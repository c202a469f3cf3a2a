"""Solves and cycles whose dense coarse inverse could not be formed: the tail takes over.

A density of 1 in one corner and of `contrast` everywhere else puts the level's pivots that far from its first
diagonal entry, by which the inversion scales: a contrast of 1e12 leaves the range of the
complex64 elimination, one of 1e90 that of the complex128 one, and neither is anything the rest of the
solver cannot hold. Bars: the cycle is that of the tail bit for bit (the same kernels on the same
inputs); a solve ends on the tail (dense_level 0) with the residual it was asked for.
"""
import numpy as np
import pytest

import oracle
import oracle.helmholtz as hz
from synth import models

pytestmark = pytest.mark.gpu

NPML = 8


@pytest.fixture(scope="module")
def hg(lib):
    import paper_1712_08743_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(hg):
    c = hg.Context(0)
    yield c
    c.close()


def _model(hg, ctx, nx, nz, contrast):
    rng = np.random.default_rng(nx * 1000 + nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 5, 1500.0, 3000.0)
    rho = np.full(c.shape, contrast)
    rho[:6, :6] = 1.0
    return 1.0 / c, rho, hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5, density=rho)


@pytest.mark.parametrize("nx,nz", [(62, 60), (136, 132), (300, 44)])
def test_cycle_is_the_tails(hg, ctx, nx, nz):
    _, _, model = _model(hg, ctx, nx, nz, 1e12)
    om = 2 * np.pi * np.array([3.0, 5.0])
    r = models.random_complex(np.random.default_rng(1), (2, nz, nx), np.complex64)
    z = [hg.helm_vcycle(model, om, r, (1.0, 0.5), 0.5, coarse=c) for c in (hg.HELM_COARSE_DENSE, hg.HELM_COARSE_TAIL)]
    assert np.all(np.isfinite(z[1])) and np.array_equal(z[0], z[1])
    model.close()


# 136 x 132: the dense level has 34 x 33 = 1122 nodes, more than a complex128 tail starts with
@pytest.mark.parametrize("nx,nz", [(62, 60), (136, 132)])
@pytest.mark.parametrize("precision,contrast,tol", [("mixed", 1e12, 1e-8), ("fp64", 1e90, 1e-8)])
@pytest.mark.parametrize("krylov", ["BICGSTAB", "FGMRES"])
def test_solve_ends_on_the_tail(hg, ctx, nx, nz, precision, contrast, tol, krylov):
    slow, rho, model = _model(hg, ctx, nx, nz, contrast)
    om = 2 * np.pi * np.array([3.0, 5.0])
    f = models.random_complex(np.random.default_rng(2), (2, nz, nx), np.complex64).astype(np.complex128)
    u, st, rc = hg.helm_solve(model, om, f=f, opts=dict(tol=tol, precision=precision, max_it=2000,
                                                        krylov=getattr(hg, "HELM_KRYLOV_" + krylov)))
    assert rc == hg.HELM_OK and all(s["converged"] and s["dense_level"] == 0 for s in st), st
    alpha = hz.damping_profile(nx - 2 * NPML, nz - 2 * NPML, NPML, 0.5)
    for k in range(2):
        B = hz.operator(oracle.pad_slowness(slow, NPML), 10.0, om[k], alpha, oracle.pad_slowness(rho, NPML))
        res = f[k].ravel() - B @ u[k].ravel()
        assert np.linalg.norm(res) <= tol * (1 + 1e-3) * np.linalg.norm(f[k])
    model.close()
