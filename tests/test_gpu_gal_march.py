"""Galerkin levels of large batches (one warp per right-hand side and column strip): grids whose
levels are narrower than a strip, end inside one, have odd and even sides (border
stencils differ) and more rows than a segment, with a constant and a variable density.

Bar: the batch of 17 takes these kernels, the batch of its first 16 the one-tile kernels, with the
same coarse end. Both do a node's operations in complex64, so against the CPU cycle the one may be
no further off than twice the other, or than 2e-6 (about 30 roundings), whichever is more: how
far a cycle is off depends on its levels' conditioning, which both share.
"""
import numpy as np
import pytest

import oracle
import oracle.multigrid as mg
from synth import models

pytestmark = pytest.mark.gpu

NPML = 4
SIDES = [(41, 37), (60, 124), (123, 62), (127, 126), (243, 70), (72, 301)]


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
@pytest.mark.parametrize("density", [False, True])
@pytest.mark.parametrize("coarse", ["tail", "dense"])
def test_batch_of_17_is_as_near_the_cpu_cycle_as_16(hg, ctx, nx, nz, density, coarse):
    rng = np.random.default_rng(nx + 7 * nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 5, 1500.0, 3500.0)
    rho = models.gardner_density(c) if density else None
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5, density=rho)
    om = np.sort(2 * np.pi * rng.uniform(3.0, 8.0, 17))   # the lowest, in both batches, sets the cycle's shape
    r = models.random_complex(rng, (17, nz, nx), np.complex64)
    end = hg.HELM_COARSE_TAIL if coarse == "tail" else hg.HELM_COARSE_DENSE
    z17 = hg.helm_vcycle(model, om, r, (1.0, 0.5), 0.5, coarse=end)
    z16 = hg.helm_vcycle(model, om[:16], r[:16], (1.0, 0.5), 0.5, coarse=end)
    m2 = oracle.pad_slowness(1.0 / c, NPML) ** 2
    rho_pad = None if rho is None else oracle.pad_slowness(rho, NPML)
    lf = mg.fcycle_level(mg.level_shapes(nx, nz), (10.0 * om[0]) ** 2, float(np.sqrt(m2.max())))
    for k in (0, 7, 8, 15):
        V = mg.VCycle(m2, (10.0 * om[k]) ** 2, (1.0, 0.5), 0.5, rho_pad, coarse=coarse)
        V.lt = lf
        ref = V.apply(r[k].astype(np.complex128).ravel()).reshape(nz, nx)
        e17, e16 = (np.linalg.norm(z[k] - ref) / np.linalg.norm(ref) for z in (z17, z16))
        assert e17 <= max(2e-6, 2.0 * e16), (k, e17, e16)
    model.close()
