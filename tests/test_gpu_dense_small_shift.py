"""The dense level's elimination without pivots at small shifts, where its matrix is closer to singular.

Bar: the cycle's complex64 bar of the restatement tests (2e-5 relative L2), or 2 x 2^-24 x the level's condition number
(its matrix rounded to FP32 and its inverse rounded to FP32, each amplified by the condition number) where that
is more: 150 to 7300 on these levels.
"""
import numpy as np
import pytest

import oracle
import oracle.multigrid as mg
from synth import models

pytestmark = pytest.mark.gpu

NPML = 4


@pytest.mark.parametrize("nx,nz", [(62, 60), (64, 64), (66, 70), (300, 44)])
@pytest.mark.parametrize("beta2", [0.05, 0.02, 0.005])
def test_cycle_at_small_shifts(lib, nx, nz, beta2):
    import paper_1712_08743_gb300 as hg

    rng = np.random.default_rng(nx * 1000 + nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 5, 1500.0, 3000.0)
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)
    om = 2 * np.pi * 4.0
    r = models.random_complex(np.random.default_rng(1), (1, nz, nx), np.complex64)
    z = hg.helm_vcycle(model, [om], r, (1.0, beta2), 0.5, coarse=hg.HELM_COARSE_DENSE)[0].ravel()
    V = mg.VCycle(oracle.pad_slowness(1.0 / c, NPML) ** 2, (10.0 * om) ** 2, (1.0, beta2), 0.5, coarse="dense")
    ref = V.apply(r[0].astype(np.complex128).ravel())
    bar = max(2e-5, 2.0 ** -23 * np.linalg.cond(V.M[V.exact].toarray()))
    err = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    print(f"{err:.2e} of {bar:.2e}")
    assert err < bar
    model.close()
    ctx.close()
