"""BiCGSTAB batches whose correction is summed before the preconditioner (vectors of 16 MiB and
more), at the smallest such batch and the one below it, with right-hand sides that end at
different iterations and one that is zero.

Bar: the solver's own, ||f - B u|| <= tol ||f||, evaluated with the CPU operator in FP64 (whose
rounding, about 1e-14 relative to ||f||, is what the factor 1 + 1e-3 leaves room for), and a zero
field for the zero right-hand side.
"""
import numpy as np
import pytest

import oracle
import oracle.helmholtz as hz
from synth import models

pytestmark = pytest.mark.gpu

NPML, PX, PZ = 8, 125, 75
N = (PX + 2 * NPML) * (PZ + 2 * NPML)


@pytest.fixture(scope="module")
def hg(lib):
    import paper_1712_08743_gb300 as m
    return m


@pytest.mark.parametrize("below", [0, 1])
@pytest.mark.parametrize("precision,density,tol", [("MIXED", False, 1e-9), ("MIXED", True, 1e-9),
                                                   ("FP64", False, 1e-10), ("FP32", False, 1e-3)])
def test_residual_at_both_sides_of_the_line(hg, precision, density, tol, below):
    size = 16 if precision == "FP64" else 8
    nrhs = -(-(16 << 20) // (size * N)) - below
    rng = np.random.default_rng(7)
    c = models.layered_model(rng, PX, PZ, 10.0, 5, 1500.0, 3500.0)
    rho = models.gardner_density(c) if density else None
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5, density=rho)
    om = 2 * np.pi * np.linspace(3.0, 9.0, nrhs)
    f = models.random_complex(rng, (nrhs, PZ + 2 * NPML, PX + 2 * NPML), np.complex64).astype(np.complex128)
    zero = nrhs // 2
    f[zero] = 0
    u, st, rc = hg.helm_solve(model, om, f=f, opts=dict(tol=tol, precision=getattr(hg, "HELM_PREC_" + precision)))
    assert rc == hg.HELM_OK and all(s["converged"] for s in st)
    assert not u[zero].any()
    m_pad = oracle.pad_slowness(1.0 / c, NPML)
    rho_pad = None if rho is None else oracle.pad_slowness(rho, NPML)
    alpha = hz.damping_profile(PX, PZ, NPML, 0.5)
    for k in (0, 1, nrhs // 3, nrhs - 2, nrhs - 1):
        B = hz.operator(m_pad, 10.0, om[k], alpha, rho_pad)
        res = f[k].ravel() - B @ u[k].ravel()
        assert np.linalg.norm(res) <= tol * (1 + 1e-3) * np.linalg.norm(f[k]), k
    model.close()
    ctx.close()


@pytest.mark.parametrize("coarse", ["DENSE", "FUSED"])
def test_few_large_right_hand_sides(hg, coarse):
    """Four right-hand sides of 724 x 726: the dense end and the persistent cycle, which the last V takes too."""
    px, pz, nrhs = 708, 710, 4
    assert 8 * (px + 2 * NPML) * (pz + 2 * NPML) * nrhs >= 16 << 20
    rng = np.random.default_rng(3)
    c = models.layered_model(rng, px, pz, 10.0, 6, 1500.0, 3500.0)
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)
    om = 2 * np.pi * np.linspace(3.0, 5.0, nrhs)
    f = models.random_complex(rng, (nrhs, pz + 2 * NPML, px + 2 * NPML), np.complex64).astype(np.complex128)
    u, st, rc = hg.helm_solve(model, om, f=f, opts=dict(tol=1e-8, coarse=getattr(hg, "HELM_COARSE_" + coarse)))
    assert rc == hg.HELM_OK and all(s["converged"] for s in st)
    alpha = hz.damping_profile(px, pz, NPML, 0.5)
    B = hz.operator(oracle.pad_slowness(1.0 / c, NPML), 10.0, om[-1], alpha)
    res = f[-1].ravel() - B @ u[-1].ravel()
    assert np.linalg.norm(res) <= 1e-8 * (1 + 1e-3) * np.linalg.norm(f[-1])
    model.close()
    ctx.close()
