"""Block-tridiagonal inversion of a coarse level: every register-tile width, both block
directions, both precisions, and the pivoted kernel where the shift rules the
elimination out.

Bars: the cycle's complex64 bar of the restatement tests (2e-5 relative L2). The complex128
inverse has no entry point of its own: it is seen through the tail's coarsest solve (the
same cycle bar) and through a complex128 FGMRES solve, whose field meets the refined bar
(1e-6) and whose iteration count is that of full GMRES on the CPU with the restated cycle as
the preconditioner, within one step (rounding can move the step that crosses the tolerance).
"""
import numpy as np
import pytest

import oracle
import oracle.multigrid as mg
from synth import models

pytestmark = pytest.mark.gpu

NPML = 4
# padded sides -> sides of the level with at most 1200 nodes
SHAPES = [
    (12, 13),      # 6 x 6: the smallest block count a hierarchy gives
    (62, 60),      # 31 x 30, columns as blocks
    (64, 64),      # 32 x 32, the widest of the two-tile instance
    (66, 70),      # 33 x 35, the three-tile instance
    (68, 69),      # 34 x 34
    (141, 141),    # 17 x 17, one past the one-tile instance
    (300, 44),     # 75 x 11, long and thin, columns as blocks
    (44, 300),     # 11 x 75
]


def _model(hg, ctx, nx, nz):
    rng = np.random.default_rng(nx * 1000 + nz)
    c = models.layered_model(rng, nx - 2 * NPML, nz - 2 * NPML, 10.0, 5, 1500.0, 3000.0)
    return 1.0 / c, hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)


@pytest.fixture(scope="module")
def hg(lib):
    import paper_1712_08743_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(hg):
    c = hg.Context(0)
    yield c
    c.close()


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nx,nz", SHAPES)
def test_cycle_with_the_inverted_level(hg, ctx, nx, nz):
    slow, model = _model(hg, ctx, nx, nz)
    om = 2 * np.pi * np.array([3.0, 5.0])
    r = models.random_complex(np.random.default_rng(1), (2, nz, nx), np.complex64)
    m2 = oracle.pad_slowness(slow, NPML) ** 2
    # the tail's coarsest level goes through the complex128 inversion; the last shift through
    # the pivoted kernel (|beta2| < 0.1 |beta1|)
    for coarse, kind, beta in ((hg.HELM_COARSE_DENSE, "dense", (1.0, 0.5)), (hg.HELM_COARSE_TAIL, "tail", (1.0, 0.5)),
                               (hg.HELM_COARSE_TAIL, "tail", (-1.0, 0.05))):
        z = hg.helm_vcycle(model, om, r, beta, 0.5, coarse=coarse)
        for k in range(2):
            ref = mg.VCycle(m2, (10.0 * om[k]) ** 2, beta, 0.5, coarse=kind).apply(r[k].astype(np.complex128).ravel())
            assert rel(z[k].ravel(), ref) < 2e-5, (kind, beta, k, rel(z[k].ravel(), ref))
    model.close()


def gmres_steps(B, f, precond, target, most):
    """Arnoldi steps of right-preconditioned GMRES from zero until the residual is target * |f|."""
    V, Z, H = [f / np.linalg.norm(f)], [], np.zeros((most + 1, most), complex)
    for j in range(most):
        Z.append(precond(V[j]))
        w = B @ Z[j]
        for _ in range(2):
            for i in range(j + 1):
                h = np.vdot(V[i], w)
                H[i, j] += h
                w = w - h * V[i]
        H[j + 1, j] = np.linalg.norm(w)
        V.append(w / H[j + 1, j])
        e = np.zeros(j + 2, complex)
        e[0] = 1.0
        y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
        if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= target:
            return j + 1
    return most


@pytest.mark.parametrize("nx,nz,freq", [(62, 60, 4.0), (66, 70, 4.0), (300, 44, 2.0), (141, 141, 2.0)])
def test_complex128_inverse_in_a_solve(hg, ctx, nx, nz, freq):
    slow, model = _model(hg, ctx, nx, nz)
    om, src = 2 * np.pi * np.array([freq]), np.array([[nx // 3, 2]])
    u, st, rc = hg.helm_solve(model, om, src, opts=dict(tol=1e-10, precision="fp64", krylov=hg.HELM_KRYLOV_FGMRES,
                                                        restart=32, coarse=hg.HELM_COARSE_DENSE))
    assert rc == hg.HELM_OK and st[0]["dense_level"] >= 1
    ref = oracle.solve_fields(slow, 10.0, om[0], src, NPML, 0.5)
    assert rel(u, ref) < 1e-6
    m_pad = oracle.pad_slowness(slow, NPML)
    B = 100.0 * oracle.operator(m_pad, 10.0, om[0], oracle.damping_profile(nx - 2 * NPML, nz - 2 * NPML, NPML, 0.5))
    f = np.zeros(nx * nz, complex)
    f[(src[0, 1] + NPML) * nx + src[0, 0] + NPML] = 1.0
    V = mg.VCycle(m_pad ** 2, (10.0 * om[0]) ** 2, (1.0, 0.5), 0.5, coarse="dense")
    steps = gmres_steps(B, f, V.apply, 0.9e-10, 32)
    assert steps < 32 and abs(st[0]["iters"] - steps) <= 1, (st[0]["iters"], steps)
    model.close()
