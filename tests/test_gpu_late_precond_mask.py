"""The preconditioner cycle that ends an inner solve of a large batch runs for the right-hand sides that are still being
refined: with one of 2048 that is not zero, a launch of the tail (one block per right-hand side) takes the same time in
that cycle as in the iterations.

Measured with the library's own event pairs: the mean over a BiCGSTAB solve's tail launches, of which one in ten and more
belongs to such a cycle, against the mean over an FGMRES solve of the same batch, which has none. A cycle over the whole batch takes
2048 blocks of one per SM, fourteen waves in place of one, and raises the mean by a factor of two and more; the bar is 1.5.
"""
import ctypes as C

import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu

NPML, PX, PZ, NRHS = 20, 101, 51, 2048


def _mean_tail(hg, lib, model, om, f, u, **opts):
    from paper_1712_08743_gb300 import _lib

    hg.helm_solve(model, om, f=f, opts=dict(tol=1e-8, **opts), out=u)
    lib.helm_profile_begin()
    _, st, rc = hg.helm_solve(model, om, f=f, opts=dict(tol=1e-8, **opts), out=u)
    buf, n = (_lib.helm_profile_entry * 256)(), C.c_int()
    lib.helm_profile_end(buf, 256, C.byref(n))
    assert rc == hg.HELM_OK and st[0]["converged"]
    e = [b for b in buf[:min(n.value, 256)] if b.name == b"k_tail"]
    return sum(b.ms for b in e) / sum(b.launches for b in e)


def test_one_of_many(lib):
    import torch

    import paper_1712_08743_gb300 as hg

    c = models.layered_model(np.random.default_rng(7), PX, PZ, 10.0, 6, 1500.0, 3500.0)
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, NPML, 0.5)
    om = np.full(NRHS, 2 * np.pi * 6.0)
    f = torch.zeros((NRHS, PZ + 2 * NPML, PX + 2 * NPML), dtype=torch.complex128, device="cuda")
    f[0, NPML + 2, NPML + 5] = 1.0
    u = torch.empty_like(f)
    # short inner solves: one cycle in three or so ends one
    bicg = _mean_tail(hg, lib, model, om, f, u, inner_tol=0.5, check_every=1, max_outer=100)
    fgm = _mean_tail(hg, lib, model, om, f, u, krylov=hg.HELM_KRYLOV_FGMRES, restart=10)
    print(f"{1e3 * bicg:.1f} us per tail launch against {1e3 * fgm:.1f}")
    assert bicg <= 1.5 * fgm
    model.close()
    ctx.close()
