"""Galerkin tiles chosen by the level's size: on both sides of the size rules, one right-hand side
and several, the cycle is that of the fixed tile shapes (the same operations per node; the
compiler may contract them differently, as in the other tile-shape tests: 1e-6)."""
import ctypes as C

import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu


# padded sides (with batch): levels of 7 .. 300 nodes a side; coarse nodes over the batch below and
# above 32768, fine nodes below and above 1e6
@pytest.mark.parametrize("nx,nz,nrhs", [(61, 47, 1), (141, 141, 3), (337, 290, 1), (337, 291, 16), (604, 521, 16)])
def test_size_rule_gives_the_fixed_shapes_cycle(lib, nx, nz, nrhs):
    import paper_1712_08743_gb300 as hg

    ctx = hg.Context(0)
    rng = np.random.default_rng(nx)
    c = models.layered_model(rng, nx - 8, nz - 8, 10.0, 5, 1500.0, 3000.0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, 4, 0.5)
    om = 2 * np.pi * rng.uniform(3.0, 6.0, nrhs)
    r = models.random_complex(rng, (nrhs, nz, nx), np.complex64)
    for coarse in (hg.HELM_COARSE_DENSE, hg.HELM_COARSE_TAIL):
        z = hg.helm_vcycle(model, om, r, (1.0, 0.5), 0.5, coarse=coarse)
        for code in ((0, 0), (4, 2)):
            assert lib.helm_set_tiles(model.handle, (C.c_int * 48)(*([code[0]] * 24 + [1] + [code[1]] * 23))) == 0
            q = hg.helm_vcycle(model, om, r, (1.0, 0.5), 0.5, coarse=coarse)
            assert np.linalg.norm(z - q) <= 1e-6 * np.linalg.norm(q), (coarse, code)
        assert lib.helm_set_tiles(model.handle, (C.c_int * 48)(*([1] * 48))) == 0
    model.close()
    ctx.close()
