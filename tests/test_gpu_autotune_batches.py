"""Tuning for a batch that the marching kernels take leaves the Galerkin levels' tile codes, which only smaller
batches use, as they were; the finest level's row segments are still chosen. Codes 2 (restriction) and 3
(prolongation) on every level are the ones set beforehand."""
import ctypes as C

import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("density", [False, True])
@pytest.mark.parametrize("nrhs", [17, 64])
def test_codes_of_small_batches_stay(lib, nrhs, density):
    import paper_1712_08743_gb300 as hg
    from paper_1712_08743_gb300 import autotune

    n = autotune.NTILES // 2
    rng = np.random.default_rng(3)
    c = models.layered_model(rng, 401, 201, 10.0, 5, 1500.0, 3000.0)
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, 1.0 / c, 10.0, 20, 0.5, density=models.gardner_density(c) if density else None)
    codes = [2] * n + ([1] + [3] * (n - 1))
    assert lib.helm_set_tiles(model.handle, (C.c_int * (2 * n))(*codes)) == hg.HELM_OK
    out = (C.c_int * (2 * n))()
    assert lib.helm_autotune(model.handle, nrhs, 2 * np.pi * 5.0, out) == hg.HELM_OK
    assert list(out[:n]) == codes[:n] and list(out[n + 1:]) == codes[n + 1:]
    assert out[n] in ((1,) if density else (0, 1))
    model.close()
    ctx.close()
