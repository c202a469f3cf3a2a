"""The context's memory pool: bounded between calls, shared by calls, given back with the context."""
import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu


def test_pool_is_bounded_and_given_back(lib):
    import torch

    import paper_1712_08743_gb300 as hg

    torch.cuda.synchronize()
    total = torch.cuda.mem_get_info(0)[1]
    ctx0 = hg.Context(0)   # keeps the library's module loaded while the free memory is compared
    m = models.c1_model()
    warm = hg.helm_create_model(ctx0, m.slowness, m.h, m.npml, m.alpha_max)
    hg.helm_solve(warm, m.omegas, m.sources, opts=dict(tol=1e-6))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info(0)[0]
    ctx = hg.Context(0)
    big = models.c3_model()
    model = hg.helm_create_model(ctx, big.slowness, big.h, big.npml, big.alpha_max)
    om = np.repeat(big.omegas[:2], 12)
    src = np.tile(big.sources[:12], (2, 1))
    ref = None
    for k in range(3):   # the second and third call run on the first one's memory
        u, st, rc = hg.helm_solve(model, om, src, opts=dict(tol=1e-8))
        assert rc == hg.HELM_OK
        ref = u.copy() if ref is None else ref
        assert np.array_equal(u, ref)
        held = before - torch.cuda.mem_get_info(0)[0]
        assert 0 <= held <= total // 32 + (1 << 30)   # the pool's bound, the model and page rounding
    model.close()
    ctx.close()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info(0)[0] <= 64 << 20
    warm.close()
    ctx0.close()
