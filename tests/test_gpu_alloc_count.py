"""The call that allocates nothing, seen where the library's allocations go: helm_alloc_count counts every
request to a context's own pool. helm_vcycle moves it (so a workspace allocated in the call would show), two
calls of helm_vcycle_noalloc on either coarse end do not."""
import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [(1.0, 0.5), (1.0, 0.0), (-1.0, 0.05)])
@pytest.mark.parametrize("nrhs", [3, 20])
def test_noalloc_asks_for_no_memory(lib, nrhs, beta):
    import torch

    import paper_1712_08743_gb300 as hg
    from paper_1712_08743_gb300.api import helm_vcycle_noalloc

    ctx = hg.Context(0)
    mdl = models.c1_model()
    model = hg.helm_create_model(ctx, mdl.slowness, mdl.h, mdl.npml, mdl.alpha_max)
    om = 2 * np.pi * np.linspace(4.0, 6.0, nrhs)
    r = torch.from_numpy(models.random_complex(np.random.default_rng(7), (nrhs, model.nz, model.nx), np.complex64)).cuda()
    n0 = lib.helm_alloc_count()
    ref = hg.helm_vcycle(model, om, r, beta, 0.5)
    n1 = lib.helm_alloc_count()
    assert n1 > n0
    for _ in range(2):
        z = torch.full_like(r, float("nan"))
        helm_vcycle_noalloc(model, om, r, z, beta, 0.5)
        assert lib.helm_alloc_count() == n1
        assert torch.equal(z, ref)
    model.close()
    ctx.close()
