"""A model that is destroyed after its context (an interpreter collects them in either order) gives its memory back without
reading the context, whose freed memory is overwritten here; the next call sees no error of it."""
import ctypes as C

import pytest

from synth import models

pytestmark = pytest.mark.gpu


def test_destroyed_after_its_context(lib):
    import paper_1712_08743_gb300 as hg

    mdl = models.c1_model()
    ctx = hg.Context(0)
    model = hg.helm_create_model(ctx, mdl.slowness, mdl.h, mdl.npml, mdl.alpha_max)
    ctx.close()
    libc = C.CDLL(None)
    libc.malloc.restype, libc.malloc.argtypes = C.c_void_p, [C.c_size_t]
    libc.free.argtypes = [C.c_void_p]
    blocks = [libc.malloc(n) for n in range(32, 512, 8) for _ in range(8)]
    for k, p in enumerate(blocks):
        C.memset(p, 0x7F, 32 + 8 * (k // 8))
    model.close()
    for p in blocks:
        libc.free(p)
    ctx = hg.Context(0)
    hg.helm_create_model(ctx, mdl.slowness, mdl.h, mdl.npml, mdl.alpha_max).close()
    ctx.close()
