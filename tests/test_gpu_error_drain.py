"""A call that fails after it has queued work returns with its stream idle: what it leaves behind may be
freed at once, and pool memory is freed without a wait of its own.

The context's stream is kept busy (a bounded delay of about a tenth of a second) and a call that cannot get its
workspace is made: 60000 right-hand sides of 441 x 241 need more than twice the GPU's memory, whatever
else is free (102 GB for the right-hand side, which is filled, and six times that in all).
"""
import ctypes as C

import numpy as np
import pytest

from synth import models

pytestmark = pytest.mark.gpu


def test_failed_call_leaves_the_stream_idle(lib):
    import torch

    import paper_1712_08743_gb300 as hg

    stream = torch.cuda.Stream()
    ctx = hg.Context(0, stream=stream)
    m3 = models.c3_model()
    model = hg.helm_create_model(ctx, m3.slowness, m3.h, m3.npml, m3.alpha_max)
    nrhs = 60000
    om = np.full(nrhs, 2 * np.pi * 5.0)
    omp = om.ctypes.data_as(C.POINTER(C.c_double))
    zeros = np.zeros(nrhs, dtype=np.int32).ctypes.data_as(C.POINTER(C.c_int))
    small = np.zeros(16)   # never reached: the field is written when everything is done
    sp = C.c_void_p(small.ctypes.data)
    with torch.cuda.stream(stream):
        torch.cuda._sleep(200_000_000)
    rc = lib.helm_solve(model.handle, nrhs, omp, zeros, zeros, None, sp, None, None)
    assert rc == hg.HELM_E_NOMEM, (rc, lib.helm_last_error())
    assert stream.query()
    stream.synchronize()
    model.close()
    ctx.close()
    torch.cuda.synchronize()
