"""Read-outs of a context whose chain an enqueued batch runs on another
context's stream: positions read right after the call are those at the end of
the run, as a read-out waits for the work of every stream that synchronises
with the legacy one.
"""
import ctypes

import numpy as np
import pytest

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _stream():
    import torch
    s = ctypes.c_void_p()
    assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(s))) == 0
    return s.value


def test_positions_after_an_enqueued_batch():
    import torch
    torch.cuda.synchronize()  # (creates the device's context)
    streams = [_stream(), _stream()]
    ctxs = []
    for i, s in enumerate(streams):
        pos, q = uniform_system(600, 18.0, seed=i)
        c = mcfmm.Context(pos, q, 18.0, 3, 8, stream=s)
        c.setup(mcfmm.SETUP_FMM)
        ctxs.append(c)
    b = mcfmm.Batch(ctxs)
    start = [c.positions() for c in ctxs]
    b.run(5000, [1, 2], stats=False)
    got = ctxs[1].positions()
    torch.cuda.synchronize()
    end = [c.positions() for c in ctxs]
    assert not np.array_equal(start[1], end[1])
    assert np.array_equal(got, end[1])
    b.run(5000, [1, 2], stats=False)
    loc = ctxs[1].local(3)
    torch.cuda.synchronize()
    assert np.array_equal(loc, ctxs[1].local(3))
    b.close()
    for c in ctxs:
        c.close()
    for s in streams:
        torch.cuda.cudart().cudaStreamDestroy(s)
