"""A fast setup on a device with room for the FP64 translations' table but not
for the fixed-point form's matrices or its second copy of the multipoles: the
FP64 form does the work.  The expansions agree with those of the fixed-point
form to the tolerance of the parity tests.
"""
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


def _leave(room):
    """holds all but room to room + 2 MiB of the device's memory (page tables of
    the held block take some of it too)"""
    import torch
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    for more in range(0, 64 << 20, 2 << 20):
        hold = torch.empty(free - room - more, dtype=torch.uint8, device="cuda")
        if torch.cuda.mem_get_info()[0] >= room:
            return hold
        del hold
        torch.cuda.empty_cache()
    pytest.skip("memory of the device in use by others")


# of 5 MB of matrices and 32768 x 100 words of multipoles: room for neither (the
# FP64 form's table, 1 MB, finds it), or for the matrices only
@pytest.mark.parametrize("room", [4 << 20, 20 << 20])
def test_fast_setup_without_room_for_the_integers(room):
    import torch
    n, a, L, p = 20000, 30.0, 6, 9
    pos, q = uniform_system(n, a, seed=5)
    levels = {}
    # loads every kernel, the FP64 ones too
    qq = q.copy()
    qq[int(np.argmax(q))] = 2.0 ** -10
    qq[int(np.argmin(q))] = -2.0 ** -10
    for x in (qq, q):
        c = mcfmm.Context(pos, x, a, L, p)
        c.setup(mcfmm.SETUP_FMM)
        levels = {l: c.local(l) for l in range(2, L + 1)}
        e = c.energy()
        c.close()
    c = mcfmm.Context(pos, q, a, L, p)
    c.setup(mcfmm.SETUP_MULTIPOLE)  # the multipoles' own memory
    hold = _leave(room)
    try:
        c.setup(mcfmm.SETUP_FMM)
    finally:
        del hold
        torch.cuda.empty_cache()
    for l, ref in levels.items():
        assert np.max(np.abs(c.local(l) - ref)) <= 1e-12 * np.max(np.abs(ref)), l
    assert abs(c.energy() - e) <= 1e-10 * abs(e)
    c.close()
