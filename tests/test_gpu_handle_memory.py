"""GPU: what an assembled lattice holds and what its eigenvalue calls take: a handle has no
chunk workspace of its own, and a call's stays within the context's budget (with the same
numbers as without one)."""
import re
import threading

import numpy as np
import pytest

from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu


def _needs(fock, p):
    """Bytes that a handle of p takes, from the refusal of a context too small for it."""
    tiny = fock.Context(0, budget_bytes=1 << 16)
    with pytest.raises(fock.FockError) as e:
        tiny.assemble(p)
    tiny.close()
    return int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))


def _lowest_free(torch, call):
    """call()'s result and the least free device memory seen meanwhile."""
    low, stop = [torch.cuda.mem_get_info()[0]], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=watch)
    t.start()
    try:
        out = call()
    finally:
        stop.set()
        t.join()
    return out, low[0]


def test_handles_and_their_calls_stay_within_the_budget():
    torch = pytest.importorskip("torch")
    from paper_1702_00339_gb300 import fock
    page = 4 << 20                                   # the device's memory goes in pages of 2 MB
    p = _lattice((24, 24, 24), 16)                   # chunks of all its blocks: 6940 x 15.5 KB = 108 MB
    need = _needs(fock, p)
    budget = need + (16 << 20)
    free = fock.Context(0)
    b = free.assemble(p)
    ref = b.circulant_eig()
    free.close()
    ctx = fock.Context(0, budget_bytes=budget)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    b = ctx.assemble(p)
    assert before - torch.cuda.mem_get_info()[0] <= need + page
    for call in (b.circulant_eig, lambda: b.circulant_eig_range(0, p.ncell)):
        got, low = _lowest_free(torch, call)
        assert before - low <= budget + page
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    ctx.close()
