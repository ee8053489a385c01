"""GPU: lattices queued on a server whose budget holds four of them with the least chunk
workspace go in one batch, which takes its chunks in what they leave, within the budget,
and give the numbers of a solve alone."""
import time

import numpy as np
import pytest

import lattice_inputs as li
from tests import _cases
from tests.test_gpu_handle_memory import _needs
from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spare", [0, 20 << 20])
def test_queued_lattices_share_a_batch(spare):
    from paper_1702_00339_gb300 import fock
    first = _cases.with_table(li.config2(0, L=96, n0=15, pad=32, n_perp=128, R=24))
    p = _lattice((20, 20, 20), 8)                   # chunks of all its blocks: 4004 x 4.4 KB
    ctx = fock.Context(0)
    ref = ctx.solve([p])[0]
    ctx.close()
    srv = fock.Server(0, slots=1, budget_bytes=4 * _needs(fock, p) + spare)
    t0 = srv.submit(first)
    end = time.time() + 60
    while srv.stats()["inflight"] == 0 and time.time() < end:
        time.sleep(0.0005)
    ts = [srv.submit(p) for _ in range(4)]
    rs = [srv.poll(t, timeout_ms=120000) for t in ts]
    srv.poll(t0, timeout_ms=120000)
    st = srv.stats()
    srv.stop()
    assert st["peak_reserved_bytes"] <= st["budget_bytes"]
    for r in rs:
        assert r["status"] == 0 and r["batch_size"] == 4
        assert np.array_equal(r["evals"], ref["evals"]) and np.array_equal(r["block_of"], ref["block_of"])
