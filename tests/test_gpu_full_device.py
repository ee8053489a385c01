"""GPU: a device that others have filled since the contexts were made: a lattice whose chunk
workspace no longer fits is solved in smaller chunks, by the one-shot call and by a plan, with
the same numbers."""
import numpy as np
import pytest

from tests.test_gpu_handle_memory import _needs
from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu


def _planned(ctx, p):
    plan = ctx.plan([p])
    plan.execute()
    return plan.outputs()[0]


def test_smaller_chunks_where_the_device_is_full():
    torch = pytest.importorskip("torch")
    from paper_1702_00339_gb300 import fock
    p = _lattice((24, 24, 24), 16)                   # chunks of all its blocks: 6940 x 15.5 KB = 108 MB
    need = _needs(fock, p)
    first = fock.Context(0)
    ref = first.solve([p])[0]
    first.close()
    contexts = [fock.Context(0), fock.Context(0)]
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - need - (48 << 20), dtype=torch.uint8, device="cuda")
    try:
        for ctx, call in zip(contexts, (lambda c: c.solve([p])[0], lambda c: _planned(c, p))):
            out = call(ctx)
            ctx.close()
            assert out["status"] == 0
            assert np.array_equal(out["evals"], ref["evals"]) and np.array_equal(out["block_of"], ref["block_of"])
    finally:
        del filler
        torch.cuda.empty_cache()
